"""Build of the library's host code with the CUDA runtime on host threads
(fake_cuda.cpp), and runs of a piece of Python against it in a process of its
own, ended after a limit: a call that never returns is a failed test."""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes as C, threading, time
import numpy as np
from paper_2509_10757_gb300 import _lib as L, scenes
from paper_2509_10757_gb300.batch import Context, HostFrame, PackedBatch, stream_desc_of
lib = L.load()
lib.fake_gate.restype = C.c_void_p
lib.fake_gate.argtypes = lib.fake_open.argtypes = [C.c_void_p]

def stream():
    s = C.c_void_p()
    assert lib.cudaStreamCreateWithFlags(C.byref(s), 0) == 0
    return s

def log():
    b = C.create_string_buffer(1 << 20)
    assert lib.fake_log(b, len(b)) >= 0
    return b.value.decode().split('\\n')[:-1]

def track(ctx, pb, st):
    b = pb.batch()
    return L.ft_track_batch(ctx.ptr, st, None, C.byref(b))
"""


def fake_library(tmp_path_factory) -> str:
    from paper_2509_10757_gb300 import build as B
    B.build()
    out = str(tmp_path_factory.mktemp("host") / "libft_host.so")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc())))
    objs = [os.path.join(B.BUILD, f + ".cu.o") for f in ("ft_api", "ft_serve", "ft_noalloc")]
    cmd = ["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-pthread", "-Wl,-Bsymbolic", "-I" + B.CSRC,
           "-I" + B.INCLUDE, "-I" + os.path.join(cuda, "include"), os.path.join(HERE, "fake_cuda.cpp"), *objs,
           "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-4000:]
    return out


def run_against(library: str, code: str, limit_s: float = 60.0):
    env = dict(os.environ, FT_LIB=library, PYTHONPATH=ROOT)
    try:
        r = subprocess.run([sys.executable, "-c", PRELUDE + code], env=env, cwd=ROOT, capture_output=True, text=True,
                           timeout=limit_s)
    except subprocess.TimeoutExpired:
        pytest.fail(f"the calls did not return within {limit_s:g} s")
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
