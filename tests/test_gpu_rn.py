"""The pose solver's rounded square root and reciprocals (ft_rn.h) against the
device's __fsqrt_rn and __frcp_rn, bit for bit, on every float of their range.
The check is a small program compiled here against the library's header."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SOURCE = r"""
#include <cstdio>
#include "ft_rn.h"

__global__ void check(unsigned first, unsigned count, unsigned long long *bad)
{
    const unsigned stride = gridDim.x * blockDim.x;
    unsigned wrong[3] = {0, 0, 0};
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride) {
        const float x = __uint_as_float(first + i);
        if (!ft::rn_range(x)) continue;
        float root, inv;
        ft::rn_sqrt_rcp(x, root, inv);
        const float r = __fsqrt_rn(x);
        wrong[0] += __float_as_uint(root) != __float_as_uint(r);
        wrong[1] += __float_as_uint(inv) != __float_as_uint(__frcp_rn(r));
        wrong[2] += __float_as_uint(ft::rn_rcp(x)) != __float_as_uint(__frcp_rn(x));
    }
    for (int k = 0; k < 3; ++k)
        if (wrong[k]) atomicAdd(bad + k, (unsigned long long)wrong[k]);
}

int main()
{
    unsigned long long *bad, host[3] = {1, 1, 1};
    if (cudaMalloc(&bad, sizeof(host)) != cudaSuccess) return 2;
    cudaMemset(bad, 0, sizeof(host));
    check<<<1216, 256>>>(0u, 0x7f800000u, bad);          // every positive finite float
    if (cudaMemcpy(host, bad, sizeof(host), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    std::printf("%llu %llu %llu\n", host[0], host[1], host[2]);
    return 0;
}
"""


def test_every_float_rounds_as_the_device_functions(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2509_10757_gb300 import build
    src, exe = tmp_path / "rn.cu", tmp_path / "rn"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc()] + build.ARCH + ["-O3", "-std=c++17", "-I" + build.CSRC, str(src), "-o", str(exe)],
                   check=True, cwd=os.fspath(tmp_path))
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["0", "0", "0"], f"square roots, their reciprocals, reciprocals that differ: {out}"
