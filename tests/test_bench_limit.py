"""A part of the benchmark that hangs costs its own result and no other."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run(body):
    code = ("import json, time, bench\nline = {'value': 1}\n"
            "def finish(x):\n    line['served'] = x\n    print(json.dumps(line), flush=True)\n" + body)
    return subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=60)


def test_the_line_comes_without_a_part_that_hangs():
    r = run("def hang():\n    time.sleep(50)\nbench.within(1.0, hang, finish)\n")
    assert r.returncode == 0
    lines = r.stdout.splitlines()
    assert len(lines) == 1
    got = json.loads(lines[0])
    assert got["value"] == 1 and "not ended after 1 s" in got["served"]["unavailable"]
    assert "hang" in r.stderr                # the stacks name it


def test_the_line_comes_once_with_a_part_that_ends():
    r = run("bench.within(1.0, lambda: {'x': 2}, finish)\ntime.sleep(1.5)\n")
    assert r.returncode == 0 and [json.loads(x) for x in r.stdout.splitlines()] == [{"value": 1, "served": {"x": 2}}]
