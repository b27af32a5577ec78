"""The first step of a problem is launched plainly and its graph built behind
it: a graph that cannot be built must not turn the step, which has run, into an
error (a second call would advance the state again), and must not be built
before a launch has succeeded (host build with fakes; no GPU needed)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
OK = 0


def test_step_order(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "step_order_check")
    subprocess.run([gxx, "-std=c++17", "-O1", "-o", exe, os.path.join(HERE, "native", "step_order_check.cpp")], check=True,
                   capture_output=True)
    out = {}
    for line in subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split("\n"):
        if line:
            name, *v = line.split()
            out[name] = tuple(map(int, v))
    # status, plain launches, attempts to build the graph, graph launches, steps taken
    assert out["ordinary"] == (OK, 1, 1, 2, 3)
    assert out["no_graph"] == (OK, 2, 2, 0, 2)
    assert out["graph_later"] == (OK, 3, 3, 1, 4)
    assert out["not_capturable"][1:] == (0, 1, 0, 0) and out["not_capturable"][0] != OK
    assert out["launch_fails"][1:] == (1, 0, 0, 0) and out["launch_fails"][0] != OK
