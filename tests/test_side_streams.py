"""The helper streams of the forward, on the CPU: `csrc/pq_side.cuh` is host code, compiled here against a stand-in for the runtime's
streams and events (side_streams_check.cpp)."""
import os
import subprocess

import pytest

from paper_2602_22592_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = tmp_path_factory.mktemp("side") / "check"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", build.CSRC, "-isystem", cuda, os.path.join(HERE, "side_streams_check.cpp"),
                    "-o", str(exe)], check=True)

    def run(what):
        res = subprocess.run([str(exe), what], capture_output=True, text=True, timeout=120)
        assert res.returncode == 0, res.stderr
    return run


@pytest.mark.parametrize("what", ["per_thread", "ended_threads", "handles", "plain_order", "small_calls", "failed_calls"])
def test_helper_streams(check, what):
    check(what)
