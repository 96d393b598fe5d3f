"""No exception crosses the C boundary and nothing ends the process when host memory runs out, also in the planners'
threads: every host-side piece is run with all allocations failing from the n-th on, for n from the first few to many."""
import os
import subprocess

import pytest

from paper_2005_05758_b200 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("oom") / "out_of_memory")
    lib = os.path.dirname(build.LIB)
    subprocess.run([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-o", out, os.path.join(HERE, "out_of_memory.cpp"), "-L" + lib, "-lcsb", "-lpthread",
                    "-Wl,-rpath," + lib], check=True)
    return out


@pytest.mark.parametrize("piece", ["encode", "stream plan", "panel plan", "batched plan", "unit loop plan", "block loop plan"])
def test_running_out_of_host_memory_is_a_status(program, piece):
    which = ["encode", "stream plan", "panel plan", "batched plan", "unit loop plan", "block loop plan"].index(piece)
    steps = list(range(0, 12)) + [int(14 * 1.5 ** k) for k in range(18)]
    ended = {n: subprocess.run([program, str(which), str(n)], stderr=subprocess.DEVNULL, timeout=60).returncode for n in steps}
    assert not any(ended.values()), ended
