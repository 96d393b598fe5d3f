"""The block loop's planner refuses what does not fit, and only that, before it emits anything (host side only)."""
import os
import subprocess

from paper_2005_05758_b200 import build


def test_the_planner_turns_away_what_does_not_fit_and_only_that(tmp_path):
    lib, out = os.path.dirname(build.LIB), str(tmp_path / "block_loop_limit")
    source = os.path.join(os.path.dirname(os.path.abspath(__file__)), "block_loop_limit.cpp")
    subprocess.run([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-o", out, source, "-L" + lib, "-lcsb", "-Wl,-rpath," + lib], check=True)
    done = subprocess.run([out], capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stdout
