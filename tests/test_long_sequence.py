"""Sequences of more steps than the resident time loops count are not theirs (host side only)."""
import os
import subprocess

from paper_2005_05758_b200 import build


def test_a_sequence_past_31_bits_is_left_to_the_step_by_step_path(tmp_path):
    lib, out = os.path.dirname(build.LIB), str(tmp_path / "long_sequence")
    source = os.path.join(os.path.dirname(os.path.abspath(__file__)), "long_sequence.cpp")
    subprocess.run([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-o", out, source, "-L" + lib, "-lcsb", "-Wl,-rpath," + lib], check=True)
    assert subprocess.run([out], capture_output=True, text=True, timeout=60).stdout.strip() == "1"
