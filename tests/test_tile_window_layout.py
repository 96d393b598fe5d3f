"""The layout of the batched product on tcgen05, decoded on the CPU for odd sizes, block shapes, column ranges and the gate
order of recurrent layers (tile_window_layout.cpp)."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2005_05758_b200", "csrc")


def test_every_value_at_its_place(tmp_path):
    out = str(tmp_path / "tile_window_layout")
    subprocess.run([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-pthread", "-o", out, os.path.join(HERE, "tile_window_layout.cpp"),
                    os.path.join(CSRC, "csb_umma_plan.cpp"), os.path.join(CSRC, "csb_encode.cpp")], check=True)
    res = subprocess.run([out], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout
