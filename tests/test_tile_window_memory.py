"""Plans of the batched product on tcgen05 when device memory runs out, or another call fails, at any point of their set-up
(tile_window_memory.cpp, on the CPU with a CUDA runtime of its own)."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2005_05758_b200", "csrc")
CUDA = os.path.join(os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))), "include")


def test_a_plan_is_whole_or_absent(tmp_path):
    out = str(tmp_path / "tile_window_memory")
    subprocess.run([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-pthread", "-I" + CUDA, "-o", out, os.path.join(HERE, "tile_window_memory.cpp")] +
                   [os.path.join(CSRC, f) for f in ("csb_umma_upload.cpp", "csb_umma_plan.cpp", "csb_encode.cpp")], check=True)
    res = subprocess.run([out], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout
