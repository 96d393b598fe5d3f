"""What the batched time loop cannot serve is left to the step-by-step form (batched_fallbacks.cpp, on the CPU with a CUDA
runtime of its own)."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2005_05758_b200", "csrc")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def test_the_time_loop_leaves_what_it_cannot_serve(tmp_path):
    out, objects = str(tmp_path / "batched_fallbacks"), []
    for name in ("csb_umma_rnn", "csb_rnn_step"):
        objects.append(str(tmp_path / (name + ".o")))
        subprocess.run([NVCC, "-gencode", "arch=compute_100a,code=sm_100a", "-O1", "-std=c++17", "-c", "-o", objects[-1], os.path.join(CSRC, name + ".cu")], check=True)
    subprocess.run([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", "-pthread", "-I" + os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include"), "-o", out,
                    os.path.join(HERE, "batched_fallbacks.cpp")] + objects + [os.path.join(CSRC, f) for f in ("csb_umma_upload.cpp", "csb_umma_plan.cpp", "csb_encode.cpp")], check=True)
    res = subprocess.run([out], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout
