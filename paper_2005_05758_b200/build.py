"""Build libcsb.so in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import concurrent.futures
import os
import subprocess
import sys
import sysconfig
import tempfile

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libcsb.so")
SOURCES = ["csb_api.cpp", "csb_encode.cpp", "csb_plan.cpp", "csb_schedule.cpp", "csb_spmm_plan.cpp", "csb_panel_plan.cpp", "csb_product.cu", "csb_panel.cu", "csb_spmm_mma.cu", "csb_umma_plan.cpp", "csb_umma_upload.cpp", "csb_umma.cu", "csb_umma_rnn.cu", "csb_rnn.cu", "csb_rnn_step.cu", "csb_rnn1_plan.cpp", "csb_rnn1.cu", "csb_rnn1_b1.cu", "csb_rnn1_b4.cu", "csb_rnn1_b8.cu", "csb_rnn_unit_plan.cpp", "csb_rnn_unit_b1.cu", "csb_rnn_unit_b4.cu", "csb_rnn_unit_b8.cu", "csb_cells.cu", "csb_fixed.cu", "csb_project.cu"]
HEADERS = ["csb_internal.hpp", "csb_umma.hpp", "csb_umma_kernel.cuh", "csb_umma_rnn.hpp", "csb_host.hpp", "csb_device.cuh", "csb_rnn1.hpp", "csb_rnn1_args.hpp", "csb_rnn1_kernel.cuh", "csb_rnn_unit.hpp", "csb_rnn_unit_kernel.cuh", "csb_rnn_exchange.cuh", "csb_gates.cuh", os.path.join("..", "..", "include", "csb.h")]


PY_MODULE = os.path.join(HERE, "_csb_py" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))


def build_py_module() -> str:
    """Compile the marshalling module (a CPython extension, plain C) if it is missing or older than its source."""
    src = os.path.join(CSRC, "csb_py.c")
    if not os.path.exists(PY_MODULE) or os.path.getmtime(PY_MODULE) < os.path.getmtime(src):
        res = subprocess.run([os.environ.get("CC", "gcc"), "-O2", "-fPIC", "-shared", "-I" + sysconfig.get_paths()["include"], "-o", PY_MODULE, src],
                             capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError("gcc failed:\n" + res.stdout + res.stderr)
    return PY_MODULE


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, f) for f in SOURCES + HEADERS]
    return any(os.path.getmtime(d) > t for d in deps if os.path.exists(d))


#: Instrumented variants (never the default build).  CSB_PHASE_CLOCKS makes the time-loop kernel sum
#: clock64() cycles per phase and CTA (read back with csb_debug_rnn_clocks); CSB_PANEL_CLOCKS makes
#: the SpMV panel kernel record wall-clock stamps per phase and CTA (csb_debug_panel_clocks);
#: CSB_SPMM_CLOCKS makes the batched tensor-core kernel sum cycles per phase and warp (csb_debug_spmm_clocks).
#: paper_2005_05758_b200/phase_clocks.py builds such a library beside the normal one and prints the figures.
INSTRUMENT_DEFINES = ("CSB_PHASE_CLOCKS", "CSB_PANEL_CLOCKS", "CSB_SPMM_CLOCKS")


def build(force: bool = False, verbose: bool = False, defines=(), out: str = None) -> str:
    """Compile the library if it is missing or older than its sources; return its path.
    `defines` adds -D switches (see INSTRUMENT_DEFINES) and then needs `out`, the path of the
    instrumented library, so that the normal libcsb.so is never replaced by one."""
    if defines and not out:
        raise ValueError("an instrumented build needs its own output path")
    build_py_module()
    if not defines and not force and not _stale():
        return LIB
    nvcc = [os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-Xcompiler", "-fPIC"]
    flags = ["-lineinfo", "-O3", "-std=c++17"] + ["-D" + d for d in defines] + (["-Xptxas", "-v"] if verbose else [])

    def run(cmd):
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
        if verbose:
            sys.stderr.write(res.stderr)

    # one object per source, compiled side by side
    with tempfile.TemporaryDirectory() as tmp:
        objects = [os.path.join(tmp, f + ".o") for f in SOURCES]
        with concurrent.futures.ThreadPoolExecutor(os.cpu_count() or 1) as pool:
            list(pool.map(run, [nvcc + flags + ["-c", "-o", o, os.path.join(CSRC, f)] for f, o in zip(SOURCES, objects)]))
        run(nvcc + ["-shared", "-o", out or LIB] + objects)
    return out or LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
