"""Batched products and recurrent steps with blocks whose width is not 16, 32 or a multiple of 64: mma.sync, its layouts by
batch size, the wavefront of packed inputs and the fp32 buffers."""
import numpy as np
import pytest
import torch

import test_gpu_product as product
import test_gpu_rnn as rnn
import workloads
from oracle import csb_oracle as O
from paper_2005_05758_b200 import binding

pytestmark = pytest.mark.gpu

MMA = 1                                                    # csb_last_tensor_kernel


@pytest.mark.parametrize("rows,cols,br,bc", [(127, 95, 8, 8), (300, 1177, 32, 24), (513, 2049, 64, 48), (200, 330, 24, 96), (1000, 192, 50, 20)])
@pytest.mark.parametrize("batch", [8, 16, 17, 32, 33, 64, 70])
def test_product_against_the_oracle(rows, cols, br, bc, batch):
    w = workloads.make_spmv_workload(rows + cols, rows, cols, br, bc, "uniform", lo=0.2, hi=0.9, batch=batch, w_std=0.05)
    product.run_case(w.matrix, w.X)
    assert binding.lib.csb_last_tensor_kernel() == MMA


@pytest.mark.parametrize("first,captured", [(32, 64), (17, 40), (64, 20), (9, 16)])
def test_a_class_that_one_call_has_set_up_serves_a_capture(first, captured):
    mat = workloads.make_matrix(43, 640, 500, 64, 48, "uniform", lo=0.3, hi=0.9, w_std=0.1, val_dtype="f16")
    X = np.random.default_rng(6).standard_normal((64, 500)).astype(np.float32)
    A = binding.csb_encode(mat.dense, 64, 48, mat.row_keep, mat.col_keep, "f16", 0)
    Xd = torch.from_numpy(X).cuda()
    binding.csb_spmm(A, Xd[:first], torch.empty((first, 640), device="cuda"))
    Y = torch.full((captured, 640), float("nan"), device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        binding.csb_spmm(A, Xd[:captured], Y)
    assert binding.lib.csb_last_tensor_kernel() == MMA
    graph.replay()
    torch.cuda.synchronize()
    args = (mat.dense, 64, 48, mat.row_keep, mat.col_keep, "f16")
    product.check_product(Y.cpu().numpy(), O.spmm(*args, X[:captured]), O.abs_scale(*args, X[:captured]), "f16")
    del graph
    A.free()


@pytest.mark.parametrize("cell,B,I,H,L,b", [("lstm", 32, 153, 512, 2, 48), ("lstm", 9, 40, 512, 2, 24), ("lstm", 16, 40, 48, 3, 8), ("lstm", 24, 64, 200, 1, 40),
                                            ("gru", 16, 70, 512, 2, 48), ("gru", 11, 33, 512, 2, 8), ("gru", 16, 40, 60, 3, 20)])
def test_wavefront_of_packed_inputs(monkeypatch, cell, B, I, H, L, b):
    # the oracle; the bits of a sequence cut in two, of host arrays, and of the same products over fp32 buffers
    w = workloads.make_rnn_workload(33, cell, I, H, L, b, b, "lognormal", rate=4.0, T=5, B=B, w_std=0.15, bias_std=0.2, state_std=0.4)
    first = rnn.check(w)
    assert binding.lib.csb_last_recurrent_path() == 3 and binding.lib.csb_last_tensor_kernel() == MMA
    others = [rnn.run(w, chunks=[(0, 2), (2, 5)]), rnn.run(w, host_io=True)]
    monkeypatch.setenv("CSB_RNN_STEP_UNPACKED", "1")
    others.append(rnn.run(w))
    assert binding.lib.csb_last_recurrent_path() == 4 and binding.lib.csb_last_tensor_kernel() == MMA
    for other in others:
        assert all(np.array_equal(a, b) for a, b in zip(first, other) if a is not None)


@pytest.mark.parametrize("cell,B,I,H,L,b", [("lstm", 40, 70, 192, 2, 48), ("lstm", 65, 39, 100, 1, 20), ("gru", 17, 70, 96, 2, 24), ("gru", 40, 39, 100, 1, 8)])
def test_steps_over_fp32_buffers(cell, B, I, H, L, b):
    w = workloads.make_rnn_workload(35, cell, I, H, L, b, b, "lognormal", rate=4.0, T=5, B=B, w_std=0.15, bias_std=0.2, state_std=0.4)
    first = rnn.check(w)
    assert binding.lib.csb_last_recurrent_path() == 4 and binding.lib.csb_last_tensor_kernel() == MMA
    other = rnn.run(w, chunks=[(0, 2), (2, 5)])
    assert all(np.array_equal(a, b) for a, b in zip(first, other) if a is not None)
