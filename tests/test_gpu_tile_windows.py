"""The batched product and time loop on tcgen05 at the sizes where their tiles, windows and batch tiles end."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

import workloads
from oracle import csb_oracle as O
from oracle import rnn_oracle as R
from paper_2005_05758_b200 import binding

pytestmark = pytest.mark.gpu

TILES, LOOP = 2, 3                                         # csb_last_tensor_kernel

# Error of an output in units of sum |w| |x|: the split x = hi + lo (2^-22), a chain of at most 8 truncated sums in the
# tensor cores (2^-23 each), then one rounded sum per flush group and column range, at most 64 here (2^-24 each).
TOL = 2.0 ** -22 + 8 * 2.0 ** -23 + 64 * 2.0 ** -24


@pytest.mark.parametrize("rows,cols,br,bc,batch", [(1, 1, 16, 16, 8), (127, 63, 32, 32, 9), (129, 65, 16, 16, 17), (300, 1177, 32, 32, 33),
                                                   (513, 2049, 64, 64, 64), (200, 130, 64, 128, 65), (70, 4200, 24, 64, 16), (1000, 192, 50, 32, 32)])
def test_product_against_the_oracle(rows, cols, br, bc, batch):
    w = workloads.make_spmv_workload(rows + cols, rows, cols, br, bc, "uniform", lo=0.3, hi=0.9, batch=batch, w_std=0.05)
    m = w.matrix
    A = binding.csb_encode(m.dense, br, bc, m.row_keep, m.col_keep, "f16", 0)
    args = (m.dense, br, bc, m.row_keep, m.col_keep, "f16")
    want, scale = O.spmm(*args, w.X), O.abs_scale(*args, w.X)
    for pad in (0, 3):                                   # rows of x and y with and without 16-byte alignment
        x = torch.full((batch, cols + pad), float("nan"), device="cuda")
        x[:, :cols] = torch.from_numpy(w.X).cuda()
        y = torch.full((batch, rows + pad), float("nan"), device="cuda")
        binding.csb_spmm(A, x[:, :cols], y[:, :rows])
        torch.cuda.synchronize()
        got = y.cpu().numpy()
        assert np.all(np.abs(got[:, :rows] - want) <= TOL * scale)
        assert binding.lib.csb_last_tensor_kernel() == TILES
        assert np.isnan(got[:, rows:]).all()
    A.free()


@pytest.mark.parametrize("cell,B,I,H,L,T", [("lstm", 16, 39, 100, 3, 5), ("lstm", 31, 1, 33, 1, 4), ("gru", 32, 70, 96, 2, 5), ("gru", 17, 153, 160, 1, 1)])
def test_time_loop_against_the_oracle(cell, B, I, H, L, T):
    w = workloads.make_rnn_workload(61, cell, I, H, L, 32, 32, "uniform", lo=0.3, hi=0.8, T=T, B=B, w_std=0.15, bias_std=0.2, state_std=0.4)
    mats = [binding.csb_encode(m.dense, m.block_r, m.block_c, m.row_keep, m.col_keep, m.val_dtype, 0) for m in w.layers]
    lay = [(m.dense, m.block_r, m.block_c, m.row_keep, m.col_keep, m.val_dtype) for m in w.layers]
    x, h0, bias = torch.from_numpy(w.x).cuda(), torch.from_numpy(w.h0).cuda(), [torch.from_numpy(b).cuda() for b in w.bias]
    y, hT = torch.full((T, B, H), float("nan"), device="cuda"), torch.full((L, B, H), float("nan"), device="cuda")

    def run():
        if cell == "gru":
            binding.csb_gru_forward(mats, bias, x, h0, y, hT, 0)
        else:
            binding.csb_lstm_forward(mats, bias, x, h0, torch.from_numpy(w.c0).cuda(), y, hT, None, 0)
    run()
    assert binding.lib.csb_last_tensor_kernel() == LOOP
    want = R.gru_forward(lay, w.bias, w.x, w.h0) if cell == "gru" else R.lstm_forward(lay, w.bias, w.x, w.h0, w.c0)
    # fp32 sums of fp16 weights: an absolute error of 1e-6 of a pre-activation of size 1 a step (TOL and the activations'), which
    # the recurrence carries on; 5 steps of up to 3 layers
    for got, ref in ((y, want[0]), (hT, want[1])):
        assert np.max(np.abs(got.cpu().numpy() - np.asarray(ref))) < 15 * 2e-6
    if T > 1:
        # a wait that runs out is a status, and the next call is as good as the first
        binding.lib.csb_test_barrier_hook(1, 200_000)
        try:
            with pytest.raises(binding.CsbError) as e:
                run()
            assert e.value.status == -7
        finally:
            binding.lib.csb_test_barrier_hook(0, 0)
        y.fill_(float("nan"))
        run()
        assert np.max(np.abs(y.cpu().numpy() - np.asarray(want[0]))) < 15 * 2e-6
    for m in mats:
        m.free()


@pytest.mark.parametrize("rows,cols,batch", [(200, 100, 9), (1024, 512, 16), (4096, 8192, 64)])
def test_time_in_front_of_a_product_does_not_count(tmp_path, rows, cols, batch):
    # the product's CTAs may start while the kernel in front runs (here past the limit of the product's own waits, a
    # second): with one round a CTA, with two, and with more than its rings hold
    here = os.path.dirname(os.path.abspath(__file__))
    out = str(tmp_path / "slow_front.so")
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-O2", "-shared", "-Xcompiler", "-fPIC", "-o", out,
                    os.path.join(here, "slow_front.cu")], check=True)
    w = workloads.make_spmv_workload(3, rows, cols, 32, 64, "uniform", lo=0.3, hi=0.9, batch=batch, w_std=0.05)
    m = w.matrix
    A = binding.csb_encode(m.dense, 32, 64, m.row_keep, m.col_keep, "f16", 0)
    x = torch.from_numpy(w.X).cuda()
    want, y = torch.empty((batch, rows), device="cuda"), torch.full((batch, rows), float("nan"), device="cuda")
    binding.csb_spmm(A, x, want)
    torch.cuda.synchronize()
    assert ctypes.CDLL(out).slow_front(ctypes.c_ulonglong(1_300_000_000), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    binding.csb_spmm(A, x, y)
    torch.cuda.synchronize()
    assert torch.equal(y, want)
    binding.csb_spmm(A, x, y)                            # (reports a wait that an earlier product gave up)
    A.free()


@pytest.mark.parametrize("I,H,L", [(153, 160, 1), (39, 100, 3), (512, 1024, 2)])
@pytest.mark.parametrize("step", [0, 1, 3])
def test_one_warp_that_gives_up_takes_the_sequence_along(I, H, L, step):
    # the warps that pack x_{t+1} give up at one step, everybody else has what that step needs: the call ends with the status,
    # and the next one is as good as the first
    T, B = 6, 20
    w = workloads.make_rnn_workload(7, "lstm", I, H, L, 32, 32, "uniform", lo=0.2, hi=0.5, T=T, B=B, w_std=0.1, bias_std=0.1, state_std=0.3)
    mats = [binding.csb_encode(m.dense, m.block_r, m.block_c, m.row_keep, m.col_keep, m.val_dtype, 0) for m in w.layers]
    x, bias, y = torch.from_numpy(w.x).cuda(), [torch.from_numpy(b).cuda() for b in w.bias], torch.empty((T, B, H), device="cuda")

    def run():
        binding.csb_lstm_forward(mats, bias, x, None, None, y, None, None, 0)
        return y.clone()
    want = run()
    binding.lib.csb_test_barrier_hook(2 + step, 200_000)
    try:
        with pytest.raises(binding.CsbError) as e:
            run()
        assert e.value.status == -7
    finally:
        binding.lib.csb_test_barrier_hook(0, 0)
    assert torch.equal(run(), want)
    for m in mats:
        m.free()


def kept(m):
    """[rows, cols]: is the weight stored?"""
    nbr, nbc = -(-m.rows // m.block_r), -(-m.cols // m.block_c)
    both = m.row_keep.reshape(nbr, nbc, m.block_r, 1).astype(bool) & m.col_keep.reshape(nbr, nbc, 1, m.block_c).astype(bool)
    return both.transpose(0, 2, 1, 3).reshape(nbr * m.block_r, nbc * m.block_c)[:m.rows, :m.cols]


LARGE = [float("nan"), float("inf"), -float("inf"), 65520.0, -1e30]


@pytest.mark.parametrize("rows,cols,br,bc,batch", [(127, 63, 32, 32, 9), (300, 1177, 16, 16, 17), (513, 2049, 64, 64, 64), (200, 130, 24, 128, 70), (4096, 700, 32, 32, 8),
                                                   (8192, 1000, 64, 64, 33), (130, 2100, 64, 64, 40)])
def test_an_input_past_binary16_touches_the_rows_that_keep_it(rows, cols, br, bc, batch):
    # NaN where a block keeps the column for the row, and the bits of the same inputs without it everywhere else
    w = workloads.make_spmv_workload(rows + cols, rows, cols, br, bc, "uniform", lo=0.1, hi=0.6, batch=batch, w_std=0.05)
    m = w.matrix
    A = binding.csb_encode(m.dense, br, bc, m.row_keep, m.col_keep, "f16", 0)
    rng = np.random.default_rng(rows)
    for n in (1, 5, batch * cols // 3):
        bad = np.zeros((batch, cols), bool)
        bad.reshape(-1)[rng.choice(batch * cols, n, replace=False)] = True
        bad[batch - 1, cols - 1] = True
        clean, x = np.where(bad, np.float32(0), w.X), w.X.copy()
        x[bad] = np.resize(np.array(LARGE, np.float32), int(bad.sum()))
        got, want = torch.empty((batch, rows), device="cuda"), torch.empty((batch, rows), device="cuda")
        binding.csb_spmm(A, torch.from_numpy(x).cuda(), got)
        binding.csb_spmm(A, torch.from_numpy(clean).cuda(), want)
        torch.cuda.synchronize()
        got, want, hit = got.cpu().numpy(), want.cpu().numpy(), bad.astype(np.float32) @ kept(m).T.astype(np.float32) > 0
        assert np.array_equal(np.isnan(got), hit) and np.array_equal(got[~hit], want[~hit])
    x = torch.from_numpy(w.X).cuda()
    x[0, 0], x[batch - 1, cols - 1] = 65519.0, -65504.0          # binary16 still holds these
    y = torch.empty((batch, rows), device="cuda")
    binding.csb_spmm(A, x, y)
    assert torch.isfinite(y).all()
    A.free()


@pytest.mark.parametrize("cell,B,I,H,L,br", [("lstm", 16, 39, 100, 3, 32), ("lstm", 32, 70, 96, 1, 16), ("gru", 17, 70, 96, 2, 32), ("gru", 32, 153, 160, 1, 64), ("lstm", 40, 39, 64, 2, 16),
                                             ("gru", 40, 39, 64, 2, 32), ("lstm", 20, 600, 512, 2, 64)])
def test_an_input_past_binary16_spreads_through_a_sequence_where_it_is_kept(cell, B, I, H, L, br):
    T = 5
    w = workloads.make_rnn_workload(61, cell, I, H, L, br, br, "uniform", lo=0.05, hi=0.3, T=T, B=B, w_std=0.15, bias_std=0.2, state_std=0.4)
    mats = [binding.csb_encode(m.dense, m.block_r, m.block_c, m.row_keep, m.col_keep, m.val_dtype, 0) for m in w.layers]
    bias = [torch.from_numpy(b).cuda() for b in w.bias]
    rng = np.random.default_rng(B)
    x, h0 = w.x.copy(), w.h0.copy()
    # sequence 0 stays clean, 1 gets one at the start, 2 at the end, 3 in an upper state, 4 in the second step, 5 everywhere
    bad_x, bad_h = np.zeros(x.shape, bool), np.zeros(h0.shape, bool)
    bad_x[0, 1, rng.integers(I)] = bad_x[T - 1, 2, rng.integers(I)] = bad_x[1, 4, rng.integers(I)] = bad_h[L - 1, 3, rng.integers(H)] = True
    bad_x[:, 5] = True
    x[bad_x], h0[bad_h] = 0, 0

    def run(x, h0):
        y, hT, cT = (torch.full(s, float("nan"), device="cuda") for s in ((T, B, H), (L, B, H), (L, B, H)))
        if cell == "gru":
            binding.csb_gru_forward(mats, bias, torch.from_numpy(x).cuda(), torch.from_numpy(h0).cuda(), y, hT, 0)
            cT.zero_()
        else:
            binding.csb_lstm_forward(mats, bias, torch.from_numpy(x).cuda(), torch.from_numpy(h0).cuda(), torch.from_numpy(w.c0).cuda(), y, hT, cT, 0)
        return [t.cpu().numpy() for t in (y, hT, cT)]
    want = run(x, h0)
    assert all(np.isfinite(a).all() for a in want) and binding.lib.csb_last_tensor_kernel() == (LOOP if B <= 32 else TILES)
    x[bad_x], h0[bad_h] = np.resize(np.array(LARGE, np.float32), int(bad_x.sum())), np.float32("inf") if cell == "lstm" else np.float32("nan")
    got = run(x, h0)
    K = [kept(m).astype(np.float32) for m in w.layers]
    h, c, top = bad_h.copy(), np.zeros((L, B, H), bool), np.zeros((T, B, H), bool)
    for t in range(T):
        u = bad_x[t]
        for l in range(L):
            z = (np.concatenate([u, h[l]], 1).astype(np.float32) @ K[l].T > 0).reshape(B, -1, H)
            if cell == "lstm":
                c[l] |= z[:, 0] | z[:, 1] | z[:, 2]
                h[l] = c[l] | z[:, 3]
            else:
                h[l] |= z[:, 0] | z[:, 1] | z[:, 2]
            u = h[l]
        top[t] = u
    for a, b, hit in zip(got, want, (top, h, c)):
        assert np.array_equal(np.isnan(a), hit) and np.array_equal(a[~hit], b[~hit])
    assert top.any() and not top[:, 0].any()
    for a, b in zip(run(np.where(bad_x, np.float32(0), x), np.where(bad_h, np.float32(0), h0)), want):       # nothing stays behind
        assert np.array_equal(a, b)
    for m in mats:
        m.free()


def test_more_ctas_than_the_device_holds_are_not_asked_for():
    # csb_plan_opts may name any number of CTAs; eight layers of 640 units would then make a grid of 160
    w = workloads.make_rnn_workload(31, "lstm", 640, 640, 8, 32, 32, "uniform", lo=0.2, hi=0.5, T=2, B=16, w_std=0.05)
    outs = []
    for ctas in (0, 400):
        opts = dict(ctas=ctas, warps_per_cta=0, stage_bytes=0, stages=0)
        mats = [binding.csb_encode(m.dense, 32, 32, m.row_keep, m.col_keep, "f16", 0, opts) for m in w.layers]
        y = torch.full((2, 16, 640), float("nan"), device="cuda")
        binding.csb_lstm_forward(mats, None, torch.from_numpy(w.x).cuda(), None, None, y, None, None, 0)
        outs.append(y)
        for m in mats:
            m.free()
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("rows,cols,br,bc,rate", [(513, 2049, 64, 64, 2.5), (70, 4200, 64, 64, 3.0), (512, 4096, 64, 64, 4.0), (1024, 2049, 64, 64, 25.0), (512, 4096, 32, 32, 9.0),
                                                  (2048, 4096, 64, 128, 9.0), (4096, 4096, 64, 64, 25.0), (8192, 3072, 64, 64, 25.0), (1024, 1536, 16, 16, 4.0)])
def test_the_error_is_no_larger_than_that_of_mma_sync(monkeypatch, rows, cols, br, bc, rate):
    # 2-norm of the error against 64 bits over that of the result; 3 % is what other inputs of the same size change
    f = rate ** -0.5
    w = workloads.make_spmv_workload(rows, rows, cols, br, bc, "uniform", lo=0.7 * f, hi=min(1.0, 1.3 * f), batch=64, w_std=0.05)
    m = w.matrix
    A = binding.csb_encode(m.dense, br, bc, m.row_keep, m.col_keep, "f16", 0)
    x = torch.from_numpy(w.X).cuda()
    want = x.double() @ torch.from_numpy(np.where(kept(m), m.dense.astype(np.float16), np.float16(0))).cuda().double().T
    for batch in (8, 32, 64):
        err = {}
        for other in ("1", "0"):
            monkeypatch.setenv("CSB_NO_UMMA", other)
            y = torch.empty((batch, rows), device="cuda")
            binding.csb_spmm(A, x[:batch], y)
            assert binding.lib.csb_last_tensor_kernel() == (1 if other == "1" else TILES)
            err[other] = float((y.double() - want[:batch]).norm() / want[:batch].norm())
        assert err["0"] <= 1.03 * err["1"] and err["0"] < 2e-7, err
    A.free()
