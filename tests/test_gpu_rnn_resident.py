"""The two resident time loops (batches up to 8) at the sizes where their layouts can go wrong, against the float64
oracle: units that do not fill the last warp or CTA, odd vector lengths (values are read two or three at a
time), batches below and at a tile of columns, two and four units per warp, fp32 values, stacked layers with more
steps than a vector stays readable (32)."""
import pytest
import torch

import test_gpu_cells as cells
import test_gpu_rnn as rnn
import workloads
from paper_2005_05758_b200 import binding

pytestmark = pytest.mark.gpu

UNIT_LOOP, BLOCK_LOOP, STEPS_PACKED, STEPS, PERSISTENT, CELL_STEPS = range(1, 7)      # csb_last_recurrent_path

SIZES = [   # input, hidden, layers, block, steps, batch, values, per-block keep range
    (1, 1, 1, 8, 3, 1, "f16", (1.0, 1.0)),
    (39, 17, 2, 16, 45, 1, "f16", (0.3, 0.9)),
    (40, 161, 1, 32, 9, 3, "f16", (0.3, 0.6)),
    (33, 100, 2, 32, 41, 4, "f32", (0.3, 0.6)),
    (70, 97, 3, 16, 37, 5, "f16", (0.3, 0.6)),
    (25, 130, 1, 64, 9, 8, "f32", (0.3, 0.6)),
    (64, 1229, 2, 64, 34, 1, "f16", (0.2, 0.4)),       # past 16 units a CTA on every CTA
]


@pytest.mark.parametrize("other", [False, True])
@pytest.mark.parametrize("cell", ["lstm", "gru", "lstmp", "ligru", "gru_rb"])
@pytest.mark.parametrize("I,H,L,br,T,B,vd,keep", SIZES)
def test_edges_of_units_columns_and_exchange(monkeypatch, cell, I, H, L, br, T, B, vd, keep, other):
    if other:
        monkeypatch.setenv("CSB_RNN_NO_UNIT", "1")         # the loop for large products, on the same sizes
    if cell == "gru_rb":
        H += -H % (br // 2)                                # a whole number of block rows before the candidate's
    extra = dict(proj_size=max(1, H // 2)) if cell == "lstmp" else {}
    w = workloads.make_rnn_workload(31, cell, I, H, L, br, br, "uniform", lo=keep[0], hi=keep[1], T=T, B=B,
                                    w_std=0.5 / max(1.0, (0.1 * (I + H)) ** 0.5), val_dtype=vd, bias_std=0.1, state_std=0.5, **extra)
    (rnn if cell in ("lstm", "gru") else cells).check(w)
    # (the block loop is not built for eight columns of fp32 values: the persistent kernel or the cells' steps take those)
    want = UNIT_LOOP if not other else BLOCK_LOOP if (B, vd) != (8, "f32") else PERSISTENT if cell in ("lstm", "gru") else CELL_STEPS
    assert binding.lib.csb_last_recurrent_path() == want


@pytest.mark.parametrize("cell", ["lstm", "gru"])
@pytest.mark.parametrize("I,H,L,B,T,vd", [(40, 48, 2, 1, 11, "f16"), (39, 161, 3, 1, 9, "f32"), (70, 200, 1, 1, 1, "f16"), (33, 64, 2, 3, 9, "f16"), (25, 60, 2, 8, 5, "f32")])
def test_persistent_kernel_behind_the_resident_loops(monkeypatch, cell, I, H, L, B, T, vd):
    # what serves layers that do not fit in shared memory: at batch 1 with h exchanged as flagged values, else with grid barriers
    monkeypatch.setenv("CSB_RNN_NO_RNN1", "1")
    w = workloads.make_rnn_workload(37, cell, I, H, L, 16, 16, "uniform", lo=0.3, hi=0.9, T=T, B=B, w_std=0.1, val_dtype=vd, bias_std=0.1, state_std=0.5)
    y, h, c = rnn.check(w)
    assert binding.lib.csb_last_recurrent_path() == PERSISTENT
    if T > 4:                                              # resumed: the bits of one call
        y2, h2, c2 = rnn.run(w, chunks=[(0, 4), (4, T)])
        assert (y == y2).all() and (h == h2).all() and (c is None or (c == c2).all())


def test_layers_that_do_not_fit_take_the_persistent_kernel():
    # two layers of 1024 units with nothing pruned: 34 MB of fp16 values, past what the SMs' shared memory holds
    w = workloads.make_rnn_workload(38, "lstm", 1024, 1024, 2, 64, 64, "uniform", lo=1.0, hi=1.0, T=3, B=1, w_std=0.03, bias_std=0.1, state_std=0.5)
    rnn.check(w)
    assert binding.lib.csb_last_recurrent_path() == PERSISTENT


@pytest.mark.parametrize("other", [False, True])
@pytest.mark.parametrize("cell", ["lstm", "gru", "lstmp", "ligru", "gru_rb"])
@pytest.mark.parametrize("B,T", [(1, 1), (4, 1), (8, 1), (1, 3), (6, 3)])
def test_arrays_in_each_others_places(monkeypatch, cell, B, T, other):
    # final states in the place of the initial ones, of each other's, of x or inside y, and y in the place of x: the
    # bits have to be those of arrays of their own.  (One step exchanges nothing before the states are stored, so
    # there a CTA can be done while another has not begun to read.)
    if other:
        monkeypatch.setenv("CSB_RNN_NO_UNIT", "1")
    L, H = 2, 512
    extra = dict(proj_size=256) if cell == "lstmp" else {}
    S = extra.get("proj_size", H)
    w = workloads.make_rnn_workload(19, cell, S, H, L, 32, 32, "uniform", lo=0.2, hi=0.5, T=T, B=B, w_std=0.05, bias_std=0.1, state_std=0.5, **extra)
    encode = lambda ms: [binding.csb_encode(m.dense, m.block_r, m.block_c, m.row_keep, m.col_keep, m.val_dtype, 0) for m in ms]   # noqa: E731
    mats, proj = encode(w.layers), encode(w.proj) if cell == "lstmp" else []
    bias = [torch.from_numpy(b).cuda() for b in w.bias]
    has_c = cell in ("lstm", "lstmp")

    def call(x, h0, c0, y, hT, cT):
        if cell == "lstm":
            binding.csb_lstm_forward(mats, bias, x, h0, c0, y, hT, cT)
        elif cell == "lstmp":
            binding.csb_lstmp_forward(mats, proj, bias, x, h0, c0, y, hT, cT)
        else:
            {"gru": binding.csb_gru_forward, "ligru": binding.csb_ligru_forward, "gru_rb": binding.csb_gru_reset_before_forward}[cell](
                mats, bias, x, h0, y, hT)

    def inputs():
        # x with room behind it for what may be laid over it
        x = torch.zeros(max(w.x.size, L * B * S), device="cuda")
        x[:w.x.size] = torch.from_numpy(w.x.reshape(-1)).cuda()
        return x, torch.from_numpy(w.h0).cuda(), torch.from_numpy(w.c0).cuda() if has_c else None
    n = T * B * S
    x, h, c = inputs()
    want_y, want_h = torch.empty((T, B, S), device="cuda"), torch.empty_like(h)
    want_c = torch.empty_like(c) if has_c else None
    call(x[:n].view(T, B, S), h, c, want_y, want_h, want_c)
    places = ["in place", "over x", "y over x"] + (["crossed"] if cell == "lstm" else []) + (["in y"] if T >= L else [])
    for place in places:
        for _ in range(10 if T == 1 else 2):
            x, h, c = inputs()
            y, hT, cT = torch.empty(n, device="cuda"), torch.empty_like(h), torch.empty_like(c) if has_c else None
            if place == "in place":
                hT, cT = h, c
            elif place == "over x":
                hT = x[:h.numel()].view_as(h)
            elif place == "y over x":
                y = x[:n]
            elif place == "crossed":
                hT, cT = c, h
            elif place == "in y":
                hT = y[:h.numel()].view_as(h)
            call(x[:n].view(T, B, S), h, c, y.view(T, B, S), hT, cT)
            torch.cuda.synchronize()
            assert binding.lib.csb_last_recurrent_path() == (BLOCK_LOOP if other else UNIT_LOOP)
            skip = h.numel() if place == "in y" else 0
            assert torch.equal(hT, want_h), place
            assert torch.equal(y[skip:], want_y.view(-1)[skip:]), place
            assert not has_c or torch.equal(cT, want_c), place
    for m in mats + proj:
        m.free()


@pytest.mark.parametrize("other", [False, True])
@pytest.mark.parametrize("B1,B2", [(3, 4), (5, 8)])
def test_batch_sizes_of_one_tile_may_overlap(monkeypatch, B1, B2, other):
    # calls on the same matrices with different batch sizes have exchange buffers and step numbers of their own, also
    # where both sizes run on the same tile of columns: queued on two streams at once they give the bits of calls in turn
    if other:
        monkeypatch.setenv("CSB_RNN_NO_UNIT", "1")
    L, I, H, T = 2, 40, 160, 150
    ws = [workloads.make_rnn_workload(23, "lstm", I, H, L, 32, 32, "uniform", lo=0.3, hi=0.6, T=T, B=B, w_std=0.1, bias_std=0.1, state_std=0.5) for B in (B1, B2)]
    mats = [binding.csb_encode(m.dense, m.block_r, m.block_c, m.row_keep, m.col_keep, m.val_dtype, 0) for m in ws[0].layers]
    bias = [torch.from_numpy(b).cuda() for b in ws[0].bias]
    args = [[torch.from_numpy(a).cuda() for a in (w.x, w.h0, w.c0)] for w in ws]

    def outputs():
        return [[torch.zeros((T, w.B, H), device="cuda"), torch.zeros((L, w.B, H), device="cuda"), torch.zeros((L, w.B, H), device="cuda")] for w in ws]
    want = outputs()
    for a, o in zip(args, want):
        binding.csb_lstm_forward(mats, bias, *a, *o)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(5):
        got = outputs()
        torch.cuda.synchronize()
        for a, o, st in zip(args, got, streams):
            binding.csb_lstm_forward(mats, bias, *a, *o, binding.CSB_FLAG_ASYNC, stream=st)
        torch.cuda.synchronize()
        for g, v in zip(got, want):
            assert all(torch.equal(p, q) for p, q in zip(g, v))
    for m in mats:
        m.free()
