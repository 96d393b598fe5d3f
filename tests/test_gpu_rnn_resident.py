"""The two resident time loops (batches up to 8) at the sizes where their layouts can go wrong, against the float64
oracle: units that do not fill the last warp or CTA, odd vector lengths (values are read two or three at a
time), batches below and at a tile of columns, two and four units per warp, fp32 values, stacked layers with more
steps than a vector stays readable (32)."""
import pytest

import test_gpu_cells as cells
import test_gpu_rnn as rnn
import workloads

pytestmark = pytest.mark.gpu

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
