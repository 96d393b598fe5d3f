"""The resident time loops' own tanh and logistic function (csb_rnn_exchange.cuh): the polynomial is the fit that its
comment names, and both functions keep the stated error over the whole range of fp32 inputs."""
import os
import re

import numpy as np
import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2005_05758_b200", "csrc", "csb_rnn_exchange.cuh")
SWITCH = 0.625


def test_the_polynomial_is_the_stated_fit():
    body = open(SOURCE).read().split("float activation(")[1].split("return")[0]
    assert float(re.search(r"ax < ([\d.]+)f \?", body).group(1)) == SWITCH
    found = [np.float32(v) for v in re.findall(r"(-?\d\.\d{10,})f", body)]           # degree 4 first, then 3 .. 0
    n = 200
    s = 0.5 * SWITCH ** 2 * (1 - np.cos(np.pi * (np.arange(n) + 0.5) / n))
    x = np.sqrt(s)
    y = (np.tanh(x) / x - 1) / s
    y[s < 1e-3] = np.polyval([-1382 / 155925, 62 / 2835, -17 / 315, 2 / 15, -1 / 3], s[s < 1e-3])   # the series, where the quotient cancels
    fit = np.polynomial.chebyshev.Chebyshev.fit(s, y, 4, domain=[0, SWITCH ** 2]).convert(kind=np.polynomial.Polynomial).coef
    assert np.allclose(found, fit[[4, 3, 2, 1, 0]], rtol=2e-7)
    t = np.linspace(1e-4, SWITCH, 100001)
    err = np.abs(t + t ** 3 * np.polyval(np.float64(found), t * t) - np.tanh(t)) / np.spacing(np.tanh(t).astype(np.float32))
    assert err.max() < 0.2


def ulps(got, want):
    return np.abs(got.astype(np.float64) - want) / np.spacing(np.abs(want).astype(np.float32)).astype(np.float64)


@pytest.mark.gpu
@pytest.mark.parametrize("other", [False, True])
def test_error_over_the_whole_range(monkeypatch, other):
    # through cells whose output is the bare function of a bias: a light GRU with candidate 0 and h0 = 1 gives the
    # logistic function, a GRU with a closed update gate tanh
    import torch
    from paper_2005_05758_b200 import binding
    if other:
        monkeypatch.setenv("CSB_RNN_NO_UNIT", "1")
    H, rng = 1024, np.random.default_rng(4)
    mags = np.exp(rng.uniform(np.log(1e-30), np.log(120.0), 20 * H)).astype(np.float32)
    near = np.concatenate([rng.uniform(0.0, 1.5, 20 * H), rng.uniform(1.5, 20.0, 20 * H)]).astype(np.float32)
    edge = (np.float32(SWITCH).view(np.uint32) + np.arange(-H // 2, H // 2)).astype(np.uint32).view(np.float32)
    odd = np.array([0.0, 1e-45, 1e-38, 86.0, 87.5, 88.5, 89.0, 103.0, 104.5, 1e30, 3e38, np.inf], np.float32)
    x = np.concatenate([mags, near, edge, np.resize(odd, H)])
    x = np.concatenate([x, -x]).reshape(-1, H)

    def sweep(cell):
        rows = {"ligru": 2, "gru": 3}[cell] * H
        nblk = rows // 64 * (-(-(1 + H) // 64))
        A = binding.csb_encode(np.zeros((rows, 1 + H), np.float32), 64, 64, np.ones(nblk * 64, np.uint8), np.ones(nblk * 64, np.uint8), "f16", 0)
        one = torch.zeros((1, 1, 1), device="cuda")
        h0 = torch.full((1, 1, H), 1.0 if cell == "ligru" else 0.0, device="cuda")
        out = torch.empty((len(x), 1, 1, H), device="cuda")
        for i, v in enumerate(torch.from_numpy(x).cuda()):
            if cell == "ligru":
                binding.csb_ligru_forward([A], [torch.cat([v, torch.full_like(v, -1.0)])], one, h0, out[i], None)
            else:
                zero = torch.zeros_like(v)
                binding.csb_gru_forward([A], [torch.cat([zero, zero - 1000.0, v, zero])], one, h0, out[i], None)
        torch.cuda.synchronize()
        nan = torch.full((4 * H if cell == "gru" else 2 * H,), float("nan"), device="cuda")
        y = torch.zeros((1, 1, H), device="cuda")
        {"ligru": binding.csb_ligru_forward, "gru": binding.csb_gru_forward}[cell]([A], [nan], one, h0, y, None)
        torch.cuda.synchronize()
        assert bool(torch.isnan(y).all())
        A.free()
        return out.cpu().numpy().reshape(x.shape)

    x64 = x.astype(np.float64)
    with np.errstate(over="ignore"):
        logistic, th = sweep("ligru"), sweep("gru")
        e_log = ulps(logistic, 1.0 / (1.0 + np.exp(-x64)))
        e_th = ulps(th, np.tanh(x64))
    low = np.abs(x) < SWITCH
    print("logistic %.3f, tanh below the switch %.3f, above %.3f units in the last place" % (e_log.max(), e_th[low].max(), e_th[~low].max()))
    # the bounds are those of a sweep over every seventh fp32 number (0.828, 2.084, 3.460), rounded up
    assert e_log.max() < 3.5 and e_th[low].max() < 0.85 and e_th[~low].max() < 2.1
