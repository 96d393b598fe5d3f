"""What is timed: the library's public entry points on the work that a user has them do.

The paper's own data and trained weights are not available, so weights, keep masks and inputs are
drawn: layer shapes of its benchmark models and of this repository's configurations, blocks of
16 / 32 / 64, pruning rates of 3.5x to 25x, per-block keep fractions that are uniform (a trained
recurrent layer) or lognormal (uneven blocks).  Everything comes from the seed, drawn on the GPU.

Five kinds of pass:
  product   csb_spmv (batch 1) / csb_spmm: one product of an encoded matrix with one or more vectors
  rnn       csb_lstm_forward / csb_gru_forward: a whole sequence through a stack of layers
  cell      csb_lstmp_forward / csb_ligru_forward / csb_gru_reset_before_forward
  fixed     csb_spmm_q16: the 16-bit fixed-point product
  project   csb_project: keep masks of a dense weight (one projection step of a pruning run)
Encoding is part of what a program has done before the call: it happens once per model.
"""
import math

import numpy as np
import torch

from paper_2005_05758_b200 import binding

GATES = {"lstm": 4, "gru": 3, "lstmp": 4, "ligru": 2, "gru_rb": 3}
BIAS = {"lstm": 4, "gru": 4, "lstmp": 4, "ligru": 2, "gru_rb": 3}
SIGMA = 0.8            # spread of the lognormal keep fractions
FIXED_W, FIXED_X = 16, 12   # fraction bits: weights within +-0.5, inputs within +-8


def listed():
    return [
        # one recurrent layer's weight applied to one frame: a small product with a ragged last block-column
        {"name": "spmv_4096x1177_f16", "op": "product", "rows": 4096, "cols": 1177, "block": 32, "law": "uniform", "rate": 8.16,
         "dtype": "f16", "batch": 1},
        # the large bare product at the lowest pruning rate: most bytes per call
        {"name": "spmv_8192_r4_f16", "op": "product", "rows": 8192, "cols": 8192, "block": 64, "law": "lognormal", "rate": 4.0,
         "dtype": "f16", "batch": 1},
        # the same matrix serving a full batch
        {"name": "spmm_8192_r4_b64_f16", "op": "product", "rows": 8192, "cols": 8192, "block": 64, "law": "lognormal", "rate": 4.0,
         "dtype": "f16", "batch": 64},
        # full-precision weights and a handful of requests: a GRU layer's matrix, four vectors
        {"name": "spmm_3072x1536_b4_f32", "op": "product", "rows": 3072, "cols": 1536, "block": 32, "law": "lognormal", "rate": 16.0,
         "dtype": "f32", "batch": 4},
        # a small model on a short window in full precision: the smallest sequence call
        {"name": "lstm_64_128_t16_f32", "op": "rnn", "cell": "lstm", "input": 64, "hidden": 128, "layers": 1, "block": 16, "law": "uniform",
         "rate": 4.0, "dtype": "f32", "steps": 16, "batch": 1, "states": False, "host": False},
        # streaming recognition: one frame per call, the state carried from call to call
        {"name": "lstm_153_1024_frame", "op": "rnn", "cell": "lstm", "input": 153, "hidden": 1024, "layers": 1, "block": 32, "law": "uniform",
         "rate": 8.16, "dtype": "f16", "steps": 1, "batch": 1, "states": True, "host": False},
        # the benchmark's own workload: one long sequence through two large layers
        {"name": "lstm2_2048_t512_b1", "op": "rnn", "cell": "lstm", "input": 2048, "hidden": 2048, "layers": 2, "block": 64, "law": "uniform",
         "rate": 10.0, "dtype": "f16", "steps": 512, "batch": 1, "states": False, "host": False},
        # the same stack serving 32 sequences at once
        {"name": "lstm2_2048_t128_b32", "op": "rnn", "cell": "lstm", "input": 2048, "hidden": 2048, "layers": 2, "block": 64, "law": "uniform",
         "rate": 10.0, "dtype": "f16", "steps": 128, "batch": 32, "states": False, "host": False},
        # a GRU layer with uneven blocks and a small batch
        {"name": "gru_512_1024_t256_b8", "op": "rnn", "cell": "gru", "input": 512, "hidden": 1024, "layers": 1, "block": 32, "law": "lognormal",
         "rate": 16.0, "dtype": "f16", "steps": 256, "batch": 8, "states": False, "host": False},
        # a speech model's projected LSTM layers on one utterance, from and to pinned host memory
        {"name": "lstmp2_153_1024_t100_host", "op": "cell", "cell": "lstmp", "input": 153, "hidden": 1024, "proj": 512, "layers": 2, "block": 32,
         "law": "uniform", "rate": 13.0, "dtype": "f16", "steps": 100, "batch": 1, "states": False, "host": True},
        # the paper's own arithmetic on the large matrix
        {"name": "fixed_8192_r4_b1", "op": "fixed", "rows": 8192, "cols": 8192, "block": 64, "law": "lognormal", "rate": 4.0, "batch": 1},
        # one projection of a large dense weight onto the pattern, as a pruning run does after each round of training
        {"name": "project_8192_f0.75", "op": "project", "rows": 8192, "cols": 8192, "block": 64, "fraction": 0.75},
    ]


def _between(rng, lo, hi):
    """A whole number, spread over the logarithm of the range, odd ones among them."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _weights(c):
    """Expected stored weights of all matrices of a recurrent case."""
    S = c.get("proj") or c["hidden"]
    n = sum(GATES[c["cell"]] * c["hidden"] * ((c["input"] if l == 0 else S) + S) for l in range(c["layers"]))
    if c["cell"] == "lstmp":
        n += c["layers"] * S * c["hidden"]
    return n / c["rate"]


def draw(rng):
    op = rng.choice(["product", "product", "rnn", "rnn", "rnn", "cell", "fixed", "project"])
    block = rng.choice([16, 32, 64])
    if op == "project":
        return {"op": op, "rows": _between(rng, 512, 8192), "cols": _between(rng, 512, 8192), "block": block,
                "fraction": round(rng.uniform(0.7, 0.96), 3)}
    law = rng.choice(["uniform", "lognormal"])
    rate = round(rng.uniform(4.0, 25.0), 2)
    if op == "fixed":
        return {"op": op, "rows": _between(rng, 512, 8192), "cols": _between(rng, 512, 8192), "block": block, "law": law, "rate": rate,
                "batch": rng.choice([1, 1, 2, 4])}
    if op == "product":
        dtype = rng.choice(["f16", "f16", "f16", "f32"])
        batch = rng.choice([1, 1, _between(rng, 2, 64)]) if dtype == "f16" else rng.choice([1, 2, 4, 8])
        return {"op": op, "rows": _between(rng, 512, 8192), "cols": _between(rng, 256, 8192), "block": block, "law": law, "rate": rate,
                "dtype": dtype, "batch": batch}
    c = {"op": op, "cell": rng.choice(["lstm", "gru"]) if op == "rnn" else rng.choice(["lstmp", "ligru", "gru_rb"]),
         "input": _between(rng, 39, 2048 if op == "rnn" else 512), "hidden": 0, "layers": rng.choice([1, 2]), "block": block, "law": law,
         "rate": rate, "dtype": "f16", "steps": 1, "batch": 1, "states": rng.random() < 0.5, "host": rng.random() < 0.25}
    if op == "rnn":
        c["batch"] = rng.choice([1, 1, 4, _between(rng, 8, 32)])
        c["hidden"] = _between(rng, 128, 2048 if c["batch"] == 1 or c["batch"] >= 16 else 1024)
        if rng.random() < 0.2:                      # full-precision weights: small models
            c.update(dtype="f32", hidden=_between(rng, 128, 512), batch=rng.choice([1, 4]))
        c["steps"] = 1 if rng.random() < 0.25 else _between(rng, 2, 512 if c["batch"] == 1 else 128)
        # no more work than the largest listed sequences of the same kind of batch
        most = 6.7e6 * (512 if c["batch"] == 1 else 600 if c["batch"] < 16 else 4096)
        c["steps"] = max(1, min(c["steps"], int(most / (_weights(c) * c["batch"]))))
    else:
        c["hidden"] = 32 * _between(rng, 4, 32)
        c["batch"] = rng.choice([1, 1, 8])
        c["steps"] = 1 if rng.random() < 0.25 else _between(rng, 2, 100)
        if c["cell"] == "lstmp":
            c["proj"] = c["hidden"] // 2
    return c


def _keep(gen, c, rows, cols):
    """Per-block row and column keep masks of about the wanted pruning rate, as host bytes."""
    b = c["block"]
    nbr, nbc = -(-rows // b), -(-cols // b)
    rs = torch.clamp(rows - torch.arange(nbr, device="cuda") * b, max=b).repeat_interleave(nbc)
    cs = torch.clamp(cols - torch.arange(nbc, device="cuda") * b, max=b).repeat(nbr)

    def kept(f, size):
        return torch.minimum(torch.round(f * size).clamp(min=0), size.float())

    def draw2(how):
        return how(nbr * nbc, generator=gen, device="cuda"), how(nbr * nbc, generator=gen, device="cuda")
    f0 = 1 / math.sqrt(c["rate"])
    if c["law"] == "uniform":
        fr, fc = (f0 * (0.7 + 0.6 * u) for u in draw2(torch.rand))
    else:
        er, ec = (torch.exp(SIGMA * z - 0.5 * SIGMA * SIGMA) for z in draw2(torch.randn))
        lo, hi = 0.0, 4.0                           # a keep fraction stops at 1: find the scale that gives the rate
        for _ in range(20):
            f0 = 0.5 * (lo + hi)
            share = float((kept(f0 * er, rs) * kept(f0 * ec, cs)).sum()) / (rows * cols)
            lo, hi = (f0, hi) if share < 1 / c["rate"] else (lo, f0)
        fr, fc = f0 * er, f0 * ec

    def lines(count, size):
        keys = torch.rand((nbr * nbc, b), generator=gen, device="cuda")
        keys.masked_fill_(torch.arange(b, device="cuda")[None, :] >= size[:, None], 2.0)
        rank = keys.argsort(dim=1).argsort(dim=1)
        return (rank < count[:, None]).to(torch.uint8).reshape(-1).cpu().numpy()
    return lines(kept(fr, rs), rs), lines(kept(fc, cs), cs)


def _encoded(gen, c, rows, cols, std=0.05):
    W = (torch.randn((rows, cols), generator=gen, device="cuda") * std).cpu().numpy()
    rk, ck = _keep(gen, c, rows, cols)
    if c["op"] == "fixed":
        return binding.csb_encode_q16(W, c["block"], c["block"], rk, ck, FIXED_W)
    return binding.csb_encode(W, c["block"], c["block"], rk, ck, c["dtype"])


def prepare(case, seed):
    gen = torch.Generator("cuda").manual_seed(seed)
    s = {"case": case}

    def randn(*shape, std=1.0):
        return torch.randn(shape, generator=gen, device="cuda") * std
    if case["op"] == "project":
        s["W"] = randn(case["rows"], case["cols"], std=0.05)
        return s
    if case["op"] in ("product", "fixed"):
        s["A"] = _encoded(gen, case, case["rows"], case["cols"])
        s["x"] = randn(case["batch"], case["cols"])
        s["y"] = torch.empty((case["batch"], case["rows"]), device="cuda")
        if case["op"] == "fixed":
            s["x"] = torch.round(s["x"] * 2 ** FIXED_X).clamp(-32768, 32767).to(torch.int16)
            s["y"] = s["y"].to(torch.int64)
        return s
    H, L, B, T = case["hidden"], case["layers"], case["batch"], case["steps"]
    S = case.get("proj") or H
    # weights shrink with the width so that the recurrence forgets, as a trained one does
    std = min(0.1, 1.6 / math.sqrt(H))
    s["W"] = [_encoded(gen, case, GATES[case["cell"]] * H, (case["input"] if l == 0 else S) + S, std) for l in range(L)]
    if case["cell"] == "lstmp":
        s["Wp"] = [_encoded(gen, case, S, H, std) for _ in range(L)]
    s["bias"] = [randn(BIAS[case["cell"]] * H, std=0.1) for _ in range(L)]
    place = (lambda t: t.cpu().pin_memory()) if case["host"] else (lambda t: t)
    s["x"] = place(randn(T, B, case["input"]))
    s["h0"] = place(randn(L, B, S, std=0.3)) if case["states"] else None
    s["c0"] = place(randn(L, B, H, std=0.3)) if case["states"] else None
    s["y"], s["hT"], s["cT"] = (place(torch.zeros(shape, device="cuda")) for shape in ((T, B, S), (L, B, S), (L, B, H)))
    return s


def run(state):
    c, s = state["case"], state
    if c["op"] == "project":
        row_keep, col_keep, _ = binding.csb_project(s["W"], c["block"], c["block"], c["fraction"])
        return row_keep, col_keep
    if c["op"] == "fixed":
        binding.csb_spmm_q16(s["A"], s["x"], s["y"])
        return s["y"]
    if c["op"] == "product":
        if c["batch"] == 1:
            binding.csb_spmv(s["A"], s["x"], s["y"])
        else:
            binding.csb_spmm(s["A"], s["x"], s["y"])
        return s["y"]
    flags = binding.CSB_FLAG_HOST_IO if c["host"] else 0
    if c["cell"] == "lstm":
        binding.csb_lstm_forward(s["W"], s["bias"], s["x"], s["h0"], s["c0"], s["y"], s["hT"], s["cT"], flags)
    elif c["cell"] == "lstmp":
        binding.csb_lstmp_forward(s["W"], s["Wp"], s["bias"], s["x"], s["h0"], s["c0"], s["y"], s["hT"], s["cT"], flags)
    else:
        forward = {"gru": binding.csb_gru_forward, "ligru": binding.csb_ligru_forward, "gru_rb": binding.csb_gru_reset_before_forward}[c["cell"]]
        forward(s["W"], s["bias"], s["x"], s["h0"], s["y"], s["hT"], flags)
        return s["y"], s["hT"]
    return s["y"], s["hT"], s["cT"]


def work(case):
    """Weights at their expected number, each with its share of the index lists, read once a pass; vectors in and out."""
    if case["op"] == "project":
        n = case["rows"] * case["cols"]             # one squared norm per row segment and per column segment
        return {"bytes": n * (4.0 + 2.0 / case["block"]), "flops": 4.0 * n}
    if case["op"] in ("product", "fixed"):
        cells, per, xy = case["rows"] * case["cols"], {"f32": 4, "f16": 2}.get(case.get("dtype"), 2), (4, 4) if case["op"] == "product" else (2, 8)
        vectors = case["batch"] * (case["cols"] * xy[0] + case["rows"] * xy[1])
        return {"bytes": cells / case["rate"] * per + _lists(cells, case) + vectors, "flops": 2.0 * cells / case["rate"] * case["batch"]}
    n, S, tb = _weights(case), case.get("proj") or case["hidden"], case["steps"] * case["batch"]
    vectors = 4.0 * tb * (case["input"] + S) + 8.0 * case["layers"] * case["batch"] * (S + case["hidden"])
    per = 4 if case["dtype"] == "f32" else 2
    return {"bytes": n * per + _lists(n * case["rate"], case) + vectors, "flops": 2.0 * n * tb}


def _lists(cells, case):
    """Bytes of the index lists and block headers of a matrix of so many cells."""
    blocks = cells / case["block"] ** 2
    return blocks * (6 + 2 * case["block"] / math.sqrt(case["rate"]))


def tolerance(case):
    if case["op"] in ("fixed", "project"):
        return "exact"                              # integer accumulators; masks are whole numbers
    # fp32 accumulation of exact products; through a recurrence the roundings of every step meet again
    return {"rel": 1e-5} if case["op"] == "product" else {"rel": 2e-5}
