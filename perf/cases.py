"""Workloads on which the speed of this framework is judged, through its public entry points.

A case is one call, or one short chain of calls, that a program quantizing a model makes; ``op`` names it:

  layer     quantize_layer: Hessian, grid, greedy descent and loss of one layer whose inputs are on the GPU
  stream    quantize_layers: several layers streamed from pinned host memory, results back on the host
  hessian   cdq_hessian over several batches of calibration rows, accumulated, with the regulariser at the end
  grid      cdq_init_rtn without a clipping search: the round-to-nearest baseline of a layer
  resolve   cdq_cd_solve_with_loss from a Hessian and starting codes at hand
  loss      cdq_layer_loss: total and per-column loss of given codes
  owc_cd    cdq_init_owc_cd: clipping strengths per group by descent

Inputs follow the distributions of ``paper_2406_17542_b200.inputs`` (log-normal feature scales, outlier features,
normal or Student-t entries, normal weights).
"""
from __future__ import annotations

import math

import torch

from paper_2406_17542_b200 import binding as B
from paper_2406_17542_b200 import inputs

DEV = "cuda:0"
F64 = torch.float64

_DEFAULTS = {"op": "layer", "d_in": 256, "d_out": 256, "n": 1024, "x": "bf16", "w": "f32", "bits": 4, "group": 0,
             "clip": 1, "budget": 1.0, "bcd": 0.0, "init": "rtn", "sigma": 1.0, "outliers": 0.0, "student": False,
             "batches": 1, "layers": 1}


def _case(**kw) -> dict:
    return {**_DEFAULTS, **kw}


def listed() -> list:
    return [
        # the smallest layer: launches and latency; fp32 calibration inputs
        _case(name="tiny", d_in=256, d_out=256, n=1024, x="f32", bits=4),
        # three odd-sized small layers from pinned host memory, as a program goes through a small model
        _case(name="stream-odd", op="stream", d_in=1350, d_out=677, n=4099, w="bf16", bits=3, sigma=1.5, outliers=0.01,
              layers=3),
        # MLP up-projection, short rows that stay in L2, many columns, bf16 weights, two passes
        _case(name="mlp-up", d_in=2048, d_out=16384, n=65536, w="bf16", bits=3, budget=2.0, sigma=1.5, outliers=0.01),
        # attention projection, 2 bits in groups of 128 with the clipping search, three passes
        _case(name="attention-clip", d_in=4096, d_out=4096, n=131072, bits=2, group=128, clip=20, budget=3.0, sigma=1.5,
              outliers=0.01),
        # MLP down-projection, a Hessian far larger than L2, two passes
        _case(name="mlp-down", d_in=14336, d_out=4096, n=131072, bits=4, budget=2.0, student=True),
        # a slice of columns of the widest FFN layer (one rank's share), 3 bits in groups with the clipping search
        _case(name="ffn-slice", d_in=18432, d_out=1184, n=32768, bits=3, group=128, clip=20, sigma=1.5, student=True),
        # calibration in batches: the Hessian accumulated as the batches arrive
        _case(name="hessian-batches", op="hessian", d_in=8192, d_out=1, n=4096, batches=8, sigma=1.5, outliers=0.01),
        # round-to-nearest baseline of a large layer
        _case(name="rtn-grid", op="grid", d_in=14336, d_out=16384, n=1, w="bf16", bits=3, group=128),
        # the same layer solved again for another bit width: Hessian and starting codes at hand
        _case(name="resolve", op="resolve", d_in=8192, d_out=592, n=12288, bits=3, student=True),
        # evaluation of given codes
        _case(name="loss", op="loss", d_in=4096, d_out=4096, n=8192, w="bf16", bits=4, group=128, sigma=1.5),
        # per-group clipping strengths
        _case(name="owc-cd", op="owc_cd", d_in=4096, d_out=1024, n=8192, bits=2, group=128, clip=20, sigma=1.5,
              outliers=0.01),
        # the fewer-iterations variant: a quarter of a pass, then random pairs
        _case(name="short-pairs", d_in=3072, d_out=4096, n=16384, bits=3, budget=0.25, bcd=0.125, student=True),
    ]


def _log_int(rng, lo: int, hi: int, multiple: int = 1) -> int:
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / multiple)) * multiple))


def draw(rng) -> dict:
    """One more case of the listed ranges; none costs more than the largest listed one."""
    op = rng.choice(["layer"] * 5 + ["stream", "hessian", "grid", "resolve", "loss", "owc_cd"])
    data = {"sigma": rng.choice([1.0, 1.5]), "outliers": rng.choice([0.0, 0.01]), "student": rng.random() < 0.4,
            "w": rng.choice(["f32", "bf16"]), "bits": rng.choice([2, 3, 3, 4])}
    if op == "stream":
        return _case(op=op, d_in=_log_int(rng, 300, 2000), d_out=_log_int(rng, 200, 2000), n=_log_int(rng, 2000, 8000),
                     layers=rng.choice([2, 3]), **data)
    if op == "hessian":
        return _case(op=op, d_in=_log_int(rng, 512, 12288, 8), d_out=1, n=_log_int(rng, 1024, 8192),
                     batches=rng.choice([2, 4, 8]), **data)
    if op == "grid":
        d_in = _log_int(rng, 512, 16384, 128)
        return _case(op=op, d_in=d_in, d_out=_log_int(rng, 512, 16384), n=1, group=rng.choice([0, 64, 128]), **data)
    if op == "loss":
        d_in = _log_int(rng, 512, 8192, 128)
        return _case(op=op, d_in=d_in, d_out=_log_int(rng, 200, 4096), n=2 * d_in, group=rng.choice([0, 128]), **data)
    if op == "owc_cd":
        d_in = _log_int(rng, 1024, 4096, 128)
        return _case(op=op, d_in=d_in, d_out=_log_int(rng, 200, 1024), n=2 * d_in, group=128, clip=20, **data)
    if op == "resolve":
        d_in = _log_int(rng, 1500, 12288, rng.choice([4, 64, 256]))
        return _case(op=op, d_in=d_in, d_out=_log_int(rng, 150, min(4096, int(4e10 / d_in ** 2))), n=d_in + d_in // 2, **data)
    kind = rng.random()
    if kind < 0.25:    # odd sizes: every row misaligned
        d_in = _log_int(rng, 300, 5000)
        group, n, x = 0, _log_int(rng, 1000, 8192), rng.choice(["bf16", "f32"])
    elif kind < 0.6:   # groups
        d_in = _log_int(rng, 512, 16384, 128)
        group, n, x = rng.choice([64, 128]), _log_int(rng, 8192, 65536), "bf16"
    else:              # per channel
        d_in = _log_int(rng, 256, 18432, 64)
        group, n, x = 0, _log_int(rng, 8192, 65536), "bf16"
    clip = 20 if group and rng.random() < 0.6 else 1
    d_out = _log_int(rng, 150, max(300, min(8192, int(2e11 / d_in ** 2))))
    return _case(op="layer", d_in=d_in, d_out=d_out, n=n, x=x, group=group, clip=clip,
                 budget=rng.choice([0.25, 1.0, 2.0]), **data)


# --------------------------------------------------------------------------------------------- inputs


def _config(case: dict, seed: int, part: int = 0) -> inputs.LayerConfig:
    d_in, d_out = case["d_in"], case["d_out"]
    for _ in range(part):   # the further layers of a stream: other shapes of the same kind
        d_in, d_out = d_out + 173, d_in
    return inputs.LayerConfig("case", d_in, d_out, case["n"], case["x"], case["w"], case["sigma"], case["outliers"],
                              case["student"], 0.015, case["bits"], case["group"], case["clip"],
                              0.5 if case["clip"] > 1 else 1.0, 1.0, 1, 101 * (int(seed) % 100003) + part)


def _grid(case: dict) -> B.Grid:
    return B.Grid(case["bits"], case["group"], case["clip"], 0.5 if case["clip"] > 1 else 1.0, 1.0)


def _steps(case: dict, what: str, d_in: int) -> int:
    return int(case[what] * d_in)


def _hessian64(batches) -> torch.Tensor:
    """X^T X in 64 bits, rows in pieces."""
    H = None
    for X in batches:
        for r in range(0, X.shape[0], 16384):
            Z = X[r:r + 16384].to(F64)
            P = Z.T @ Z
            H = P if H is None else H.add_(P)
            del Z, P
    return H


def _minmax(W: torch.Tensor, case: dict):
    """(scale, zero) of Eq. 2 in 64 bits for a clipping strength of one."""
    d_in, d_out = W.shape
    g = case["group"] or d_in
    lo = W.view(d_in // g, g, d_out).amin(1).to(F64)
    hi = W.view(d_in // g, g, d_out).amax(1).to(F64)
    return (hi - lo) / (2 ** case["bits"] - 1), lo


def _round_codes(W: torch.Tensor, scale: torch.Tensor, zero: torch.Tensor, case: dict) -> torch.Tensor:
    g = case["group"] or W.shape[0]
    a = scale.to(F64).repeat_interleave(g, 0)
    b = zero.to(F64).repeat_interleave(g, 0)
    q = torch.where(a > 0, torch.round((W.to(F64) - b) / a), torch.zeros_like(a))
    return q.clamp_(0, 2 ** case["bits"] - 1).to(torch.uint8)


def prepare(case: dict, seed: int) -> dict:
    op = case["op"]
    if op == "stream":
        layers = []
        for k in range(case["layers"]):
            X, W = inputs.make_layer(_config(case, seed, k), DEV)
            layers.append((X.cpu().pin_memory(), W.cpu().pin_memory()))
        return {"case": case, "layers": layers, "host": {}}
    if op == "hessian":
        return {"case": case, "X": [inputs.make_x(_config(case, 64 * seed + k), DEV) for k in range(case["batches"])]}
    cfg = _config(case, seed)
    state = {"case": case, "W": inputs.make_w(cfg, DEV)}
    if op == "layer":
        state["X"] = inputs.make_x(cfg, DEV)
    elif op != "grid":
        state["H"] = _hessian64([inputs.make_x(cfg, DEV)]).float()
    if op in ("resolve", "loss"):
        scale, zero = _minmax(state["W"], case)
        state["scale"], state["zero"] = scale.float(), zero.float()
        state["Q"] = _round_codes(state["W"], state["scale"], state["zero"], case)
    return state


# --------------------------------------------------------------------------------------------- one pass

_LAYER_KEYS = ("H", "scale", "zero", "Q", "gamma", "loss")


def run(state: dict):
    case = state["case"]
    op, grid = case["op"], _grid(case)
    if op == "layer":
        d_in = state["W"].shape[0]
        out = B.quantize_layer(state["X"], state["W"], grid, 1, device=DEV, init=case["init"],
                               steps_per_col=_steps(case, "budget", d_in), bcd_steps=_steps(case, "bcd", d_in))
        return {k: out[k] for k in _LAYER_KEYS}
    if op == "stream":
        return [{k: out[k] for k in _LAYER_KEYS}
                for out in B.quantize_layers(state["layers"], grid, 1, device=DEV, host_buffers=state["host"])]
    if op == "hessian":
        last = len(state["X"]) - 1
        H = None
        for k, X in enumerate(state["X"]):
            H = B.cdq_hessian(X, lambda_rel=0.01 if k == last else 0.0, accumulate=k > 0, out=H)
        return H
    if op == "grid":
        scale, zero, Q, _ = B.cdq_init_rtn(state["W"], grid)
        return {"scale": scale, "zero": zero, "Q": Q}
    if op == "owc_cd":
        scale, zero, Q, gamma, stats = B.cdq_init_owc_cd(state["W"], grid, state["H"])
        return {"scale": scale, "zero": zero, "Q": Q, "gamma": gamma, "loss": stats["loss_after"]}
    if op == "resolve":
        Q = state["Q"].clone()
        _, loss, cols = B.cdq_cd_solve_with_loss(state["H"], state["W"], grid, state["scale"], state["zero"], Q,
                                                 _steps(case, "budget", Q.shape[0]), per_col=True)
        return {"Q": Q, "loss": loss, "per_col": cols}
    loss, cols = B.cdq_layer_loss(state["H"], state["W"], grid, state["scale"], state["zero"], state["Q"], per_col=True)
    return {"loss": loss, "per_col": cols}


# --------------------------------------------------------------------------------------------- what a pass needs


def _work_layer(case: dict, d_in: int, d_out: int, hessian: bool = True) -> dict:
    ng = d_in // (case["group"] or d_in)
    wb, xb = (2 if case["w"] == "bf16" else 4), (2 if case["x"] == "bf16" else 4)
    # a column commits about 0.4 d_in moves before nothing improves it, or as many as its budget allows
    moves = min(_steps(case, "budget", d_in), 0.4 * d_in)
    by = wb * d_in * d_out + d_in * d_out + 8 * ng * d_out + 4 * d_in * d_in
    fl = 2 * d_in * d_in * d_out + 2 * moves * d_in * d_out
    if case["clip"] > 1:
        fl += 2 * case["clip"] * d_in * d_in * d_out
    if hessian:
        by += xb * case["n"] * d_in
        fl += case["n"] * d_in * (d_in + 1)
    return {"bytes": by, "flops": fl}


def work(case: dict) -> dict:
    op, d_in, d_out, n = case["op"], case["d_in"], case["d_out"], case["n"]
    wb = 2 if case["w"] == "bf16" else 4
    ng = d_in // (case["group"] or d_in)
    if op == "layer":
        return _work_layer(case, d_in, d_out)
    if op == "stream":
        parts = [_config(case, 0, k) for k in range(case["layers"])]
        got = [_work_layer(case, c.d_in, c.d_out) for c in parts]
        return {k: sum(g[k] for g in got) for k in ("bytes", "flops")}
    if op == "hessian":
        return {"bytes": case["batches"] * 2 * n * d_in + 4 * d_in * d_in, "flops": case["batches"] * n * d_in * (d_in + 1)}
    if op == "grid":
        return {"bytes": (wb + 1) * d_in * d_out + 8 * ng * d_out, "flops": 4 * d_in * d_out}
    if op == "resolve":
        w = _work_layer(case, d_in, d_out, hessian=False)
        return {"bytes": w["bytes"] + d_in * d_out, "flops": w["flops"]}
    if op == "loss":
        return {"bytes": 4 * d_in * d_in + (wb + 1) * d_in * d_out + 8 * ng * d_out, "flops": 2 * d_in * d_in * d_out}
    # owc_cd: the starting gradient, the products of a group's block with its residuals, one update per group
    fl = 2 * d_in * d_in * d_out + 2 * case["clip"] * case["group"] * d_in * d_out + 2 * d_in * d_in * d_out
    return {"bytes": 4 * d_in * d_in + (wb + 1) * d_in * d_out + 12 * ng * d_out, "flops": fl}


def tolerance(case: dict):
    """About four times what was measured against 64 bits: Hessians of the tensor cores' fp32 sums are 1e-5 to 7e-5 off,
    the column losses 3e-13 (a total passes through fp32 when it is compared).  Codes come from a greedy search over
    fp32 scores, in which two moves that tie to the last bits send a column along another valid path: 2e-4 of the codes
    of a solved layer differed from the 64-bit search, its column losses by 2.6e-4 together and 4e-3 at most."""
    op = case["op"]
    if op == "grid":
        return {"rel": 1e-6, "max": 1e-5, "differ": 1e-6}
    if op == "hessian":
        return {"rel": 1e-4, "max": 1e-3}
    if op == "loss":
        return {"rel": 1e-7, "max": 1e-6}
    return {"rel": 1e-3, "max": 0.1, "differ": 2e-3}


# --------------------------------------------------------------------------------------------- 64 bits


def _greedy64(H32, W, scale, zero, Q, case):
    """The descent as the paper states it, all columns at once: (codes, column losses)."""
    H = H32.to(F64)
    d_in, d_out = W.shape
    g = case["group"] or d_in
    L = 2 ** case["bits"] - 1
    a = scale.to(F64).repeat_interleave(g, 0).T.contiguous()
    q = Q.T.to(F64).contiguous()
    e0 = (a * q + zero.to(F64).repeat_interleave(g, 0).T) - W.to(F64).T
    G = 2 * (e0 @ H)
    h = torch.diagonal(H)
    inv = torch.where((h > 0) & (a > 0), 1 / (2 * a * h).clamp_min(1e-300), torch.zeros_like(a))
    cols = torch.arange(d_out, device=W.device)
    for step in range(_steps(case, "budget", d_in)):
        d = a * (torch.round(q - G * inv).clamp_(0, L) - q)
        gain, at = ((d * h + G) * d).min(1)
        act = gain < 0
        if step % 64 == 0 and not bool(act.any()):
            break
        move = torch.where(act, d[cols, at], torch.zeros_like(gain))
        q[cols, at] += torch.where(act, torch.round(move / a[cols, at].clamp_min(1e-300)), torch.zeros_like(gain))
        G += 2 * move[:, None] * H[at]
    e = (a * q + zero.to(F64).repeat_interleave(g, 0).T) - W.to(F64).T
    return q.T.to(torch.uint8).contiguous(), ((e @ H) * e).sum(1)


def exact(case: dict, seed: int):
    op = case["op"]
    if op == "stream":
        got = []
        for k in range(case["layers"]):
            X, W = inputs.make_layer(_config(case, seed, k), DEV)
            scale, zero = _minmax(W, case)
            got.append({"H": _hessian64([X]), "scale": scale.cpu(), "zero": zero.cpu(), "Q": None, "gamma": None, "loss": None})
        return got
    state = prepare(case, seed)
    if op == "hessian":
        H = _hessian64(state["X"])
        H.diagonal().add_(torch.tensor(0.01, dtype=torch.float32, device=DEV).to(F64) * H.diagonal().mean())
        return H
    scale, zero = _minmax(state["W"], case)
    if op == "grid":
        return {"scale": scale, "zero": zero, "Q": None}
    if op == "layer":   # the codes hang on ties between scores and have no 64-bit value of their own
        known = case["clip"] <= 1
        return {"H": _hessian64([state["X"]]), "scale": scale if known else None, "zero": zero, "Q": None, "gamma": None,
                "loss": None}
    if op == "owc_cd":
        return {"scale": None, "zero": zero, "Q": None, "gamma": None, "loss": None}
    if op == "loss":
        g = case["group"] or case["d_in"]
        a = state["scale"].to(F64).repeat_interleave(g, 0)
        E = a * state["Q"].to(F64) + state["zero"].to(F64).repeat_interleave(g, 0) - state["W"].to(F64)
        cols = ((state["H"].to(F64) @ E) * E).sum(0)
        return {"loss": float(cols.sum()), "per_col": cols}
    Q, cols = _greedy64(state["H"], state["W"], state["scale"], state["zero"], state["Q"], case)
    return {"Q": Q, "loss": float(cols.sum()), "per_col": cols}
