"""The work this library is measured on: softmax forward and backward over
uniform and ragged batches, and the batched matrix product, each through the
entry point a program calls.

Every case uses the DYNAMIC policy, the one a program that wants speed asks
for (the others compute the same bits under other schedules).  A case is a
dict:
  kind    "softmax" (bsm_softmax_ex), "ragged" (bsm_softmax_ragged),
          "plan" (bsm_plan_create once, bsm_plan_execute per pass),
          "backward" (bsm_softmax_backward), "bmm" (bsm_bmm)
  dtype   "f32" or "bf16": the data type of the output (and of the inputs;
          the product's operands are always bf16)
  B, R, C         slices of R rows of C elements ("ragged": B slices, R and C
                  the largest, shapes drawn from the case's own fields)
  M, N, K         the product's sizes per slice
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2002_07062_gb300 import bsm

_TORCH = {"f32": torch.float32, "bf16": torch.bfloat16}
_BSM = {"f32": bsm.F32, "bf16": bsm.BF16}
_SIZE = {"f32": 4, "bf16": 2}

# bytes a drawn case moves at most; the largest listed case moves 4.7 GB
_MAX_BYTES = 1 << 30
_MIN_BYTES = 1 << 17
# a drawn product's operations at most: the largest listed one's
_MAX_FLOPS = 8 * 2 * 2048 ** 3


def listed():
    return [
        # a few attention heads of a short sequence: one call's latency
        dict(name="small_f32", kind="softmax", dtype="f32", B=8, R=64, C=64, causal=False, scale=1.0),
        # one layer's causal attention scores at batch 1, 16 heads of 512
        # positions: about one block of rows per SM
        dict(name="layer_bf16_causal", kind="softmax", dtype="bf16", B=16, R=512, C=512, causal=True, scale=8.0),
        # attention scores of a whole batch, 384 slices of 512 x 512
        dict(name="batch_f32", kind="softmax", dtype="f32", B=384, R=512, C=512, causal=False, scale=3.0),
        # the same in bf16 under the causal mask, on a plan kept by the program
        dict(name="batch_bf16_causal", kind="plan", dtype="bf16", B=384, R=512, C=512, causal=True, scale=8.0),
        # many tiny slices: per-slice overhead
        dict(name="tiny_bf16", kind="softmax", dtype="bf16", B=65536, R=32, C=128, causal=False, scale=1.0),
        # a batch of slices of different shapes: the largest call
        dict(name="ragged_f32", kind="ragged", dtype="f32", B=1000, R=1024, C=2048, r_unit=64, c_unit=64,
             shape_seed=4, causal=False, scale=2.0),
        # vocabulary-sized rows of an output layer, one row per position
        dict(name="vocab_bf16", kind="softmax", dtype="bf16", B=1, R=4096, C=32000, causal=False, scale=2.0),
        # rows of 1 MiB: softmax over a whole index of candidates
        dict(name="long_f32", kind="softmax", dtype="f32", B=256, R=1, C=262144, causal=False, scale=1.0),
        # the training step's backward pass over the batch of attention scores
        dict(name="backward_bf16", kind="backward", dtype="bf16", B=384, R=512, C=512, scale=8.0),
        # and over an output layer's rows
        dict(name="backward_vocab_f32", kind="backward", dtype="f32", B=1, R=2048, C=32000, scale=2.0),
        # attention scores as a batched product: 384 of (512 x 64)(64 x 512)
        dict(name="bmm_scores", kind="bmm", dtype="bf16", B=384, M=512, N=512, K=64),
        # a batch of square products, where the tensor cores are the bound
        dict(name="bmm_square", kind="bmm", dtype="bf16", B=8, M=2048, N=2048, K=2048),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(2.0 ** rng.uniform(np.log2(lo), np.log2(hi))))


def draw(rng):
    """One more case of the same ranges: rows of 64 bytes to 4 MiB (a multiple
    of 16 bytes, as every entry point wants), batches of 128 KiB to 1 GiB."""
    kind = rng.choice(["softmax", "softmax", "plan", "ragged", "backward", "backward", "bmm"])
    dtype = rng.choice(["f32", "bf16"])
    es = _SIZE[dtype]
    if kind == "bmm":
        while True:
            M = 128 * _log_uniform(rng, 1, 16)
            N = 64 * _log_uniform(rng, 1, 32)
            K = 64 * _log_uniform(rng, 1, 32)
            B = _log_uniform(rng, 1, 512)
            c = dict(kind=kind, dtype=dtype, B=B, M=M, N=N, K=K)
            w = work(c)
            if _MIN_BYTES <= w["bytes"] <= _MAX_BYTES and w["flops"] <= _MAX_FLOPS:
                return c
    if kind == "ragged":
        n = _log_uniform(rng, 4, 1000)
        rmax = _log_uniform(rng, 8, 512)
        cmax = 16 // es * _log_uniform(rng, 8, 512)
        return dict(kind=kind, dtype=dtype, B=n, R=rmax, C=cmax, r_unit=1, c_unit=16 // es,
                    shape_seed=rng.randrange(1 << 30), causal=rng.random() < 0.25,
                    scale=rng.choice([1.0, 2.0, 8.0]))
    arrays = 3 if kind == "backward" else 2
    vec = _log_uniform(rng, 4, (1 << 20 if kind == "backward" else 1 << 22) // 16)
    C = vec * (16 // es)
    total = _log_uniform(rng, max(_MIN_BYTES, arrays * vec * 16), _MAX_BYTES)
    rows = max(1, total // (arrays * vec * 16))
    R = min(rows, _log_uniform(rng, 1, 1024))
    c = dict(kind=kind, dtype=dtype, B=max(1, rows // R), R=R, C=C, scale=rng.choice([1.0, 2.0, 8.0]))
    if kind != "backward":
        # the causal mask belongs to slices about as high as they are wide
        c["causal"] = R > 1 and C <= 4096 and rng.random() < 0.4
    return c


def _shapes(case):
    """(offsets, rows, cols) of the ragged batch, packed back to back."""
    g = np.random.default_rng(case["shape_seed"])
    rows = (g.integers(1, case["R"] // case["r_unit"] + 1, case["B"]) * case["r_unit"]).astype(np.int32)
    cols = (g.integers(1, case["C"] // case["c_unit"] + 1, case["B"]) * case["c_unit"]).astype(np.int32)
    n = rows.astype(np.int64) * cols
    return np.concatenate([[0], np.cumsum(n)[:-1]]).astype(np.int64), rows, cols


def _elements(case):
    if case["kind"] == "ragged":
        _, rows, cols = _shapes(case)
        return int(np.sum(rows.astype(np.int64) * cols))
    return case["B"] * case["R"] * case["C"]


def _normal(n, seed, scale, dtype):
    """n draws of N(0, scale) in the given type, in pieces of 2^28 values."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = torch.empty(n, dtype=_TORCH[dtype], device="cuda")
    for o in range(0, n, 1 << 28):
        m = min(1 << 28, n - o)
        out[o:o + m] = torch.randn(m, generator=g, device="cuda").mul_(scale)
    return out


def _inputs(case, seed):
    if case["kind"] == "bmm":
        B, M, N, K = case["B"], case["M"], case["N"], case["K"]
        return {"a": _normal(B * M * K, 2 * seed, 1.0, "bf16"),
                "bt": _normal(B * N * K, 2 * seed + 1, 1.0, "bf16")}
    n = _elements(case)
    if case["kind"] == "backward":
        # y as a forward pass leaves it, dy a gradient of unit size
        v = _normal(n, 2 * seed, case["scale"], "f32").view(-1, case["C"])
        y = torch.empty(v.shape, dtype=_TORCH[case["dtype"]], device="cuda")
        step = max(1, (1 << 26) // case["C"])
        for r in range(0, v.shape[0], step):
            y[r:r + step] = torch.softmax(v[r:r + step], -1)
        return {"y": y.view(-1), "dy": _normal(n, 2 * seed + 1, 1.0, case["dtype"])}
    return {"x": _normal(n, 2 * seed, case["scale"], case["dtype"])}


def prepare(case, seed):
    st = dict(_inputs(case, seed), case=case)
    dt = case["dtype"]
    if case["kind"] == "bmm":
        st["out"] = torch.empty(case["B"] * case["M"] * case["N"], dtype=_TORCH[dt], device="cuda")
        return st
    st["out"] = torch.empty(_elements(case), dtype=_TORCH[dt], device="cuda")
    if case["kind"] == "ragged":
        st["offsets"], st["rows"], st["cols"] = _shapes(case)
    if case["kind"] == "plan":
        st["plan"] = bsm.bsm_plan_create(
            st["x"], st["out"], np.full(case["B"], case["R"], np.int32), np.full(case["B"], case["C"], np.int32),
            _BSM[dt], bsm.POLICY_DYNAMIC, flags=bsm.FLAG_CAUSAL if case["causal"] else 0)
    return st


def run(state):
    c = state["case"]
    out, dt, stream = state["out"], _BSM[c["dtype"]], torch.cuda.current_stream()
    flags = bsm.FLAG_CAUSAL if c.get("causal") else 0
    if c["kind"] == "softmax":
        bsm.bsm_softmax_ex(state["x"], out, c["B"], c["R"], c["C"], dt, bsm.POLICY_DYNAMIC, flags, stream)
    elif c["kind"] == "plan":
        state["plan"].execute(stream)
    elif c["kind"] == "ragged":
        bsm.bsm_softmax_ragged(state["x"], out, state["offsets"], state["rows"], state["cols"], dt,
                               bsm.POLICY_DYNAMIC, flags, stream)
    elif c["kind"] == "backward":
        bsm.bsm_softmax_backward(state["y"], state["dy"], out, c["B"], c["R"], c["C"], dt, bsm.POLICY_DYNAMIC,
                                 stream)
    else:
        bsm.bsm_bmm(state["a"], state["bt"], out, c["B"], c["M"], c["N"], c["K"], dt, bsm.POLICY_DYNAMIC, stream)
    return out


def work(case):
    """Each input read once, each output written once; a softmax costs about
    five operations an element (maximum, exponent, exponential, sum, scale),
    its backward pass four, a product 2 K per output."""
    es = _SIZE[case["dtype"]]
    if case["kind"] == "bmm":
        B, M, N, K = case["B"], case["M"], case["N"], case["K"]
        return {"bytes": 2 * B * (M + N) * K + es * B * M * N, "flops": 2 * B * M * N * K}
    n = _elements(case)
    if case["kind"] == "backward":
        return {"bytes": 3 * n * es, "flops": 4 * n}
    return {"bytes": 2 * n * es, "flops": 5 * n}


def tolerance(case):
    """About four times what the library differs from exact()."""
    if case["dtype"] == "bf16":
        return {"rel": 7e-3, "max": 1.6e-2}
    return {"rel": 1e-6, "max": 2e-5}


def exact(case, seed):
    inp = _inputs(case, seed)
    if case["kind"] == "bmm":
        B, M, N, K = case["B"], case["M"], case["N"], case["K"]
        a, bt = inp["a"].view(B, M, K), inp["bt"].view(B, N, K)
        out = torch.empty((B, M, N), dtype=torch.float64, device="cuda")
        for s in range(B):
            torch.matmul(a[s].double(), bt[s].double().t(), out=out[s])
        return out.view(-1)
    n = _elements(case)
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    if case["kind"] == "backward":
        C = case["C"]
        y, dy, o = inp["y"].view(-1, C), inp["dy"].view(-1, C), out.view(-1, C)
        step = max(1, (1 << 26) // C)
        for r in range(0, y.shape[0], step):
            yd, gd = y[r:r + step].double(), dy[r:r + step].double()
            o[r:r + step] = yd * (gd - (yd * gd).sum(-1, keepdim=True))
        return out
    if case["kind"] == "ragged":
        blocks = [(int(o), int(r), int(c), int(r)) for o, r, c in zip(*_shapes(case))]
    else:
        # whole slices at a time, about 2^26 elements
        B, R, C = case["B"], case["R"], case["C"]
        step = max(1, (1 << 26) // (R * C))
        blocks = [(s * R * C, min(step, B - s) * R, C, R) for s in range(0, B, step)]
    for off, rows, cols, per in blocks:
        v = inp["x"][off:off + rows * cols].double().view(rows, cols)
        if case["causal"]:
            row = torch.arange(rows, device="cuda").remainder(per)
            v = v.masked_fill(torch.arange(cols, device="cuda")[None, :] > row[:, None], float("-inf"))
        out[off:off + rows * cols] = torch.softmax(v, -1).view(-1)
    return out
