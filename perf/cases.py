"""Workloads of the optimizer step, for timing and for comparing one build's results with another's.

A case names one call that a training program makes over and over: the step of one weight matrix (`step`), of several
matrices of one shape that share A (`group`), of a matrix split into chunks (`mesgc`), of a projected matrix (`cesgc`),
and the selection on its own (`sparsify`).  Shapes are those of the Llama-2-7B projections, of the (k, s) sweep and of the
chunked variants' published settings, a toy, and odd ones in between.

Gradients are quasi-sparse as the method assumes: Student-t noise (1e-3) under planted entries of magnitude U(0.5, 1).  A
state holds a ring of gradients, a fresh one for every pass; in `drift` of the planted positions two consecutive gradients
differ.  States have made a few steps before the first pass, as those of a running program have.
"""
import math

import numpy as np
import torch

from paper_2502_00311_b200 import binding, inputs

RING = 4                # gradients a state cycles through
WARM = 3                # steps made before the first pass
SEED_A = 1              # names the measurement matrix

DEFAULTS = dict(kind="step", rows=0, cols=0, k=0, s=0, states=1, chunks=1, rank=0, drift=0, shared=False)


def _case(**kw):
    c = dict(DEFAULTS)
    c.update(kw)
    return c


def listed():
    return [
        # the toy: launches and latency are everything
        _case(name="step_64x64_k256_s16", rows=64, cols=64, k=256, s=16),
        # one attention projection at the headline setting: the recovery is exact, one screening pass per step
        _case(name="step_4096x4096_k2048_s64", rows=4096, cols=4096, k=2048, s=64),
        # one MLP projection of the single-layer setting: more entries kept than k rows can tell apart
        _case(name="step_4096x11008_k2048_s128", rows=4096, cols=11008, k=2048, s=128),
        # the corners of the (k, s) sweep on that shape: the fewest rows of A, and many rows with many kept entries
        _case(name="step_4096x11008_k256_s16", rows=4096, cols=11008, k=256, s=16),
        _case(name="step_4096x11008_k4096_s256", rows=4096, cols=11008, k=4096, s=256),
        # an odd vector with k = 7 s rows (the paper's ratio), no multiple of anything
        _case(name="step_1000x3001_k700_s100", rows=1000, cols=3001, k=700, s=100),
        # q, k, v, o of one layer of the whole-model setting, with supports that drift from step to step
        _case(name="group4_4096x4096_k1024_s64", kind="group", rows=4096, cols=4096, k=1024, s=64, states=4, drift=2),
        # the same four matrices with few kept entries: their residuals share one pass
        _case(name="group4_4096x4096_k1024_s16", kind="group", rows=4096, cols=4096, k=1024, s=16, states=4),
        # the paper's memory-efficient setting (one kept entry per chunk), and a corner of its chunk study
        _case(name="mesgc_4096x4096_c256_k8_s1", kind="mesgc", rows=4096, cols=4096, chunks=256, k=8, s=1),
        _case(name="mesgc_4096x4096_c256_k112_s16", kind="mesgc", rows=4096, cols=4096, chunks=256, k=112, s=16),
        # the paper's compute-efficient setting
        _case(name="cesgc_4096x4096_r32_c64_k217_s31", kind="cesgc", rows=4096, cols=4096, rank=32, chunks=64, k=217, s=31),
        # the selection on its own, for programs that cannot allocate
        _case(name="sparsify_4096x11008_s64", kind="sparsify", rows=4096, cols=11008, s=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "group", "mesgc", "mesgc", "cesgc", "sparsify"])
    if kind == "sparsify":
        s = _log_int(rng, 1, 1024)
        return _case(kind=kind, rows=1, cols=_log_int(rng, max(s, 1 << 10), 1 << 26), s=s)
    if kind == "mesgc":
        s = _log_int(rng, 1, 31)
        chunks = rng.choice([16, 48, 64, 100, 256, 300, 1024])
        per = _log_int(rng, 256, (1 << 24) // chunks) // 4 * 4
        return _case(kind=kind, rows=chunks, cols=per, chunks=chunks, k=rng.choice([7, 8]) * s, s=s)
    if kind == "cesgc":
        s = _log_int(rng, 1, 31)
        rank, chunks = rng.choice([8, 16, 32, 48, 64]), rng.choice([16, 32, 64])
        return _case(kind=kind, rows=_log_int(rng, 256, 4096), cols=_log_int(rng, 256, 4096) // 64 * 64, rank=rank,
                     chunks=chunks, k=7 * s, s=s)
    # whole matrices: any length, rows of A in whole chunks of 64 or (a quarter of the time) k = 7 s
    while True:
        s = _log_int(rng, 4, 200)
        ragged = rng.random() < 0.25
        k = 7 * s if ragged else 64 * max(1, round(s * rng.choice([8, 16, 32, 64]) / 64))
        rows = _log_int(rng, 64, 4096)
        cols = _log_int(rng, 64, 11008)
        states = rng.choice([2, 3, 4]) if kind == "group" else 1
        cost = 4.0 * k * s * rows * cols * states
        # k is far below d; the cost stays below that of the largest listed case (k = 7 s takes longer for the same work)
        if k <= 8192 and 16 * k <= rows * cols and cost <= (1.0e12 if ragged else 4.0e13):
            break
    return _case(kind=kind, rows=rows, cols=cols, k=k, s=s, states=states, drift=rng.choice([0, 0, 0, 2]),
                 shared=kind == "step" and rng.random() < 0.15)


# ---- inputs -----------------------------------------------------------------------------------------------------
def _gradients(d, s, drift, seed):
    """RING gradients of length d with s planted entries; `drift` of the positions move from one to the next."""
    rng = np.random.Generator(np.random.PCG64(seed))
    supp, sign = inputs.planted_support(d, s, seed)
    supp = supp.astype(np.int64)
    sign = torch.from_numpy(sign).cuda()
    out = []
    for i in range(RING):
        if i and drift:
            free = np.setdiff1d(rng.integers(0, d, size=4 * drift + 16), supp)[:drift]
            supp[rng.choice(s, size=free.size, replace=False)] = free
        g = torch.empty(d, dtype=torch.float32, device="cuda")
        out.append(inputs.gradient_on_device(g, torch.from_numpy(supp).cuda(), sign, seed * RING + i))
    return out


def _weights(shape, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, device="cuda", generator=gen) * 0.02


def _projection(m, r, seed):
    """An r x m matrix with orthonormal rows, and the m x 6 factor (spanned by its first rows) of a low-rank gradient."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    q, _ = torch.linalg.qr(torch.randn(m, r, device="cuda", generator=gen))
    return q.t().contiguous(), q[:, :6].contiguous()


def prepare(case, seed):
    kind, d, k, s = case["kind"], case["rows"] * case["cols"], case["k"], case["s"]
    hp = inputs.ADAM
    adam = (hp["lr"], hp["beta1"], hp["beta2"], hp["eps"])
    base = 100_003 * (seed % 20_000_003)
    st = dict(kind=kind, i=0)
    if kind == "sparsify":
        st["grads"] = _gradients(d, min(s, 64), 0, base)
        st["idx"] = torch.empty(s, dtype=torch.int32, device="cuda")
        st["val"] = torch.empty(s, dtype=torch.float32, device="cuda")
        st["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        st["s"] = s
    elif kind == "mesgc":
        st["opt"] = binding.Mesgc(d, case["chunks"], k, s, SEED_A, *adam, alpha=2.0)
        st["grads"] = _gradients(d, s * case["chunks"], case["drift"], base)
        st["weight"] = _weights(d, base + 1)
    elif kind == "cesgc":
        m, n, r = case["rows"], case["cols"], case["rank"]
        st["opt"] = binding.Cesgc(m, n, r, case["chunks"], k, s, SEED_A, *adam, alpha=2.0)
        B, left = _projection(m, r, base)
        st["opt"].set_projection(B)
        right = _gradients(left.shape[1] * n, s, 0, base + 2)              # sparse right factors: few large entries after B
        noise = _gradients(d, s, 0, base + 3)
        st["grads"] = [x.view(m, n) + left @ y.view(-1, n) for x, y in zip(noise, right)]
        st["weight"] = _weights((m, n), base + 1)
    else:
        n = case["states"]
        st["opt"] = [binding.Sgc(d, k, s, SEED_A, *adam) for _ in range(n)]
        for o in st["opt"]:
            if case["shared"]:
                o.set_recovery(True)
        st["grads"] = [_gradients(d, s, case["drift"], base + 11 * j) for j in range(n)]
        st["weight"] = [_weights(d, base + 11 * j + 1) for j in range(n)]
    for _ in range(WARM):
        run(st)
    return st


# ---- one pass ---------------------------------------------------------------------------------------------------
def run(state):
    kind, i = state["kind"], state["i"] % RING
    state["i"] += 1
    if kind == "sparsify":
        binding.sparsify_static(state["grads"][i], state["s"], state["idx"], state["val"], state["status"])
        return state["idx"], state["val"], state["status"]
    if kind in ("mesgc", "cesgc"):
        state["opt"].step(state["grads"][i], state["weight"])
    elif kind == "step":
        state["opt"][0].step(state["grads"][0][i], state["weight"][0])
    else:
        binding.step_group(state["opt"], [g[i] for g in state["grads"]], state["weight"])
    return state["weight"]


# ---- what a pass cannot do without ----------------------------------------------------------------------------------
def work(case):
    kind, d, k, s = case["kind"], case["rows"] * case["cols"], case["k"], case["s"]
    if kind == "sparsify":
        return {"bytes": 4.0 * d + 8.0 * s, "flops": 0.0}
    n = case["states"] * case["chunks"]                                     # problems, each with its own moments
    small = n * (16.0 * k + 8.0 * s)                                        # M and V read and written, the updated weights
    if kind == "cesgc":
        r, p = case["rank"], case["rank"] * case["cols"]
        return {"bytes": 4.0 * d + 4.0 * r * case["rows"] + small, "flops": 2.0 * r * d + 4.0 * k * s * p}
    if kind == "mesgc":
        return {"bytes": 4.0 * d + small, "flops": 4.0 * k * s * d}
    # every pick of both recoveries correlates its residual with every column of A
    streams = 1 if case["shared"] else 2
    return {"bytes": case["states"] * 4.0 * d + small, "flops": case["states"] * 2.0 * streams * k * s * d}


def tolerance(case):
    if case["kind"] == "sparsify":
        return "exact"
    if case["kind"] == "cesgc":
        return {"rel": 1e-5, "max": 1e-3}                                   # a product of the projection may round the other way
    # weights are float32 and an update is a few percent of a weight, good to 1e-4 of itself
    return {"rel": 1e-6, "max": 1e-5}
