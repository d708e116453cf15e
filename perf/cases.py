"""Timed cases of the public entry points (Chain, Server), over the range of sizes and options that
the workloads, the tests and the request stream of this repository span.

Kinds of call:
  sweep   Chain.sweep: K normalised sweeps with their stats, one chunk of a solve (block-tridiagonal,
          paired block-pentadiagonal or block-banded generators, inverse or coupled, stair type 1 or 2)
  host    Chain.sweep_host: one sweep through pinned host vectors
  solve   Chain.solve to a residual of 1e-12, FP64 or FP32 / BF16 storage with FP64 refinement
  setup   Chain(...): layout, factorisation and the sweep's operators, read back with Chain.export
  serve   Server: a mix of requests submitted from host memory, run until idle, results fetched

Generators are made from the seed alone, on the GPU, by the recipe of the synthetic QBD workloads:
each rate is present with probability 1/2 and lies in [0.1, 1), diagonals of the up and down blocks
are always present, the down blocks are scaled to the up / down rate ratio, and rows sum to zero.
"""
import math

import numpy as np
import torch

import paper_2302_07551_gb300 as mc

F64 = torch.float64
L2_BYTES = 126e6


def listed():
    return [
        # one sweep of a tiny chain inside a caller's own loop: latency and launches only
        dict(name="step_L64_m8", kind="sweep", L=64, m=8, K=1, apply="inverse", stair=1, shape="qbd", ratio=0.8),
        # the oracle-sized chain solved from uniform: many short chunks, one host check each
        dict(name="solve_L64_m8", kind="solve", L=64, m=8, apply="inverse", dtype="f64", ratio=0.8, check=32, x0=False),
        # one solve chunk of the benchmark chain (3.2 GB of blocks a sweep)
        dict(name="chunk_L32768_m64", kind="sweep", L=32768, m=64, K=64, apply="inverse", stair=1, shape="qbd", ratio=0.9),
        # odd level count, block size that is no multiple of 32, the other apply mode and stair type
        dict(name="chunk_L5001_m100_coupled", kind="sweep", L=5001, m=100, K=32, apply="coupled", stair=2, shape="qbd", ratio=0.9),
        # one sweep a call between pinned host vectors: the end-to-end step of the benchmark
        dict(name="host_L32768_m64", kind="host", L=32768, m=64, apply="inverse", ratio=0.9),
        # batch arrivals and services of one or two: pentadiagonal, paired to 4096 blocks of 256
        dict(name="penta_L4096_m256", kind="sweep", L=4096, m=256, K=16, apply="inverse", stair=1, shape="penta", ratio=0.8),
        # block Hessenberg: batch arrivals of up to four levels
        dict(name="hessenberg_L4096_m64", kind="sweep", L=4096, m=64, K=64, apply="inverse", stair=1, shape="banded", lower=1, upper=4, ratio=0.8),
        # refinement with the least bytes a sweep, large blocks
        dict(name="refine_bf16_L512_m256", kind="solve", L=512, m=256, apply="coupled", dtype="bf16", ratio=0.8, check=64, x0=False),
        # refinement of small blocks that are no power of two, warm start from a given vector
        dict(name="refine_f32_L2048_m24", kind="solve", L=2048, m=24, apply="inverse", dtype="f32", ratio=0.7, check=64, x0=True),
        # set-up of a chain that is solved once: paid in full by every new generator
        dict(name="setup_L8192_m64", kind="setup", L=8192, m=64, apply="inverse", dtype="f64", ratio=0.9),
        # set-up for the low-precision coupled form with large blocks
        dict(name="setup_L512_m256_bf16", kind="setup", L=512, m=256, apply="coupled", dtype="bf16", ratio=0.9),
        # a mix of the request stream's sizes through the solve server, from host memory to results
        dict(name="serve_bf16_mix", kind="serve", dtype="bf16", apply="coupled", check=64, requests="128x16:0.6 300x32:0.7 517x64:0.75 1024x16:0.8 200x128:0.6 160x64:0.9 731x32:0.65 256x128:0.5"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["sweep", "solve", "setup", "host", "serve"], [6, 4, 2, 1, 2])[0]
    apply = rng.choice(["inverse", "coupled"])
    ratio = round(rng.uniform(0.5, 0.95), 3)
    if kind in ("sweep", "host"):
        shape = rng.choices(["qbd", "penta", "banded"], [4, 1, 1])[0] if kind == "sweep" else "qbd"
        if shape == "penta":
            m = 64 * rng.randint(1, 4)
        elif shape == "banded":
            m = _logint(rng, 4, 96)
        else:
            m = _logint(rng, 1, 256)
        L = min(_logint(rng, 33, 32768), int(32768 * 4096 / (m * m * (2 if shape == "banded" else 1))))
        if kind == "host":
            return dict(kind="host", L=L, m=m, apply=apply, ratio=ratio)
        c = dict(kind="sweep", L=L, m=m, K=_logint(rng, 1, 64), apply="inverse" if shape == "banded" else apply,
                 stair=rng.randint(1, 2), shape=shape, ratio=ratio)
        if shape == "banded":
            c["lower"], c["upper"] = rng.choice([(1, 4), (3, 1), (2, 3), (1, 2)])
        return c
    if kind == "solve":
        dtype = rng.choice(["f64", "f32", "bf16"])
        m = _logint(rng, 3, 200) if dtype == "f64" else 4 * _logint(rng, 1, 64)
        L = _logint(rng, 33, max(40, min(900, int(8e6 / (m * m)))))
        return dict(kind="solve", L=L, m=m, apply=apply, dtype=dtype, ratio=round(rng.uniform(0.5, 0.8), 3), check=rng.choice([32, 48, 64]), x0=rng.random() < 0.5)
    if kind == "setup":
        dtype = rng.choice(["f64", "bf16"])
        m = _logint(rng, 4, 256) if dtype == "f64" else 4 * _logint(rng, 1, 64)
        L = min(_logint(rng, 33, 8192), max(33, int(512 * 256 ** 3 / m ** 3)))
        return dict(kind="setup", L=L, m=m, apply=apply, dtype=dtype, ratio=ratio)
    reqs = " ".join("%dx%d:%.2f" % (_logint(rng, 128, 700), rng.choice([16, 32, 64, 128]), rng.uniform(0.5, 0.75)) for _ in range(rng.randint(2, 6)))
    return dict(kind="serve", dtype=rng.choice(["f64", "bf16", "bf16"]), apply=apply, check=64, requests=reqs)


# ---- generators ------------------------------------------------------------------------------

def _rates(g, L, m, diag):
    """L x m x m rates: present with probability 1/2, in [0.1, 1); diag: True present, False zero."""
    a = torch.rand(L, m, m, generator=g, device="cuda", dtype=F64).mul_(0.9).add_(0.1)
    keep = torch.rand(L, m, m, generator=g, device="cuda", dtype=torch.float32) < 0.5
    d = keep.diagonal(dim1=1, dim2=2)
    d.fill_(diag)
    return a.mul_(keep)


def _close(loc, *others):
    """Diagonal of the local blocks such that every row of Q sums to zero."""
    s = loc.sum(2)
    for o in others:
        s += o.sum(2)
    loc.diagonal(dim1=1, dim2=2).sub_(s)


def _qbd(g, L, m, ratio):
    up, dn, loc = _rates(g, L, m, True), _rates(g, L, m, True), _rates(g, L, m, False)
    dn.mul_((up.sum((1, 2)) / (ratio * dn.sum((1, 2))))[:, None, None])
    up[-1] = 0.0
    dn[0] = 0.0
    _close(loc, up, dn)
    return dn, loc, up


def _penta(g, L, m, ratio):
    """Jumps of +-1 and +-2 levels of m/2 phases, paired into L levels of m phases."""
    h = m // 2
    u1, u2, d1, d2 = (_rates(g, 1, h, True)[0] * s for s in (1.0, 0.3, 1.0, 0.3))
    a = _rates(g, 1, h, False)[0]
    f = (u1.sum() + u2.sum()) / (ratio * (d1.sum() + d2.sum()))
    d1, d2 = d1 * f, d2 * f
    z = torch.zeros_like(a)
    pair = lambda p, q, r, s: torch.cat([torch.cat([p, q], 1), torch.cat([r, s], 1)], 0)  # noqa: E731
    rep = lambda b: b.unsqueeze(0).repeat(L, 1, 1)  # noqa: E731
    dn, loc, up = rep(pair(d2, d1, z, d2)), rep(pair(a, u1, d1, a)), rep(pair(u2, z, u1, u2))
    up[-1] = 0.0
    dn[0] = 0.0
    _close(loc, up, dn)
    return dn, loc, up


def _banded(g, L, m, lower, upper, ratio):
    """Jumps of up to `upper` levels up and `lower` down, rates halving with each further level."""
    d = {e: _rates(g, L, m, e != 0) * 0.5 ** max(0, abs(e) - 1) for e in range(-lower, upper + 1)}
    f = sum(d[e].sum() for e in d if e > 0) / (ratio * sum(d[e].sum() for e in d if e < 0))
    for e in d:
        if e < 0:
            d[e].mul_(f)
            d[e][:-e] = 0.0
        elif e > 0:
            d[e][L - e:] = 0.0
    _close(d[0], *(d[e] for e in d if e))
    return d


def _blocks(case, g):
    if case.get("shape") == "banded":
        return _banded(g, case["L"], case["m"], case["lower"], case["upper"], case["ratio"])
    make = _penta if case.get("shape") == "penta" else _qbd
    return make(g, case["L"], case["m"], case["ratio"])


def _inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    b = _blocks(case, g)
    x = torch.rand(case["L"] * case["m"], generator=g, device="cuda", dtype=F64).add_(0.05)
    return b, x / x.sum()


def _requests(case, seed):
    out = []
    for i, r in enumerate(case["requests"].split()):
        size, ratio = r.split(":")
        L, m = (int(v) for v in size.split("x"))
        g = torch.Generator(device="cuda")
        g.manual_seed(int(seed) * 64 + i)
        out.append(_qbd(g, L, m, float(ratio)))
    return out


# ---- the passes ------------------------------------------------------------------------------

def _chain(case, b, **kw):
    if isinstance(b, dict):
        return mc.Chain.banded(b, stair=case.get("stair", 1), **kw)
    return mc.Chain(*b, stair=case.get("stair", 1), apply=case["apply"], dtype=case.get("dtype", "f64"), paired=case.get("shape") == "penta", **kw)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        reqs = [tuple(t.cpu().numpy() for t in r) for r in _requests(case, seed)]
        srv = mc.Server(2 << 30, dtype=case["dtype"], apply=case["apply"], check_every=case["check"], tol=1e-10)
        return dict(kind=kind, reqs=reqs, srv=srv)
    b, x = _inputs(case, seed)
    if kind == "setup":
        return dict(kind=kind, case=case, b=b)
    st = dict(kind=kind, case=case, ch=_chain(case, b), x=x)
    if kind == "sweep":
        st.update(y=torch.empty_like(x), stats=torch.zeros(3, dtype=F64, device="cuda"))
    elif kind == "host":
        st.update(x=x.cpu().pin_memory(), y=torch.empty(x.numel(), dtype=F64).pin_memory())
    elif kind == "solve":
        st.update(x0=x if case["x0"] else None)
    return st


def run(s):
    kind = s["kind"]
    if kind == "sweep":
        s["ch"].sweep(s["x"], s["y"], nsweeps=s["case"]["K"], stats=s["stats"])
        return [s["y"], s["stats"]]
    if kind == "host":
        stats = s["ch"].sweep_host(s["x"], s["y"])
        return [s["y"], stats]
    if kind == "solve":
        pi, _ = s["ch"].solve(x0=s["x0"], tol=1e-12, check_every=s["case"]["check"])
        return pi
    if kind == "setup":
        ch = _chain(s["case"], s["b"])
        return [ch.export(p) for p in (("wlo", "wup") if s["case"]["apply"] == "coupled" else ("lu", "ninv"))]
    srv = s["srv"]
    for tag, blocks in enumerate(s["reqs"]):
        srv.submit(tag, *blocks)
    done = {tag: pi for tag, pi, _, status in srv.run_until_idle() if status == 0}
    return [done[tag] for tag in range(len(s["reqs"]))]


# ---- what a pass cannot do without -----------------------------------------------------------

def _sweep_work(L, m, K, coupled, shape="qbd", far=0, esize=8, inv_esize=8, vec=16):
    """K sweeps: every operator block once a sweep (once in all where they fit on chip), vectors in and out."""
    mm = float(m) * m
    near = 1.5 if shape == "penta" and not coupled else 2.0
    block = (near + far) * mm * esize + (0 if coupled else mm * inv_esize)
    entries = (near + far) * mm + (0 if coupled else mm)
    times = K if block * L > L2_BYTES else 1
    return dict(bytes=block * L * times + vec * float(L) * m * times, flops=2.0 * entries * L * K)


def _solve_work(L, m, dtype, coupled, ratio):
    # sweeps to convergence from a far start: corrections travel the chain, faster at smaller ratios
    K = 12.0 * L * (0.3 + ratio)
    e = {"f64": 8, "f32": 4, "bf16": 2}[dtype]
    return _sweep_work(L, m, K, coupled, esize=e, inv_esize=8 if dtype == "f64" else 4)


def work(case):
    kind = case["kind"]
    if kind == "serve":
        w = dict(bytes=0.0, flops=0.0)
        for r in case["requests"].split():
            size, ratio = r.split(":")
            L, m = (int(v) for v in size.split("x"))
            v = _solve_work(L, m, case["dtype"], case["apply"] == "coupled", float(ratio))
            w = dict(bytes=w["bytes"] + v["bytes"] + 24.0 * L * m * m, flops=w["flops"] + v["flops"] + 2.0 * L * m ** 3)
        return w
    L, m = case["L"], case["m"]
    coupled = case["apply"] == "coupled"
    if kind == "setup":
        return dict(bytes=8.0 * L * m * m * 5, flops=L * float(m) ** 3 * (6 if coupled else 2))
    if kind == "solve":
        return _solve_work(L, m, case["dtype"], coupled, case["ratio"])
    far = max(0, case.get("lower", 1) - 1) + max(0, case.get("upper", 1) - 1)
    return _sweep_work(L, m, case.get("K", 1), coupled, case.get("shape", "qbd"), far)


# ---- the same in plain 64-bit torch ----------------------------------------------------------

def _mv(a, v):
    return torch.matmul(a, v.unsqueeze(2)).squeeze(2)


def _transposed(b, L):
    """{d: Q^T blocks (l, l + d)}, zero where l + d lies outside the chain."""
    if not isinstance(b, dict):
        b = {-1: b[0], 0: b[1], 1: b[2]}
    out = {}
    for e, q in b.items():
        d, t = -e, q.transpose(1, 2)
        r = torch.zeros_like(q)
        lo, hi = max(0, -d), min(L, L - d)
        r[lo:hi] = t[lo + d:hi + d]
        out[d] = r
    return out


def _shifted(v, d):
    """v[l + d], zero outside."""
    r = torch.zeros_like(v)
    L = v.shape[0]
    lo, hi = max(0, -d), min(L, L - d)
    if hi > lo:
        r[lo:hi] = v[lo + d:hi + d]
    return r


def _exact_sweeps(case, b, x):
    L, m, K = case["L"], case["m"], case.get("K", 1)
    T = _transposed(b, L)
    ninv = torch.linalg.inv(T.pop(0)).neg_()
    p = 0 if case.get("stair", 1) == 1 else 1
    h1 = torch.arange(L, device="cuda") % 2 == p
    x = x.reshape(L, m)
    for _ in range(K):
        far = sum((_mv(t, _shifted(x, d)) for d, t in T.items() if abs(d) > 1), torch.zeros_like(x))
        near = lambda v: _mv(T[-1], _shifted(v, -1)) + _mv(T[1], _shifted(v, 1))  # noqa: E731
        z = torch.where(h1[:, None], _mv(ninv, far + near(x)), x)
        z = torch.where(h1[:, None], z, _mv(ninv, far + near(z)))
        s = z.sum()
        y = z / s
        step, x = (y - x).abs().sum(), y
    r = sum(_mv(t, _shifted(x, d)) for d, t in T.items()) - torch.linalg.solve(ninv, x)
    return x.reshape(-1), torch.stack([s, step, r.abs().sum()])


def _exact_pi(b):
    """Stationary vector of a QBD by level reduction from the top (every step keeps its sign)."""
    dn, loc, up = (t if t.shape[1] > 64 else t.cpu() for t in b)
    L, m, _ = loc.shape
    R, S = [None] * L, loc[L - 1]
    for k in range(L - 2, -1, -1):
        R[k] = torch.linalg.solve(S.t(), -up[k].t()).t()
        S = loc[k] + R[k] @ dn[k + 1]
    A = S.t().clone()
    A[-1] = 1.0
    e = torch.zeros(m, dtype=F64, device=A.device)
    e[-1] = 1.0
    v = [torch.linalg.solve(A, e)]
    for k in range(L - 1):
        v.append(v[-1] @ R[k])
    pi = torch.stack(v)
    return (pi / pi.sum()).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return [_exact_pi(r).cpu().numpy() for r in _requests(case, seed)]
    b, x = _inputs(case, seed)
    if kind == "setup":
        T = _transposed(b, case["L"])
        ninv = torch.linalg.inv(T[0]).neg_()
        if case["apply"] == "coupled":   # exported blocks are column-major
            return [(ninv @ T[-1]).transpose(1, 2), (ninv @ T[1]).transpose(1, 2)]
        return [None, ninv.transpose(1, 2)]
    if kind == "solve":
        return _exact_pi(b)
    y, stats = _exact_sweeps(case, b, x)
    if kind == "host":
        return [y.cpu(), stats.tolist()]
    return [y, stats]
