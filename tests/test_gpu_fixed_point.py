"""Sweeps whose products are shared between the FP64 pipe and the integer pipes: every block size
that changes the team of warps or the bounds checks, and inputs that must leave the fixed-point path
(negative, tiny, wide-ranging and zero entries), against the same products in extended
precision from the library's own operators."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

mc = pytest.importorskip("paper_2302_07551_gb300")

U = 2.0 ** -53


def planes(ch, names):
    """Exported operators as (L, m, m) long double arrays, entry (i, j) at [l, i, j]."""
    return [ch.export(n).cpu().numpy().transpose(0, 2, 1).astype(np.longdouble) for n in names]


def one_sweep(ch, x, coupled, stair):
    """One unnormalised sweep from x in long double and the same with absolute values (the scale of
    its rounding errors)."""
    L, m = ch.L, ch.m
    ops = planes(ch, ("wlo", "wup") if coupled else ("tlo", "tup", "ninv"))
    out = []
    for f in (lambda a: a, np.abs):
        y = f(x.reshape(L, m).astype(np.longdouble)).copy()
        for p in (stair - 1, 2 - stair):
            for l in range(p, L, 2):
                g = np.zeros(m, np.longdouble)
                if l > 0:
                    g += f(ops[0][l]) @ y[l - 1]
                if l < L - 1:
                    g += f(ops[1][l]) @ y[l + 1]
                y[l] = g if coupled else f(ops[2][l]) @ g
        out.append(y)
    return out


def check(ch, x, coupled=False, stair=1):
    """One sweep on the GPU.  Every row is at most 2 x 3m products and sums of two half-sweeps, a sum
    of N terms and a division: (6m + N/64 + 32) roundings of the absolute sums bound the error (the
    sum over N is a tree)."""
    got = ch.sweep(torch.from_numpy(x).cuda(), nsweeps=1).cpu().numpy().reshape(ch.L, ch.m)
    ref, mag = one_sweep(ch, x, coupled, stair)
    s = ref.sum()
    tol = (6 * ch.m + ch.N / 64 + 32) * U * (mag / abs(s) + np.abs(ref / s) * (mag.sum() / abs(s)))
    err = np.abs(got - ref / s)
    assert np.all(np.isfinite(got))
    assert np.all(err <= tol + 5e-324), (float((err / (tol + 1e-320)).max()), np.argmax(err))
    return got


def chain(blocks, **kw):
    return mc.Chain(*(torch.from_numpy(np.ascontiguousarray(b)).cuda() for b in blocks), **kw)


def start(L, m, seed=3):
    x = np.random.default_rng(seed).random(L * m) + 0.01
    return x / x.sum()


# m: edges of the 32-row groups and of the teams; L: shorter and longer than the teams in flight
@pytest.mark.parametrize("apply,stair", [("inverse", 1), ("coupled", 2)])
@pytest.mark.parametrize("L,m", [(2, 1), (9, 7), (40, 31), (41, 32), (40, 33), (33, 64), (9000, 17), (12001, 64),
                                 (21, 65), (20, 96), (19, 100), (21, 128), (9, 129), (8, 160), (9, 192), (7, 193),
                                 (6, 255), (7, 256), (2800, 96), (2000, 130)])
def test_block_sizes(L, m, apply, stair):
    if L * m * m > 4e7:
        pytest.skip("extended-precision reference would take too long")
    ch = chain(synth.qbd(L, m, 0.8, seed=L + m), apply=apply, stair=stair)
    check(ch, start(L, m), apply == "coupled", stair)


@pytest.mark.parametrize("apply", ["inverse", "coupled"])
@pytest.mark.parametrize("m", [24, 64, 100])
@pytest.mark.parametrize("kind", ["negative", "tiny_rows", "zero_rows", "tiny_block", "wide_vector", "tiny_level",
                                  "zero_vector_parts"])
def test_inputs_outside_the_window(kind, m, apply):
    L = 280 if m == 24 else 12   # beyond the chains that stay resident in one cluster
    dn, loc, up = (b.copy() for b in synth.qbd(L, m, 0.8, seed=5))
    x = start(L, m)
    if kind == "negative":            # one negative rate: that block runs in FP64 alone
        up[3, 2, 4] = -abs(up[3, 2, 5]) - 0.01
    elif kind == "tiny_rows":         # rows of Q^T far below the block's largest entry
        dn[:, :, : m // 3] *= 2.0 ** -75
        up[:, :, : m // 3] *= 2.0 ** -75
    elif kind == "zero_rows":
        dn[:, :, : m // 3] = 0.0
        up[:, :, : m // 3] = 0.0
    elif kind == "tiny_block":        # largest entry below the smallest exponent of the path
        up[4] *= 1e-270
    elif kind == "wide_vector":
        x.reshape(L, m)[:, ::3] *= 2.0 ** -80
    elif kind == "tiny_level":
        x.reshape(L, m)[5:] *= 1e-290
    elif kind == "zero_vector_parts":
        x.reshape(L, m)[:, m // 2:] = 0.0
        x.reshape(L, m)[7] = 0.0
    ch = chain((dn, loc, up), apply=apply)
    check(ch, x, apply == "coupled")


@pytest.mark.parametrize("m", [20, 64])
def test_not_a_number_propagates(m):
    ch = chain(synth.qbd(8, m, 0.8, seed=9))
    x = start(8, m)
    x[m + 3] = np.nan        # level 1: read by the first half-sweep
    y = torch.empty(8 * m, dtype=torch.float64, device="cuda")
    ch.sweep(torch.from_numpy(x).cuda(), y, nsweeps=1)
    with pytest.raises(mc.McError):
        ch.sync()
    assert torch.isnan(y).any()


# ---- chains through global memory, in every team form ----------------------------------------

def rates(L, m, seed, ratio=0.8, line=False):
    """Generator blocks on the GPU: random rates, or (line) phases that only exchange with their neighbours, weakly
    upwards, and levels that keep the phase."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    r = lambda: (torch.rand(L, m, m, generator=g, device="cuda", dtype=torch.float64) * 0.9 + 0.1)  # noqa: E731
    up, dn, loc = r(), r(), r()
    if line:
        i = torch.arange(m, device="cuda")
        near = (i[:, None] - i[None, :]).abs()
        up, dn = up * (near == 0), dn * (near == 0)
        loc = loc * (near == 1) * torch.where(i[None, :] > i[:, None], 0.1, 1.0)
    return dn / ratio, loc, up


def close_rows(dn, loc, up):
    up[-1] = 0.0
    dn[0] = 0.0
    loc.diagonal(dim1=1, dim2=2).zero_()
    loc.diagonal(dim1=1, dim2=2).sub_(dn.sum(2) + loc.sum(2) + up.sum(2))
    return dn, loc, up


def check_levels(ch, x, coupled, levels, stair=1):
    """check() on some levels of a long chain: the sweep's own e^T z scales them, and the result sums to 1."""
    L, m = ch.L, ch.m
    st = torch.zeros(3, dtype=torch.float64, device="cuda")
    got = ch.sweep(torch.from_numpy(x).cuda(), nsweeps=1, stats=st).cpu().numpy().reshape(L, m)
    ch.sync()
    s = float(st[0])
    assert abs(got.sum() - 1.0) <= (L * m / 64 + 32) * U * np.abs(got).sum()
    x = x.reshape(L, m).astype(np.longdouble)

    def level(l, y, f):
        names = ("wlo", "wup") if coupled else ("tlo", "tup", "ninv")
        ops = [f(ch.export(n, l, 1).cpu().numpy()[0].T.astype(np.longdouble)) for n in names]
        g = sum((op @ y(l + d) for op, d in zip(ops, (-1, 1)) if 0 <= l + d < L), np.zeros(m, np.longdouble))
        return g if coupled else ops[2] @ g

    for l in levels:
        for f in (lambda a: a, np.abs):
            first = lambda k: f(x[k])  # noqa: E731
            z = level(l, first if l % 2 == stair - 1 else lambda k: level(k, first, f), f)
            if f is np.abs:
                mag = z
            else:
                ref = z
        tol = (6 * m + ch.N / 64 + 32) * U * (mag / abs(s) + 2 * np.abs(ref / s))
        err = np.abs(got[l] - ref / s)
        assert np.all(err <= tol + 5e-324), (l, float((err / (tol + 1e-320)).max()))


# teams of one to eight warps with one or two rows a lane, with and without bounds checks: shorter and
# longer than half as many levels again as a half-sweep has teams
TEAMS = [(4000, 24), (2200, 32), (2200, 33), (600, 64), (40, 100), (30, 128), (24, 150), (20, 192), (16, 224), (16, 256),
         (11000, 40), (11000, 64), (5500, 72), (5500, 128), (3700, 136), (3700, 192), (2750, 200), (2750, 256)]


def sample(L, n=10, seed=1):
    return sorted({0, 1, L - 2, L - 1, *(int(v) for v in np.random.default_rng(seed).integers(0, L, n))})


@pytest.mark.parametrize("apply,stair", [("inverse", 1), ("coupled", 2)])
@pytest.mark.parametrize("L,m", TEAMS)
def test_every_team(L, m, apply, stair):
    ch = mc.Chain(*close_rows(*rates(L, m, m)), apply=apply, stair=stair)
    x = start(L, m)
    assert ch.profile(torch.from_numpy(x).cuda())[1]["launches"] == 3     # sweeps, scale, normalisation
    check_levels(ch, x, apply == "coupled", sample(L), stair)


KINDS = ["negative", "weak_rows", "zero_rows", "small_block", "wide_vector", "wide_both", "small_level", "zeros", "line", "line_zeros"]


@pytest.mark.parametrize("apply", ["inverse", "coupled"])
@pytest.mark.parametrize("L,m", [(4000, 24), (2200, 32), (2200, 33), (600, 64), (40, 100), (11000, 64), (5500, 100)])
@pytest.mark.parametrize("kind", KINDS)
def test_outside_the_window_in_every_form(kind, L, m, apply):
    dn, loc, up = rates(L, m, 7, line=kind.startswith("line"))
    x = start(L, m).reshape(L, m)
    k = L // 2
    if kind == "weak_rows":           # rows of Q^T below the block's largest entry by more than the window
        up[:, :, : m // 3] *= 2.0 ** -75
    elif kind == "zero_rows":
        dn[:, :, : m // 3] = 0.0
        up[:, :, : m // 3] = 0.0
    elif kind == "small_block":
        up[k] *= 1e-270
    elif kind == "wide_vector":       # rows keep a large entry, but it may meet a small one
        x[:, ::3] *= 2.0 ** -60
    elif kind == "wide_both":         # block and vector together beyond the window, neither alone
        dn[:, :, : m // 3] *= 2.0 ** -30
        up[:, :, : m // 3] *= 2.0 ** -30
        x[:, 1::2] *= 2.0 ** -30
    elif kind == "small_level":
        x[k:] *= 1e-290
    elif kind in ("zeros", "line_zeros"):
        x[:, m // 2:] = 0.0
        x[k] = 0.0
    elif kind == "line":
        x *= 0.1 ** np.arange(m)
    close_rows(dn, loc, up)
    if kind == "negative":
        up[k, 2, 4] = -0.25
    ch = mc.Chain(dn, loc, up, apply=apply)
    x = np.ascontiguousarray(x.reshape(-1) / x.sum())
    assert ch.profile(torch.from_numpy(x).cuda())[1]["launches"] == 3
    check_levels(ch, x, apply == "coupled", sorted({*sample(L, 4), k - 1, k, k + 1}))


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("L,m", [(4000, 24), (600, 64), (40, 100), (11000, 64)])
def test_non_finite_entries_propagate(L, m, value):
    ch = mc.Chain(*close_rows(*rates(L, m, 3)))
    x = start(L, m)
    x[m + 3] = value         # level 1: read by the first half-sweep
    y = ch.sweep(torch.from_numpy(x).cuda(), nsweeps=1)
    with pytest.raises(mc.McError):
        ch.sync()
    assert not torch.isfinite(y).all()


@pytest.mark.parametrize("kind", ["weak_rows", "line", "transient"])
@pytest.mark.parametrize("apply", ["inverse", "coupled"])
def test_banded_and_served_chains_outside_the_window(kind, apply):
    """192 sweeps by the server's teams against a chain of its own and, inverse, the far terms of a banded chain against
    the same chain with its near blocks only (the further ones vanish beside them): 6 m roundings a sweep."""
    L, m, K, n = 600, 40, 64, 3
    dn, loc, up = rates(L, m, 9, line=kind == "line")
    if kind == "weak_rows":
        up[:, :, : m // 3] *= 2.0 ** -75
    elif kind == "transient":         # the second half of the phases is left and never entered
        for t in (dn, loc, up):
            t[:, : m // 2, m // 2:] = 0.0
    dn, loc, up = close_rows(dn, loc, up)

    def sweeps(ch):
        x = torch.full((L * m,), 1.0 / (L * m), dtype=torch.float64, device="cuda")
        for _ in range(n):
            x = ch.sweep(x, nsweeps=K)
        ch.sync()
        return x.cpu().numpy()

    pi = sweeps(mc.Chain(dn, loc, up, apply=apply))
    srv = mc.Server(1 << 30, dtype="f64", apply=apply, check_every=K, tol=0.0, maxit=n * K, autotune=False)
    assert srv.submit(0, *(t.cpu().numpy() for t in (dn, loc, up)))
    (_, ps, _, _), = srv.run_until_idle()
    assert np.abs(ps - pi).sum() <= n * K * 6 * m * U
    srv.close()
    if apply == "inverse":
        far = torch.zeros_like(dn)
        far[:L - 2] = 2.0 ** -80 * dn[:L - 2]          # its rows lie far below those of the near blocks
        pb = sweeps(mc.Chain.banded({-1: dn, 0: loc, 1: up, 2: far}))
        assert np.abs(pb - pi).sum() <= n * K * 6 * m * U
