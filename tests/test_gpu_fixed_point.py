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
