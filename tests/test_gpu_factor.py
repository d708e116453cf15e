"""Set-up kernels at the sizes where their tiles, grids and launches change: the LU factors, the
inverse and the coupled operators against the blocks themselves in extended precision, and blocks
without a usable pivot."""
from fractions import Fraction

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

mc = pytest.importorskip("paper_2302_07551_gb300")

U = 2.0 ** -53
LD = np.longdouble
SIZES = [1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 47, 48, 49, 64, 65, 80, 81, 96, 97, 112, 113, 127, 128, 129, 160,
         161, 192, 193, 224, 225, 255, 256]


def chain(blocks, **kw):
    return mc.Chain(*(torch.from_numpy(np.ascontiguousarray(b)).cuda() for b in blocks), **kw)


def plane(ch, name):
    return ch.export(name).cpu().numpy().transpose(0, 2, 1).astype(LD)


@pytest.mark.parametrize("m", SIZES)
def test_factors_inverse_and_products(m):
    """|L U - T| <= (3m + 8) u |L||U| (m updates of an entry, three roundings each); the inverse's
    residual |N T + I| <= 16 m u |N||L||U| entrywise (Gauss-Jordan, dominant columns); each entry of
    W = N T is m products and sums: (m + 8) u |N||T|."""
    L = 5 if m > 64 else 37       # more than one round of half-warps, ragged
    ch = chain(synth.qbd(L, m, 0.85, seed=m), apply="coupled")
    T, LU, N = plane(ch, "tdd"), plane(ch, "lu"), plane(ch, "ninv")
    lo, wl = plane(ch, "tlo"), plane(ch, "wlo")
    up, wu = plane(ch, "tup"), plane(ch, "wup")
    for l in range(0, L, 1 if m > 64 else 6):
        lower, upper = np.tril(LU[l], -1) + np.eye(m, dtype=LD), np.triu(LU[l])
        size = np.abs(lower) @ np.abs(upper)
        assert np.all(np.abs(lower @ upper - T[l]) <= (3 * m + 8) * U * size)
        assert np.all(np.abs(N[l] @ T[l] + np.eye(m)) <= 16 * m * U * (np.abs(N[l]) @ size) + 8 * U)
        for w, t in ((wl, lo), (wu, up)):
            assert np.all(np.abs(w[l] - N[l] @ t[l]) <= (m + 8) * U * (np.abs(N[l]) @ np.abs(t[l])))


@pytest.mark.parametrize("m", [20, 40, 130])
@pytest.mark.parametrize("kind", ["negative", "tiny_rows", "tiny_block", "zero_columns"])
def test_products_outside_the_fixed_point_window(kind, m):
    L = 4
    dn, loc, up = (b.copy() for b in synth.qbd(L, m, 0.85, seed=m + 1))
    if kind == "negative":
        up[1, 3, 2] = -0.25
    elif kind == "tiny_rows":
        up[:, :, : m // 2] *= 2.0 ** -90
    elif kind == "tiny_block":
        up[1] *= 1e-280
    else:
        up[:, m // 3:, :] = 0.0
    ch = chain((dn, loc, up), apply="coupled")
    N, lo, w = plane(ch, "ninv"), plane(ch, "tlo"), plane(ch, "wlo")
    for l in range(L):
        assert np.all(np.abs(w[l] - N[l] @ lo[l]) <= (m + 8) * U * (np.abs(N[l]) @ np.abs(lo[l])))


@pytest.mark.parametrize("m", [1, 8, 16, 33, 64, 128, 129, 256])
@pytest.mark.parametrize("where", [0.0, 0.5, 1.0])
def test_a_block_without_pivot_is_reported(m, where):
    """A zero pivot at the first, a middle and the last step of one block of several."""
    L, k = 6, int(round(where * (m - 1)))
    dn, loc, up = (b.copy() for b in synth.qbd(L, m, 0.85, seed=3))
    loc[4, k, :] = 0.0            # Q^T's column k: the pivot of step k is zero
    with pytest.raises(mc.McError) as e:
        chain((dn, loc, up))
    assert e.value.status == 4
    chain(synth.qbd(L, m, 0.85, seed=3)).close()


def closed_pair(loc, level, k, a, b):
    """Phases k and k + 1 of one level only exchange with each other: a generator block of its own."""
    loc[level, k:k + 2, :] = 0.0
    loc[level, :, k:k + 2] = 0.0
    loc[level, k:k + 2, k:k + 2] = [[-a, a], [b, -b]]


@pytest.mark.parametrize("m,k,n", [(2, 0, 200), (2, 0, 0), (12, 3, 24), (24, 20, 24), (130, 0, 12)])
def test_a_level_that_exchanges_with_itself_only_is_reported(m, k, n):
    """The second pivot of such a pair is b - a (b / a) = 0 exactly when a / -a is -1, whatever the rates: n random
    pairs, or (n = 0) the integers up to 199, of which some have a (1 / a) != 1."""
    base = [np.ascontiguousarray(b) for b in synth.qbd(3, m, 0.85, seed=3)]
    rng = np.random.default_rng(11)
    pairs = rng.random((n, 2)) + 0.01 if n else [(float(i), 1.0 + i % 7) for i in range(1, 200)]
    dn, up = (torch.from_numpy(base[i]).cuda() for i in (0, 2))
    for a, b in pairs:
        loc = base[1].copy()
        closed_pair(loc, 1, k, a, b)
        with pytest.raises(mc.McError) as e:
            mc.Chain(dn, torch.from_numpy(loc).cuda(), up)
        assert e.value.status == 4, (a, b)


@pytest.mark.parametrize("m,k", [(2, 0), (12, 3), (24, 20), (64, 62), (130, 0)])
def test_a_pair_that_nearly_closes_is_factored_as_by_plain_lu(m, k):
    """The pair loses a few units in the last place of its rates: the second pivot is what one division and one
    fused multiply-add leave, accepted unless that is zero; the inverse as in the other blocks."""
    base = [np.ascontiguousarray(b) for b in synth.qbd(30, m, 0.85, seed=3)]
    rng = np.random.default_rng(5)
    dn, loc, up = base
    want, l = {}, 1
    while len(want) < 20:
        a, b = rng.random(2) + 0.01
        closed_pair(loc, l, k, a, b)
        loc[l, k, k] -= int(rng.integers(0, 9)) * np.spacing(a)
        loc[l, k + 1, k + 1] -= int(rng.integers(0, 9)) * np.spacing(b)
        t = loc[l, k:k + 2, k:k + 2].T                  # the block of Q^T
        c = t[1, 0] / t[0, 0]
        piv = float(Fraction(t[1, 1]) - Fraction(c) * Fraction(t[0, 1]))
        if piv != 0.0:
            want[l] = (c, piv)
            l += 1
    ch = chain((dn, loc, up))
    T, LU, N = plane(ch, "tdd"), plane(ch, "lu"), plane(ch, "ninv")
    for l, (c, piv) in want.items():
        assert LU[l, k + 1, k] == c and LU[l, k + 1, k + 1] == piv
        size = np.abs(np.tril(LU[l], -1) + np.eye(m)) @ np.abs(np.triu(LU[l]))
        assert np.all(np.abs(N[l] @ T[l] + np.eye(m)) <= 16 * m * U * (np.abs(N[l]) @ size) + 8 * U)
