"""The solve server's three ways to run a request's correction sweeps (one cluster, teams of warps,
shared queue): sizes on both sides of the lines between them, against the oracle, and bitwise the same
alone and in a mix that uses all of them at once."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

mc = pytest.importorskip("paper_2302_07551_gb300")

# cluster: L below, at and above 2 x 16, m to 32; teams: m = 36 (FP32), 40, 72, 136; queue: m = 36
# (BF16: no 16-byte columns) and more levels than teams
SIZES = [(2, 4), (31, 8), (32, 16), (33, 12), (300, 32), (20, 36), (40, 40), (21, 72), (12, 136), (7, 256), (1300, 64)]


def blocks(i, L, m):
    return synth.qbd(L, m, 0.5, seed=900 + i)


@pytest.mark.parametrize("apply,stair", [("inverse", 1), ("coupled", 2)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_every_path_alone_and_together(dtype, apply, stair):
    kw = dict(dtype=dtype, apply=apply, stair=stair, tol=1e-11, check_every=24)
    srv = mc.Server(2 << 30, autotune=True, **kw)
    for i, (L, m) in enumerate(SIZES):
        assert srv.submit(i, *blocks(i, L, m))
    mixed = {t: (pi, r, st) for t, pi, r, st in srv.run_until_idle()}
    srv.close()
    alone = mc.Server(1 << 30, autotune=False, **kw)
    for i, (L, m) in enumerate(SIZES):
        pi, r, st = mixed[i]
        assert st == 0 and r["residual"] <= 1e-11
        if L < 1000:
            ref = oracle.Chain(*blocks(i, L, m)).solve(tol=1e-13, maxit=100000, check_every=24)["x"]
            assert np.abs(pi - ref).sum() <= 1e-9      # residual 1e-11: the suite's 1e-10 needs 1e-12
        alone.submit(i, *blocks(i, L, m))
        (_, pa, ra, _), = alone.run_until_idle()
        assert ra["sweeps"] == r["sweeps"] and np.array_equal(pa, pi), (L, m)
    alone.close()


# FP64: clusters of 1 to 16 CTAs, below and above one cluster's shared memory (147 and 300 levels of
# 32), teams of 2, 4 and 8 warps at the edges of their rows, odd sizes
SIZES64 = [(2, 3), (31, 8), (33, 16), (140, 32), (300, 32), (2, 33), (41, 64), (20, 65), (17, 100), (16, 128), (9, 129), (7, 256)]


@pytest.mark.parametrize("apply,stair", [("inverse", 1), ("inverse", 2), ("coupled", 1), ("coupled", 2)])
@pytest.mark.parametrize("check", [1, 24])
def test_every_fp64_path_alone_and_together(apply, stair, check):
    kw = dict(dtype="f64", apply=apply, stair=stair, tol=1e-12, check_every=check)
    sizes = SIZES64 if check > 1 else SIZES64[::3]
    srv = mc.Server(2 << 30, autotune=check > 1, **kw)
    for i, (L, m) in enumerate(sizes):
        assert srv.submit(i, *blocks(i, L, m))
    mixed = {t: (pi, r, st) for t, pi, r, st in srv.run_until_idle()}
    srv.close()
    alone = mc.Server(1 << 30, autotune=False, **kw)
    for i, (L, m) in enumerate(sizes):
        pi, r, st = mixed[i]
        assert st == 0 and r["residual"] <= 1e-12
        ref = oracle.Chain(*blocks(i, L, m)).solve(tol=1e-13, maxit=2000, check_every=24)["x"]   # 864 at most; 7 x 256 ends at its floor, 1.6e-13
        assert np.abs(pi - ref).sum() <= 1e-10
        alone.submit(i, *blocks(i, L, m))
        (_, pa, ra, _), = alone.run_until_idle()
        assert ra["sweeps"] == r["sweeps"] and np.array_equal(pa, pi), (L, m)
    alone.close()


def test_long_chains_of_small_fp64_blocks():
    """Both sides of the line between teams of one warp and the shared queue (m <= 16, a level a half-sweep for
    each of 24 warps an SM), against the oracle and bitwise as alone."""
    n = 2 * 24 * torch.cuda.get_device_properties(0).multi_processor_count
    kw = dict(dtype="f64", apply="coupled", tol=0.0, check_every=4, autotune=False, maxit=4)
    sizes = [(n, 3), (n - 2, 4), (n + 1, 16), (n + 3, 17)]
    srv = mc.Server(4 << 30, **kw)
    for i, (L, m) in enumerate(sizes):
        assert srv.submit(i, *blocks(i, L, m))
    mixed = {t: pi for t, pi, r, st in srv.run_until_idle()}
    for i, (L, m) in enumerate(sizes):
        srv.submit(i, *blocks(i, L, m))
        (_, pa, _, _), = srv.run_until_idle()
        assert np.array_equal(pa, mixed[i])
        ref = oracle.Chain(*blocks(i, L, m)).sweeps(np.full(L * m, 1.0 / (L * m)), 4)
        assert np.abs(pa - ref).sum() <= 1e-12     # 4 sweeps of sums of 3 m terms >= 0: below 1e-14
    srv.close()


def copies(sizes, n, **kw):
    """Every size n times in one server, and once in a server of its own: statuses and results."""
    srv = mc.Server(4 << 30, autotune=False, max_active=1000, **kw)
    for c in range(n):
        for i, (L, m) in enumerate(sizes):
            assert srv.submit(c * len(sizes) + i, *blocks(i, L, m))
    mixed = {t: (pi, r["sweeps"]) for t, pi, r, st in srv.run_until_idle()}
    assert len(mixed) == n * len(sizes)
    srv.close()
    alone = mc.Server(1 << 30, autotune=False, **kw)
    for i, (L, m) in enumerate(sizes):
        alone.submit(i, *blocks(i, L, m))
        (_, pa, ra, _), = alone.run_until_idle()
        for c in range(n):
            pi, sweeps = mixed[c * len(sizes) + i]
            assert sweeps == ra["sweeps"] and np.array_equal(pa, pi), (L, m, c)
    alone.close()


# every way the resident kernels split a row's columns (by lanes, by warps, not at all), clusters of 1 to
# 16 CTAs with equal and unequal shares; four of each are more than clusters are given, and fewer again
# once the first have converged
SMALL64 = [(2, 3), (3, 1), (5, 2), (8, 4), (31, 8), (33, 16), (60, 32), (140, 32), (90, 24), (64, 5), (200, 8), (100, 13),
           (35, 20), (17, 31), (500, 3), (16, 17), (70, 11), (33, 2), (400, 10), (250, 16)]


@pytest.mark.parametrize("apply,stair", [("inverse", 1), ("coupled", 2)])
@pytest.mark.parametrize("check,stop", [(24, dict(tol=1e-12)), (1, dict(tol=0.0, maxit=5)), (2, dict(tol=0.0, maxit=6))])
def test_many_small_fp64_requests_are_as_alone(apply, stair, check, stop):
    """Below and above the line between clusters and the shared queue the iterates are the same bits."""
    copies(SMALL64, 4, dtype="f64", apply=apply, stair=stair, check_every=check, **stop)


# shared memory of a CTA for four, two and one to an SM, blocks of up to 16 rows and wider
@pytest.mark.parametrize("apply", ["inverse", "coupled"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_many_small_low_precision_requests_are_as_alone(dtype, apply):
    copies([(128, 16), (33, 4), (1500, 8), (2600, 8), (64, 32), (40, 24), (100, 28), (140, 32), (200, 32), (300, 32), (450, 32)], 4,
           dtype=dtype, apply=apply, check_every=24, tol=1e-11)


@pytest.mark.parametrize("apply,check", [("inverse", 24), ("coupled", 24), ("coupled", 1)])
def test_small_blocks_move_between_teams_and_queue(apply, check):
    """Long FP64 chains of up to 16 rows run by teams while few are active and on the queue while many are; a
    request that goes from one to the other and back has the bits of one that never did."""
    kw = dict(dtype="f64", apply=apply, check_every=check, tol=0.0, maxit=5 * check, autotune=False)
    waves = {0: [(2000, 16), (9000, 5), (4000, 9)], 2: [(2500, 12)] * 6 + [(3001, 10)], 3: [(2000, 16), (4001, 9)]}
    srv, got, want, tag = mc.Server(4 << 30, **kw), {}, [], 0
    for step in range(8):
        for size in waves.get(step, []):
            assert srv.submit(tag, *blocks(tag, *size))
            want.append(size)
            tag += 1
        srv.step()
        while (r := srv.fetch()) is not None:
            got[r[0]] = r[1]
    srv.close()
    assert len(got) == len(want)
    alone = mc.Server(1 << 30, **kw)
    for i, size in enumerate(want):
        alone.submit(i, *blocks(i, *size))
        (_, pa, _, _), = alone.run_until_idle()
        assert np.array_equal(pa, got[i]), (i, size)
    alone.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_every_group_beside_teams(dtype):
    """All resident groups, teams of all size classes and the queue in one batch: each gets its part."""
    copies([(128, 16), (2600, 8), (64, 32), (100, 28), (200, 32), (450, 32), (40, 40), (21, 72), (12, 136), (1300, 64)], 2,
           dtype=dtype, apply="inverse", check_every=24, tol=1e-11)


def test_a_queue_has_a_signature_of_its_own():
    """Batches of the same size classes and level count, one by teams alone, one with the queue: what the autotuner
    kept for the first does not decide for the second."""
    srv = mc.Server(4 << 30, dtype="f32", apply="coupled", check_every=8, tol=0.0, maxit=160, max_active=1000)
    sigs = []
    for L, m, n in [(300, 64, 8), (2400, 64, 1)]:       # 2400 levels: more than teams for all of a half-sweep
        before = len(srv.trials())
        for i in range(n):
            assert srv.submit(i, *blocks(i, L, m))
        srv.run_until_idle()
        sigs.append({t["signature"] for t in srv.trials()[before:]})
    srv.close()
    assert sigs[0] and sigs[1] and not sigs[0] & sigs[1]
    assert all(s & 16 for s in sigs[1]) and not any(s & 16 for s in sigs[0])
