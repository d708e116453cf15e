"""Chains kept on chip, in one thread-block cluster or over all SMs: sizes at the edges of the cluster
sizes, of the lanes per level, of the register-held operators and of the shared memory, against the
oracle, and the neighbouring sizes that run through global memory."""
import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

mc = pytest.importorskip("paper_2302_07551_gb300")


# 2 x cluster sizes 1..16, level counts that do not divide, m through every lane group, threads' worth of
# rows (256 per half-sweep and CTA), more, and the largest blocks that still fit
@pytest.mark.parametrize("apply,stair", [("inverse", 1), ("inverse", 2), ("coupled", 1)])
@pytest.mark.parametrize("L,m", [(2, 3), (3, 2), (4, 5), (5, 1), (8, 16), (15, 4), (16, 9), (17, 8), (31, 7),
                                 (32, 1), (33, 16), (63, 15), (100, 8), (257, 16), (300, 12), (513, 4), (1030, 8),
                                 (1100, 3), (700, 2), (90, 33), (35, 47), (34, 60), (150, 32), (2, 90), (2, 160),
                                 (303, 33), (304, 17), (305, 60), (640, 40), (2500, 20), (1250, 32), (5000, 8)])
def test_sweeps_match_the_oracle(L, m, apply, stair):
    """Iterates after K sweeps: 1e-12 relative L1, the suite's bound; e^T z and the residual of the
    last sweep as in the other sweep tests."""
    blocks = synth.qbd(L, m, 0.8, seed=7 * L + m)
    ch = mc.Chain(*(torch.from_numpy(b).cuda() for b in blocks), apply=apply, stair=stair)
    oc = oracle.Chain(*blocks)
    x0 = np.full(L * m, 1.0 / (L * m))
    method = oracle.STAIR1 if stair == 1 else oracle.STAIR2
    for K in (1, 2, 33):
        st = torch.zeros(3, dtype=torch.float64, device="cuda")
        x = ch.sweep(torch.from_numpy(x0).cuda(), nsweeps=K, stats=st).cpu().numpy()
        ref = oc.sweeps(x0, K, method)
        assert np.abs(x - ref).sum() <= 1e-12 * np.abs(ref).sum(), K
        assert abs(float(st[2]) - oc.residual(x)) <= 1e-12 * oc.residual(x) + 8 * m * 2.0 ** -53 * np.abs(blocks[1]).max()
    ch.sync()


def test_in_place_and_repeated_calls_are_bitwise_equal():
    L, m = 200, 8
    blocks = synth.qbd(L, m, 0.8, seed=1)
    ch = mc.Chain(*(torch.from_numpy(b).cuda() for b in blocks))
    x = torch.rand(L * m, dtype=torch.float64, device="cuda")
    x /= x.sum()
    a = ch.sweep(x, nsweeps=5)
    b = ch.sweep(x, nsweeps=5)
    y = x.clone()
    ch.sweep(y, y, nsweeps=5)
    assert torch.equal(a, b) and torch.equal(a, y)


@pytest.mark.parametrize("L,m,n", [(64, 8, 24), (320, 32, 6)])
def test_chains_on_several_streams_at_once(L, m, n):
    """Independent chains, as clusters or as launches over all SMs, in flight on several streams:
    every result equals the one alone."""
    K = 400
    chains, alone = [], []
    x = torch.full((L * m,), 1.0 / (L * m), dtype=torch.float64, device="cuda")
    for i in range(n):
        b = [torch.from_numpy(t).cuda() for t in synth.qbd(L, m, 0.8, seed=i)]
        torch.cuda.synchronize()
        chains.append(mc.Chain(*b, stream=torch.cuda.Stream()))
        alone.append(chains[-1].sweep(x, nsweeps=K))
        torch.cuda.synchronize()
    outs = [torch.empty_like(x) for _ in chains]
    torch.cuda.synchronize()
    for ch, o in zip(chains, outs):
        ch.sweep(x, o, nsweeps=K)
    torch.cuda.synchronize()
    assert all(torch.equal(a, o) for a, o in zip(alone, outs))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("apply", ["inverse", "coupled"])
@pytest.mark.parametrize("L,m", [(2, 4), (33, 8), (64, 12), (305, 32), (600, 24), (400, 64), (40, 100), (900, 96), (306, 256)])
def test_refinement_solutions(L, m, apply, dtype):
    """Solutions from low-precision correction sweeps on chip and by teams of warps, against the
    oracle's FP64 solution: the suite's 1e-10 relative L1."""
    blocks = synth.qbd(L, m, 0.5, seed=L + m)
    ch = mc.Chain(*(torch.from_numpy(b).cuda() for b in blocks), apply=apply, dtype=dtype)
    pi, res = ch.solve(tol=1e-12, check_every=24, maxit=40000)
    assert res["residual"] <= 1e-12
    if L * m * m > 3e6:       # the oracle would take too long: the residual decides
        return
    ref = oracle.Chain(*blocks).solve(tol=1e-13, maxit=40000, check_every=24)["x"]
    assert np.abs(pi.cpu().numpy() - ref).sum() <= 1e-10
    again, _ = ch.solve(tol=1e-12, check_every=24, maxit=40000)
    assert torch.equal(pi, again)


@pytest.mark.parametrize("L,m,apply", [(64, 8, "inverse"), (300, 20, "coupled")])
def test_solve_is_its_chunks(L, m, apply):
    """A solve runs its chunks on the device: the iterate, the sweep count, the step error and the
    contraction are those of the same chunks called one by one (bitwise), whatever stops it."""
    C, n = 7, 5
    ch = mc.Chain(*(torch.from_numpy(b).cuda() for b in synth.qbd(L, m, 0.8, seed=2)), apply=apply)
    x = torch.full((L * m,), 1.0 / (L * m), dtype=torch.float64, device="cuda")
    xs, steps = [], []
    for k in range(n):
        st = torch.zeros(3, dtype=torch.float64, device="cuda")
        x = ch.sweep(x, nsweeps=C, stats=st)
        xs.append(x)
        steps.append(float(st[1]))
    tail = ch.sweep(x, nsweeps=3)
    pi, res = ch.solve(tol=1e-30, maxit=n * C + 3, check_every=C, raise_on_maxit=False)
    assert res["sweeps"] == n * C + 3 and not res["converged"] and torch.equal(pi, tail)
    pi, res = ch.solve(tol=0.0, eps=steps[2], maxit=n * C, check_every=C)
    assert res["sweeps"] == 3 * C and res["converged"] and torch.equal(pi, xs[2])
    assert res["step"] == steps[2]
    assert abs(res["contraction"] - (steps[2] / steps[1]) ** (1 / C)) <= 1e-12
    r = ch.residual(xs[3])
    if r < min(ch.residual(v) for v in xs[:3]):
        pi, res = ch.solve(tol=r * (1 + 1e-6), maxit=n * C, check_every=C)
        assert res["sweeps"] == 4 * C and torch.equal(pi, xs[3])


# both links, the low-precision teams, and chains that never stay on chip
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("apply,stair", [("inverse", 1), ("coupled", 2)])
@pytest.mark.parametrize("L,m", [(2, 4), (64, 8), (305, 32), (600, 24), (2048, 24), (400, 64), (900, 96)])
def test_fp64_sweeps_of_low_precision_chains(L, m, apply, stair, dtype):
    """sweep and sweep_host of a low-precision chain run on its FP64 blocks: the FP64 chain's iterates (the
    suite's 1e-12 relative L1), and they leave the chain's refinement as it was (bitwise)."""
    blocks = [torch.from_numpy(b).cuda() for b in synth.qbd(L, m, 0.5, seed=L + m)]
    ch, ref = mc.Chain(*blocks, apply=apply, stair=stair, dtype=dtype), mc.Chain(*blocks, apply=apply, stair=stair)
    before, _ = ch.solve(tol=1e-12, check_every=24, maxit=40000)
    x = torch.rand(L * m, dtype=torch.float64, device="cuda") + 0.05
    x /= x.sum()
    xh, yh = x.cpu().pin_memory(), torch.empty(L * m, dtype=torch.float64).pin_memory()
    for K in (1, 2, 33):
        st, rs = (torch.zeros(3, dtype=torch.float64, device="cuda") for _ in range(2))
        y, r = ch.sweep(x, nsweeps=K, stats=st), ref.sweep(x, nsweeps=K, stats=rs)
        assert float((y - r).abs().sum()) <= 1e-12
        assert torch.allclose(st[:2], rs[:2], rtol=1e-11, atol=1e-14)
        sh = ch.sweep_host(xh, yh, K)
        assert torch.equal(yh, y.cpu()) and sh == st.tolist()
        after, _ = ch.solve(tol=1e-12, check_every=24, maxit=40000)
        assert torch.equal(before, after)
    ch.sync()


@pytest.mark.parametrize("L,m", [(64, 8), (6000, 64)])
def test_close_keeps_the_workspace_until_the_stream_is_done(L, m):
    """Sweeps may still run on a side stream when a chain is closed: the allocator does not give its workspace,
    which belongs to the stream current at construction, to anyone before they end."""
    blocks = [torch.from_numpy(b).cuda() for b in synth.qbd(L, m, 0.8, seed=1)]
    x = torch.full((L * m,), 1.0 / (L * m), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    ch = mc.Chain(*blocks, stream=st)
    ref = ch.sweep(x, nsweeps=64)
    torch.cuda.synchronize()
    y = torch.empty_like(ref)
    for _ in range(40):
        ch.sweep(x, y, nsweeps=1024)             # tens of milliseconds
    ch.sweep(x, y, nsweeps=64)
    at, size = ch._ws.data_ptr(), ch._ws.numel()
    ch.close()
    del ch
    other = torch.empty(size, dtype=torch.uint8, device="cuda")     # never written
    busy = not st.query()
    assert busy and other.data_ptr() != at
    st.synchronize()
    assert torch.equal(y, ref)
