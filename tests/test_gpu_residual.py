"""The direct residual where its kernel changes: teams of warps on short chains, one warp per level on long
ones, against the same sums in plain torch; and the refinement that takes q from the same pass."""
import pytest
import torch

pytestmark = pytest.mark.gpu

mc = pytest.importorskip("paper_2302_07551_gb300")

U = 2.0 ** -53


def generator(L, m, seed, ratio=0.5):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    dn, loc, up = (torch.rand(L, m, m, generator=g, device="cuda", dtype=torch.float64) * 0.9 + 0.1 for _ in range(3))
    up *= ratio
    up[-1] = 0.0
    dn[0] = 0.0
    loc.diagonal(dim1=1, dim2=2).zero_()
    loc.diagonal(dim1=1, dim2=2).sub_(dn.sum(2) + loc.sum(2) + up.sum(2))
    return dn, loc, up


def lines():
    """Level counts on both sides of 6 and 30 times the SMs."""
    n = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152
    return dict(short=6 * n - 1, long=6 * n, most=30 * n)


@pytest.mark.parametrize("which", ["short", "long", "most"])
@pytest.mark.parametrize("m", [8, 33, 40, 48, 65, 72, 96, 100, 104, 127, 130, 160, 161, 200])
def test_residual(m, which):
    """Every row is 3 m products and their sums, the norm a sum over N: (3 m + N / 64 + 32) roundings of the absolute
    sums."""
    L = lines()[which]
    dn, loc, up = generator(L, m, m)
    ch = mc.Chain(dn, loc, up)
    x = torch.rand(L * m, dtype=torch.float64, device="cuda") + 0.01
    x /= x.sum()
    v = x.reshape(L, 1, m)
    # (Q^T x)_l = up_{l-1}^T x_{l-1} + loc_l^T x_l + dn_{l+1}^T x_{l+1}
    parts = [torch.bmm(v, loc), torch.zeros_like(v), torch.zeros_like(v)]
    size = torch.bmm(v, loc.abs())
    parts[1][1:] = torch.bmm(v[:-1], up[:-1])
    parts[2][:-1] = torch.bmm(v[1:], dn[1:])
    ref = sum(parts).abs().sum()
    size = float((size + parts[1] + parts[2]).sum())
    assert abs(ch.residual(x) - float(ref)) <= (3 * m + L * m / 64 + 32) * U * size


@pytest.mark.parametrize("which", ["short", "long"])
@pytest.mark.parametrize("m", [40, 72, 100, 132])
def test_refinement(m, which):
    """q = (-T_dd)^{-1} r comes from the same pass: refinement reaches the FP64 chain's solution."""
    b = generator(lines()[which], m, 2)
    pi, res = mc.Chain(*b, dtype="f32", apply="coupled").solve(tol=1e-12, check_every=32)
    ref, _ = mc.Chain(*b, apply="coupled").solve(tol=1e-12, check_every=32)
    assert res["residual"] <= 1e-12 and float((pi - ref).abs().sum()) <= 1e-10
