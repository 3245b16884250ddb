"""Splits and synchronisations of matrices that hold a NaN or an infinity: every kernel stays inside its buffers (indices come from
comparisons), what comes out is not finite either, and the next call is as good as any.  Workspaces are filled with ones first, so that
an index nobody wrote would show."""
import pytest
import torch

from paper_2405_01067_b200 import binding as ab

pytestmark = pytest.mark.gpu


def _normal(*shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda")


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("m,n", [(70, 64), (256, 300), (300, 257), (800, 768), (1200, 1190), (1250, 1200)])
def test_split(m, n, value):
    W, k = _normal(m, n, seed=1), min(m, n) // 4
    good = ab.ab_svd_split(W, k, 0.0)
    bad = W.clone()
    bad[m // 2, 7] = value
    ws = ab.workspace(ab.ab_workspace_bytes(ab.AB_OP_SVD_SPLIT, 0, m, n, k, 1, ab.AB_F32), "cuda")
    ws.fill_(1)
    A, B, sigma, r_out, _ = ab.ab_svd_split(bad, k, 0.0, ws=ws)
    torch.cuda.synchronize()
    assert not bool(torch.isfinite(sigma).all()) and 1 <= int(r_out) <= k
    assert not bool(torch.isfinite(A).all() and torch.isfinite(B).all())
    again = ab.ab_svd_split(W, k, 0.0, ws=ws)
    assert all(torch.equal(a, b) for a, b in zip(good, again))


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("s", [64, 300, 768])
def test_fallback(s, value):
    """The Jacobi routes, also beside matrices that are fine."""
    W = torch.stack([_normal(s + 8, s, seed=i) for i in range(3)])
    bad = W.clone()
    bad[1, 3, 5] = value
    good = ab.ab_selftest_split_fallback(W, s // 4, 0b110)
    got = ab.ab_selftest_split_fallback(bad, s // 4, 0b110)
    torch.cuda.synchronize()
    assert not bool(torch.isfinite(got[0][1]).all() and torch.isfinite(got[1][1]).all())
    assert all(torch.equal(a[i], b[i]) for a, b in zip(good, got) for i in (0, 2))


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("path", [ab.AB_SYNC_FACTORED, ab.AB_SYNC_DENSE])
@pytest.mark.parametrize("r", [20, 130, 192])
def test_group_sync(r, path, value):
    A, B = [_normal(2, 300, r, seed=i) for i in range(3)], [_normal(2, r, 260, seed=9 + i) for i in range(3)]
    good = ab.SyncPlan(A, B, 0.1)
    ab.ab_group_sync(good, path=path)
    bad = [a.clone() for a in A]
    bad[1][0, 3, 5] = value
    plan = ab.SyncPlan(bad, B, 0.1)
    plan.ws.fill_(1)
    ab.ab_group_sync(plan, path=path)
    torch.cuda.synchronize()
    assert not bool(torch.isfinite(plan.A_out[1]).all() and torch.isfinite(plan.B_out[1]).all())
    for i in (0, 2):
        assert torch.equal(plan.A_out[i], good.A_out[i]) and torch.equal(plan.sigma[i], good.sigma[i])
