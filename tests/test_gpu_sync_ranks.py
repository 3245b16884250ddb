"""The factored group synchronisation at ranks around the panels and steps of its Cholesky elimination, against float64.

Tolerance: Gram matrices are good to 1e-6 (the split product's bound); the factors' condition number is at most
(1 + 1/2) / (1 - 1/2) = 3 for sides of at least 4 r, it enters squared, once for each side: 2 * 9 * 1e-6.
"""
import pytest
import torch

from paper_2405_01067_b200 import binding as ab

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ranks", [(1, 7, 8, 9), (16, 31, 33, 63), (64, 65, 100, 129), (192,), (228,)])
def test_sync_keeps_the_mean_product(ranks):
    g = torch.Generator(device="cuda").manual_seed(sum(ranks))
    K, A, B = 2, [], []
    for i, r in enumerate(ranks):
        m, n = 4 * r + 5 + i, 4 * r + 64
        A.append(torch.randn((K, m, r), generator=g, device="cuda"))
        B.append(torch.randn((K, r, n), generator=g, device="cuda"))
    plan = ab.SyncPlan(A, B, 0.0)
    ab.ab_group_sync(plan)
    for a, b, ao, bo in zip(A, B, plan.A_out, plan.B_out):
        W = a.double().mean(0) @ b.double().mean(0)
        assert float((ao.double() @ bo.double() - W).norm() / W.norm()) <= 1.8e-5
