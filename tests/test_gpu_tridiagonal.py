"""The tridiagonal problem of the direct eigensolver where its recurrences scale: couplings between rows from the size of the
diagonal down to the one at which the matrix is split, in runs, alternating, and across the groups of eight rows that are
scaled together.

W is upper bidiagonal, so W^T W is tridiagonal before the solver touches it.  Tolerance: as in test_gpu_eig.py (the fp32 Gram matrix
fixes sigma to 2^-24 sqrt(s) sigma_1^2 / sigma; values stay above 0.2 sigma_1).
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ab():
    from paper_2405_01067_b200 import binding
    binding.lib()
    return binding


def couplings(kind, s):
    k = np.arange(s - 1)
    if kind == "graded":                     # 1e-1 ... 1e-17: some split, some only just do not
        return 10.0 ** -(1 + 16 * k / max(1, s - 2))
    if kind == "alternating":                # beta of the scaled recurrence swings by 1e30 from row to row
        return np.where(k % 2 == 0, 0.1, 1e-15)
    if kind == "tiny":                       # eight rows at a time at the edge of a split
        return np.full(s - 1, 1e-15)
    if kind == "groups":                     # splits in the middle of groups of eight rows
        return np.where(k % 11 == 5, 0.0, 0.05)
    return np.where(k % 16 < 8, 0.1, 3e-16)


@pytest.mark.parametrize("kind", ["graded", "alternating", "tiny", "groups", "blocks"])
@pytest.mark.parametrize("s,need", [(7, 7), (40, 12), (64, 64), (192, 50), (256, 256), (300, 100), (768, 192)])
def test_small_couplings(ab, s, need, kind):
    W = np.diag(np.linspace(1.0, 0.2, s)) + np.diag(couplings(kind, s), 1)
    W = W.astype(np.float32)
    A, B, sigma, r_out, status = ab.ab_svd_split(torch.from_numpy(W).cuda(), need, 0.0)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and int(r_out.item()) == need
    ref = np.linalg.svd(W.astype(np.float64), compute_uv=False)
    sg = sigma.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(sg - ref[:need]) <= 1e-4 * ref[:need])
    Ah, Bh = A.cpu().numpy().astype(np.float64), B.cpu().numpy().astype(np.float64)
    res = np.linalg.norm(W - Ah @ Bh)
    assert abs(res - np.linalg.norm(ref[need:])) <= 1e-5 * np.linalg.norm(ref)
    assert np.linalg.norm(Bh @ Bh.T - np.diag(sg)) <= 1e-4 * np.sqrt(need)
