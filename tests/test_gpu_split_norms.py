"""sigma of tall splits whose long side is a few rows, so that most CTAs of the cluster that forms the norms have nothing to load and
pass their sums on at once: the same bits in a hundred calls, and float64's values.

Tolerance: the rows are unit vectors in fp32 and Y is rounded to fp32, a few 2^-24 of the largest value in each column, and the fp32
Gram matrix turns vectors by 2^-24 sqrt(s) / gap but moves W v's norm only by the square of that: 2e-6 of the largest value."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,r", [(1, 1, 1), (2, 1, 1), (7, 5, 5), (8, 8, 4), (9, 3, 2), (33, 32, 32), (40, 33, 33), (63, 17, 9), (64, 64, 64),
                                   (65, 40, 35)])
def test_short_columns(m, n, r):
    from paper_2405_01067_b200 import binding as ab
    rng = np.random.default_rng(100 * m + n)
    q, p = np.linalg.qr(rng.standard_normal((m, n)))[0], np.linalg.qr(rng.standard_normal((n, n)))[0]
    ref = np.linspace(1.0, 0.5, n)
    W = torch.from_numpy(((q * ref) @ p.T).astype(np.float32)).cuda()
    runs = [ab.ab_svd_split(W, r, 0.0)[2] for _ in range(100)]
    torch.cuda.synchronize()
    sigma = torch.stack(runs).cpu().numpy()
    assert np.all(sigma == sigma[0])
    assert np.all(np.abs(sigma[0].astype(np.float64) - ref[:r]) <= 2e-6)
