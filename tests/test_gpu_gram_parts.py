"""Gram matrix and long product of a dense split with the reduction in parts: odd short sides (tables and partial sums behind an odd
number of floats), long sides that leave a short last part or fill none, either side long.

Tolerance: 16 products at a time are summed in fp32 and those sums in fp64, one rounding to fp32 at the end, so sigma is as good
as an fp32 Gram matrix lets it be: 2^-24 sqrt(s) sigma_1^2 / sigma, below 1e-4 for the values above 0.2 sigma_1 that are compared; the
residual as in test_gpu_eig.py.

Whether a product goes in parts is its size's matter (test_gpu_gram_route.py has the line of the Gram matrix): test_route_and_values says
for each shape which of its two products does and counts the launches, test_gram_in_parts has shapes on both sides.
"""
import numpy as np
import pytest
import torch

from paper_2405_01067_b200 import synth
from test_gpu_gram_route import launches

pytestmark = pytest.mark.gpu


def check(W, A, B, sigma, k):
    ref = np.linalg.svd(W.astype(np.float64), compute_uv=False)
    sg = sigma.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(sg - ref[:k]) <= 1e-4 * ref[:k])
    res = np.linalg.norm(W - A.double().cpu().numpy() @ B.double().cpu().numpy())
    assert abs(res - np.linalg.norm(ref[k:])) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("m,n,k", [(2713, 192, 40), (2476, 201, 150), (201, 2600, 33), (1664, 257, 64), (385, 769, 300), (769, 385, 8),
                                   (3072, 768, 192), (1000, 999, 100)])
def test_gram_in_parts(m, n, k):
    from paper_2405_01067_b200 import binding as ab
    W = synth.planted_matrix(np.random.default_rng(m + n), m, n, np.linspace(1.0, 0.2, min(m, n)))
    A, B, sigma, r_out, status = ab.ab_svd_split(torch.from_numpy(W).cuda(), k, 0.0)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and int(r_out.item()) == k
    check(W, A, B, sigma, k)


def test_gram_in_parts_of_a_batch():
    from paper_2405_01067_b200 import binding as ab
    m, n, count = 1700, 257, 4
    W = np.stack([synth.planted_matrix(np.random.default_rng(i), m, n, np.linspace(1.0 + i, 0.3 + i, n)) for i in range(count)])
    A, B, sigma, r_out, status = ab.ab_selftest_split_fallback(torch.from_numpy(W).cuda(), 60, 0)
    torch.cuda.synchronize()
    assert status.tolist() == [0] * count and r_out.tolist() == [60] * count
    for i in range(count):
        check(W[i], A[i], B[i], sigma[i], 60)


def parts_launched(call):
    names = launches(call)
    return tuple(sum(kernel in name for name in names) for kernel in ("gemm_parts_kernel", "sum_gram_kernel", "sum_parts_kernel"))


# wide and tall with odd sides; ranks that are multiples of no tile; a last part of the long side shorter than the others; one, two
# and three parts of the long product; a rank at which it has no room; the whole rank
@pytest.mark.parametrize("m,n,k,gram,long", [(449, 2101, 440, 1, 0), (2101, 449, 440, 1, 0), (385, 2701, 16, 1, 0), (601, 1501, 520, 1, 1),
                                             (1501, 601, 520, 1, 1), (1025, 1100, 700, 1, 1), (1100, 1025, 1025, 1, 1), (3072, 768, 192, 1, 1)])
def test_route_and_values(m, n, k, gram, long):
    from paper_2405_01067_b200 import binding as ab
    W = synth.planted_matrix(np.random.default_rng(m + n), m, n, np.linspace(1.0, 0.2, min(m, n)))
    Wd = torch.from_numpy(W).cuda()
    A, B, sigma, r_out, status = ab.ab_svd_split(Wd, k, 0.0)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and int(r_out.item()) == k
    check(W, A, B, sigma, k)
    assert parts_launched(lambda: ab.ab_svd_split(Wd, k, 0.0)) == (gram + long, gram, long)


def test_both_products_of_a_batch():
    from paper_2405_01067_b200 import binding as ab
    m, n, k, count = 1501, 601, 520, 3
    W = np.stack([synth.planted_matrix(np.random.default_rng(i), m, n, np.linspace(1.0 + i, 0.3 + i, n)) for i in range(count)])
    Wd = torch.from_numpy(W).cuda()
    A, B, sigma, r_out, status = ab.ab_selftest_split_fallback(Wd, k, 0)
    torch.cuda.synchronize()
    assert status.tolist() == [0] * count and r_out.tolist() == [k] * count
    for i in range(count):
        check(W[i], A[i], B[i], sigma[i], k)
    assert parts_launched(lambda: ab.ab_selftest_split_fallback(Wd, k, 0)) == (2 * count, count, count)
