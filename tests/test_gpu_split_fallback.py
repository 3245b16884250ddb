"""What follows the direct eigensolver of the splits: its report of a wait that ran out, and the Jacobi fallback.

Both are set by the self-test entry: no input is known that makes the solver flag its vectors, and no wait is made to run out.
"""
import numpy as np
import pytest
import torch

from paper_2405_01067_b200 import binding as ab
from paper_2405_01067_b200 import synth

pytestmark = pytest.mark.gpu


def _matrices(count, m, n):
    rng = np.random.default_rng(m + n)
    s = min(m, n)
    return np.stack([synth.planted_matrix(rng, m, n, np.linspace(1.0, 0.3, s) * (1.0 + i)) for i in range(count)]).astype(np.float32)


@pytest.mark.parametrize("s,count,covered", [(64, 3, 3), (256, 2, 2), (300, 14, 12), (768, 3, 3)])
@pytest.mark.parametrize("flagged", [0, 1, 4])
def test_a_wait_that_ran_out_reaches_every_matrix_of_its_call(s, count, covered, flagged):
    """The solver takes all matrices of a short side up to 256 in one call, larger ones twelve at a time."""
    W = torch.from_numpy(_matrices(count, s + 10, s)).cuda()
    status = ab.ab_selftest_split_fallback(W, s // 4, flagged, ab.AB_ERR_TIMEOUT)[4]
    assert status.tolist() == [ab.AB_ERR_TIMEOUT] * covered + [0] * (count - covered)


@pytest.mark.parametrize("s,tall,count,flagged", [(31, True, 3, 0b101), (192, False, 3, 0b010), (256, True, 2, 0b11), (257, True, 1, 0b1),
                                                  (257, False, 3, 0b110), (500, True, 13, 0b1000000000010), (768, True, 3, 0b001),
                                                  (768, False, 1, 0b1), (1184, True, 3, 0b010)])
def test_fallback_of_flagged_matrices(s, tall, count, flagged):
    """Flagged matrices against float64 at the bounds of the library (values 1e-4, product 1e-4 of the norm); the others keep
    the direct solver's bits."""
    W = _matrices(count, s + 40, s) if tall else np.ascontiguousarray(_matrices(count, s + 40, s).transpose(0, 2, 1))
    t, k = torch.from_numpy(W).cuda(), max(1, s // 2)
    plain = ab.ab_selftest_split_fallback(t, k, 0)
    got = ab.ab_selftest_split_fallback(t, k, flagged)
    assert got[4].tolist() == [0] * count and got[3].tolist() == [k] * count
    for i in range(count):
        if not flagged >> i & 1:
            assert all(torch.equal(a[i], b[i]) for a, b in zip(got, plain))
            continue
        assert not torch.equal(got[0][i], plain[0][i]) or not torch.equal(got[1][i], plain[1][i])      # it did go another way
        ref = np.linalg.svd(W[i].astype(np.float64), compute_uv=False)
        A, B, sigma = (x[i].cpu().numpy().astype(np.float64) for x in got[:3])
        assert np.all(np.abs(np.sort(sigma)[::-1] - ref[:k]) <= 1e-4 * ref[:k])
        assert abs(np.linalg.norm(W[i] - A @ B) - np.linalg.norm(ref[k:])) <= 1e-4 * np.linalg.norm(ref)
        for f in (A.T @ A, B @ B.T):
            assert np.linalg.norm(f - np.diag(sigma)) <= 1e-4 * ref[0] * np.sqrt(k)
