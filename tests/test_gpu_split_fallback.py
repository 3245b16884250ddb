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
