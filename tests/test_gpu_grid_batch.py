"""Several matrices of one order above 256 in one call: the reduction over the device gives each group of CTAs its matrices in turn,
with the barriers and buffers of the one before.  Bounds as in test_gpu_eig.py."""
import numpy as np
import pytest
import torch

from paper_2405_01067_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s,count", [(257, 7), (300, 13), (520, 3), (769, 2)])
def test_batches_of_large_orders(s, count):
    from paper_2405_01067_b200 import binding as ab
    rng = np.random.default_rng(s)
    m, n, r = s + 24, s, 32
    As, Bs = [], []
    for i in range(count):
        a, b = synth.planted_factors(rng, m, n, np.linspace(1.0 + i, 0.3, r))
        As.append(torch.from_numpy(a[None].copy()).cuda())
        Bs.append(torch.from_numpy(b[None].copy()).cuda())
    plan = ab.SyncPlan(As, Bs, 0.046)         # no value of these spectra lies within 2e-3 of it
    A_out, B_out, sigma, r_out, status = ab.ab_group_sync(plan, path=ab.AB_SYNC_DENSE)
    torch.cuda.synchronize()
    assert torch.count_nonzero(status) == 0
    for i in range(count):
        W = As[i][0].double().cpu().numpy() @ Bs[i][0].double().cpu().numpy()
        ref = np.linalg.svd(W, compute_uv=False)
        keep = int(r_out[i].item())
        assert keep == int(np.sum(ref[:r] >= 0.046 * ref[0]))
        sg = sigma[i].cpu().numpy().astype(np.float64)
        assert np.all(np.abs(sg[:keep] - ref[:keep]) <= 1e-4 * ref[:keep])
        prod = A_out[i].double().cpu().numpy() @ B_out[i].double().cpu().numpy()
        assert abs(np.linalg.norm(prod - W) - np.linalg.norm(ref[keep:])) <= 1e-4 * np.linalg.norm(W)
