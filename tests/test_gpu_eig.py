"""The direct eigensolver behind the splits, at the orders where its kernels change or end a tile, on spectra
that are easy, graded, clustered, decoupled and rank deficient.

Tolerance: the split works on the fp32 Gram matrix G (entries rounded to 2^-24), whose eigenvalues are therefore
known to 2^-24 sqrt(s) of the largest at worst; a singular value sigma moves by that times sigma_1^2 / (2 sigma).
Values above 0.1 sigma_1 are held to 1e-4 (the library's bound; the estimate gives 5e-6 at s = 256), the residual
of the truncated product to the discarded values (Eckart-Young) within 1e-5 of the norm.
"""
import numpy as np
import pytest
import torch

from paper_2405_01067_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ab():
    from paper_2405_01067_b200 import binding
    binding.lib()
    return binding


def spectrum(kind, s):
    if kind == "random":
        return np.linspace(1.0, 0.2, s)
    if kind == "clustered":                 # groups of equal values: vectors determined only up to rotation
        return np.repeat([1.0, 0.7, 0.4, 0.4, 0.2], (s + 4) // 5)[:s]
    if kind == "equal":                     # an orthogonal matrix, e.g. a freshly initialised layer
        return np.ones(s)
    return np.where(np.arange(s) < max(1, s // 3), np.linspace(1.0, 0.3, s), 0.0)     # low rank


@pytest.mark.parametrize("kind", ["random", "clustered", "equal", "low_rank", "zero_columns", "diagonal"])
@pytest.mark.parametrize("s", [1, 2, 3, 31, 32, 33, 64, 65, 97, 128, 129, 160, 192, 193, 225, 256,
                               257, 512, 513, 765, 768, 769, 1024, 1025, 1184])
def test_split_by_order_and_spectrum(ab, s, kind):
    rng = np.random.default_rng(1000 * s + len(kind))
    m, n = s + 40, s
    if kind == "diagonal":                  # decouples completely: every off-diagonal of T is zero
        W = np.zeros((m, n), dtype=np.float32)
        W[np.arange(s), np.arange(s)] = np.linspace(0.2, 1.0, s)
    elif kind == "zero_columns":            # what a factor truncated by an earlier rank rule looks like
        W = synth.planted_matrix(rng, m, n, np.linspace(1.0, 0.3, s))
        W[:, n - n // 2:] = 0.0
    else:
        W = synth.planted_matrix(rng, m, n, spectrum(kind, s))
    k = max(1, (3 * s) // 4)
    t = torch.from_numpy(W).cuda()
    A, B, sigma, r_out, status = ab.ab_svd_split(t, k, 0.0)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and int(r_out.item()) == k
    ref = np.linalg.svd(W.astype(np.float64), compute_uv=False)
    sg = sigma.cpu().numpy().astype(np.float64)
    big = ref[:k] >= 0.1 * ref[0]
    assert np.all(np.abs(sg - ref[:k])[big] <= 1e-4 * ref[:k][big])
    assert np.all(sg[~big] <= 1e-5 * ref[0])
    Ah, Bh = A.cpu().numpy().astype(np.float64), B.cpu().numpy().astype(np.float64)
    norm = np.linalg.norm(ref)
    res = np.linalg.norm(W - Ah @ Bh)
    assert abs(res - np.linalg.norm(ref[k:])) <= 1e-5 * norm
    live = sg > 1e-4 * ref[0]
    assert np.linalg.norm((Ah.T @ Ah - np.diag(sg))[np.ix_(live, live)]) <= 1e-4 * ref[0] * np.sqrt(k)
    assert np.linalg.norm((Bh @ Bh.T - np.diag(sg))[np.ix_(live, live)]) <= 1e-4 * ref[0] * np.sqrt(k)


@pytest.mark.parametrize("count", [1, 40])
@pytest.mark.parametrize("r", [4, 36, 64, 100, 148, 192, 228])
def test_factored_sync_by_rank_and_batch(ab, r, count):
    """The core of the factored sync (Gram form, fp64) for a lone matrix and for a batch, with a zero tail in the
    factors of every second matrix."""
    m, n = r + 60, r + 28
    rng = np.random.default_rng(r)
    As, Bs = [], []
    for i in range(min(count, 2)):
        a, b = synth.planted_factors(rng, m, n, np.linspace(1.0, 0.2, r))
        if i:
            a[:, r - r // 3:] = 0.0
            b[r - r // 3:] = 0.0
        As.append(a[None].copy())
        Bs.append(b[None].copy())
    dA, dB = [torch.from_numpy(a).cuda() for a in As], [torch.from_numpy(b).cuda() for b in Bs]
    plan = ab.SyncPlan([dA[i % len(dA)] for i in range(count)], [dB[i % len(dB)] for i in range(count)], 0.1)
    A_out, B_out, sigma, r_out, status = ab.ab_group_sync(plan, path=ab.AB_SYNC_FACTORED)
    torch.cuda.synchronize()
    assert torch.count_nonzero(status) == 0
    for i in range(count):
        W = As[i % len(As)][0].astype(np.float64) @ Bs[i % len(Bs)][0].astype(np.float64)
        ref = np.linalg.svd(W, compute_uv=False)
        keep = int(np.sum(ref[:r] >= 0.1 * ref[0]))
        assert int(r_out[i].item()) == keep
        sg = sigma[i].cpu().numpy().astype(np.float64)
        assert np.all(np.abs(sg[:keep] - ref[:keep]) <= 1e-4 * ref[:keep])
        prod = A_out[i].cpu().numpy().astype(np.float64) @ B_out[i].cpu().numpy().astype(np.float64)
        assert np.linalg.norm(prod - W) <= 1e-4 * np.linalg.norm(W)
