"""The Householder reduction of the direct eigensolver, read back from the workspace of a split: every reflector I - gamma v v^T is
orthogonal as far as fp64 goes, for spectra whose columns cancel in each step (a flat floor) and for those that seldom do.

Bound: gamma v.v = 2 holds but for the rounding of the sum of squares (up to 10 terms a lane, eight levels of partial sums), of the root
and of the four operations behind it, each 2^-53 of the result: 24 of them, on a value of 2."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# words of a problem's record in the workspace: X, (gram, s), need, rows, vals, flag, xbuf, refl, tmat, zp, zm, d, e, gam, ...
REFL, GAM = 7, 13


def record(ws, s):
    words = ws[:ws.numel() // 8 * 8].view(torch.int64)
    at = (words == ws.data_ptr()).nonzero().flatten().tolist()       # X lies first in the workspace
    found = [words[i:i + 18].tolist() for i in at if i + 18 <= words.numel() and words[i + 1].item() == s << 32]
    assert len(found) == 1
    return found[0]


def doubles(ws, address, count):
    at = address - ws.data_ptr()
    return ws[at:at + 8 * count].view(torch.float64).cpu().numpy()


@pytest.mark.parametrize("kind", ["noise", "flat", "linear"])
@pytest.mark.parametrize("s,r", [(5, 5), (64, 20), (100, 30), (192, 48), (256, 64), (300, 20), (520, 20), (800, 20), (1100, 20)])
def test_reflectors_orthogonal(s, r, kind):
    from paper_2405_01067_b200 import binding as ab
    rng = np.random.default_rng(s)
    m = s + 3
    if kind == "noise":
        W = rng.standard_normal((m, s))
    else:
        values = np.linspace(1.0, 0.2, s) if kind == "linear" else np.where(np.arange(s) < s // 8, 1.0, 0.3)
        W = (np.linalg.qr(rng.standard_normal((m, s)))[0] * values) @ np.linalg.qr(rng.standard_normal((s, s)))[0].T
    ws = ab.workspace(ab.ab_workspace_bytes(ab.AB_OP_SVD_SPLIT, 0, m, s, r, 1, ab.AB_F32), "cuda")
    ab.ab_svd_split(torch.from_numpy(W.astype(np.float32)).cuda(), r, 0.0, ws=ws)
    torch.cuda.synchronize()
    job, ld = record(ws, s), (s + 1) // 2 * 2
    v = doubles(ws, job[REFL], s * ld).reshape(s, ld).astype(np.longdouble)
    gam = doubles(ws, job[GAM], s).astype(np.longdouble)
    live = gam > 0
    assert live.sum() >= s - 3
    assert np.max(np.abs(gam * (v * v).sum(1) - 2)[live]) <= 24 * 2 * 2.0 ** -53
