"""Vectors of the direct eigensolver that are close to others: the matrix is flagged for the Jacobi route exactly when a pair of them is less
than orthogonal, whether few or many lie above one (they are compared one by one or a lane each), and what comes out is orthogonal.

Copies of one block that hang together by a coupling of 1e-12 have their eigenvalues in clusters of as many as there are copies, 1e-13 or
so apart, whose vectors cannot come out orthogonal to better than 1e-3; a flat spectrum's come out orthogonal enough.
"""
import numpy as np
import pytest
import torch

from test_gpu_reduction import doubles, record

pytestmark = pytest.mark.gpu

CLOSE, NULL, TOL = 1e-7, 1e-7, 4e-6             # the solver's lines, fractions of the norm
FLAG, ZP, LAM, INV = 5, 9, 14, 15               # words of a problem's record


def copies(block, count):
    s = block * count
    d = np.tile(np.linspace(1.0, 0.5, block), count)
    e = np.full(s - 1, 0.125)
    e[block - 1::block] = 1e-12                 # coupling of the copies: what holds the values of a cluster apart
    return np.diag(d) + np.diag(e, 1)


def flat(s):
    rng = np.random.default_rng(s)
    values = np.where(np.arange(s) < s // 8, np.linspace(1.0, 0.5, s), 0.3)
    return (np.linalg.qr(rng.standard_normal((s, s)))[0] * values) @ np.linalg.qr(rng.standard_normal((s, s)))[0].T


@pytest.mark.parametrize("kind,a,b", [("copies", 8, 2), ("copies", 8, 12), ("copies", 8, 13), ("copies", 8, 14), ("copies", 7, 32), ("copies", 6, 33),
                                      ("copies", 6, 34), ("copies", 4, 64), ("copies", 8, 45), ("flat", 48, 0), ("flat", 256, 0), ("flat", 400, 0)])
def test_flag(kind, a, b):
    from paper_2405_01067_b200 import binding as ab
    W = (copies(a, b) if kind == "copies" else flat(a)).astype(np.float32)
    s = W.shape[0]
    ws = ab.workspace(ab.ab_workspace_bytes(ab.AB_OP_SVD_SPLIT, 0, s, s, s, 1, ab.AB_F32), "cuda")
    A, B, sigma, r_out, status = ab.ab_svd_split(torch.from_numpy(W).cuda(), s, 0.0, ws=ws)
    torch.cuda.synchronize()
    assert int(status.item()) == 0 and int(r_out.item()) == s
    job = record(ws, s)
    lam, inv, zp = doubles(ws, job[LAM], s), doubles(ws, job[INV], s), doubles(ws, job[ZP], s * s).reshape(s, s)
    dots = np.abs((zp * inv).T @ (zp * inv))
    pairs = (np.abs(lam[:, None] - lam[None]) < CLOSE) & (np.minimum(lam[:, None], lam[None]) > NULL) & ~np.eye(s, dtype=bool)
    assert kind == "flat" or pairs.sum(0).max() == b - 1
    worst = dots[pairs].max()
    assert kind == "flat" or worst > 10 * TOL
    flag = ws[job[FLAG] - ws.data_ptr():][:4].view(torch.int32).item()
    if not 0.99 * TOL < worst < 1.01 * TOL:
        assert flag == (1 if worst > TOL else 0)
    sg, Bh = sigma.cpu().numpy().astype(np.float64), B.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(Bh @ Bh.T - np.diag(sg)) <= 1e-4 * np.sqrt(s)
