"""fp32 layers and products on both sides of every line between their kernels, against float64.

Tolerance: the small kernels and the 64 x 64 kernel add 16 products in fp32 and those sums in fp64 (2.4e-7 relative, see
test_gpu_layer_small.py); the register-tiled kernel of the large products adds all of them in fp32, sqrt(K) 2^-24 for K <= 1100 there:
2e-6, and a layer's two products with the rounding of T between them 4e-6.
"""
import pytest
import torch

from paper_2405_01067_b200 import binding as ab

pytestmark = pytest.mark.gpu


def _normal(*shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda")


def _rel(got, want):
    return float((got.double() - want).norm() / want.norm())


# rows at the ends of one, two and four turns of 16 rows a CTA; ranks and widths that are on either side
@pytest.mark.parametrize("N,m,n,r", [(296, 256, 256, 64), (297, 256, 256, 64), (592, 130, 256, 64), (593, 256, 130, 128), (1184, 200, 512, 32),
                                     (1185, 64, 260, 32), (2368, 256, 100, 16), (2369, 256, 300, 16), (4736, 1024, 64, 1), (4737, 48, 1030, 8),
                                     (9472, 1030, 40, 8), (9473, 40, 1024, 8), (50432, 16, 16, 1), (20000, 64, 64, 16)])
def test_layer_either_side_of_the_lines(N, m, n, r):
    x, dY, A, B = _normal(N, n, seed=1), _normal(N, m, seed=2), _normal(m, r, seed=3), _normal(r, n, seed=4)
    xd, dYd, Ad, Bd = (t.double() for t in (x, dY, A, B))
    y, T = ab.ab_layer_forward(x, A, B, save_T=True)
    Td, dTd = xd @ Bd.T, dYd @ Ad
    want = {"T": Td, "y": Td @ Ad.T, "dX": dTd @ Bd, "dA": dYd.T @ Td, "dB": dTd.T @ xd}
    ws = ab.workspace(ab.ab_workspace_bytes(ab.AB_OP_LAYER_BACKWARD, N, m, n, r, 1, ab.AB_F32), "cuda")
    ws[:4] = 255
    dX, dA, dB = ab.ab_layer_backward(x, dY, A, B, T_saved=T, ws=ws)
    assert ab.workspace_status(ws) == 0
    for k, got in dict(T=T, y=y, dX=dX, dA=dA, dB=dB).items():
        assert _rel(got, want[k]) <= 4e-6, k
    again = ab.ab_layer_backward(x, dY, A, B)                     # T taken from x again: the forward's bits
    assert all(torch.equal(a, b) for a, b in zip(again, (dX, dA, dB)))


@pytest.mark.parametrize("M,N,K", [(4672, 64, 96), (4673, 64, 96), (4673, 64, 95), (512, 290, 64), (600, 520, 64), (1184, 512, 63),
                                   (1200, 960, 100), (1216, 1024, 1100), (64, 18944, 70), (1, 1, 1),
                                   (704, 832, 16384), (704, 833, 16391)])
def test_single_products(M, N, K):
    """x W^T, dY W and dY^T x of the dense layer: every order of the operands."""
    x, W = _normal(M, K, seed=5), _normal(N, K, seed=6)
    assert _rel(ab.ab_dense_forward(x, W), x.double() @ W.double().T) <= 2e-6
    dY, V = _normal(M, K, seed=7), _normal(K, N, seed=8)
    dX = ab.ab_dense_backward(torch.empty((M, N), device="cuda"), dY, V, want=("dX",))[0]
    assert _rel(dX, dY.double() @ V.double()) <= 2e-6
    xt, dYt = _normal(K, N, seed=9), _normal(K, M, seed=10)
    dW = ab.ab_dense_backward(xt, dYt, torch.empty((M, N), device="cuda"), want=("dW",))[1]
    assert _rel(dW, dYt.double().T @ xt.double()) <= 2e-6
