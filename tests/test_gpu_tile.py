"""Layers of few rows, whose chain runs as two products by tiles, against float64: edges of the 64- and 128-row tiles, of
the 64-column pieces and of the range by rows, factors narrower than a piece, with and without the saved intermediate."""
import pytest
import torch

from paper_2405_01067_b200 import binding as ab

pytestmark = pytest.mark.gpu


def _bf16(*shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda").to(torch.bfloat16)


def _close(got, want, terms):
    """want: float64; terms: sum of the absolute products.  One bf16 rounding of the result, one bf16 step of each operand
    that was itself rounded (the intermediate may fall on the other side of a tie), fp32 sums."""
    bound = 2.0 ** -8 * (want.abs() + terms) + 1e-30
    assert bool(((got.double() - want).abs() <= bound).all())


@pytest.mark.parametrize("rows,m,n,r", [(1, 64, 768, 8), (63, 520, 72, 24), (65, 3072, 768, 192), (197, 768, 3072, 192),
                                        (129, 1000, 776, 120), (2049, 328, 2304, 256), (9472, 264, 392, 64), (9473, 264, 392, 64),
                                        (12672, 64, 3072, 16), (63, 1032, 1000, 24)])
@pytest.mark.parametrize("save", [True, False])
def test_few_rows_layer(rows, m, n, r, save):
    x, A, B, dY = _bf16(rows, n, seed=1), _bf16(m, r, seed=2), _bf16(r, n, seed=3), _bf16(rows, m, seed=4)
    xd, Ad, Bd, dYd = (t.double() for t in (x, A, B, dY))
    y, T = ab.ab_layer_forward(x, A, B, save_T=save)
    Td = (xd @ Bd.T).to(torch.bfloat16).double()
    if save:
        _close(T, xd @ Bd.T, 2.0 ** -8 * (xd.abs() @ Bd.abs().T))
    _close(y, Td @ Ad.T, Td.abs() @ Ad.abs().T)
    dX, dA, dB = ab.ab_layer_backward(x, dY, A, B, T_saved=T)
    dTd = (dYd @ Ad).to(torch.bfloat16).double()
    _close(dX, dTd @ Bd, dTd.abs() @ Bd.abs())
    # fp32 sums of exact bf16 products.  A bound on each element that grows with the rows would not see a lost row; the relative
    # Frobenius error does: one row of 12672 is worth 9e-3.  dA from the T that was used: sums alone, under sqrt(rows) 2^-23 =
    # 1.4e-5.  dT is not returned: of its values about 1 in 1000 is rounded to the other side, by 2^-8 at most: 1.3e-4.
    used = ab.ab_layer_forward(x, A, B, save_T=True)[1].double()
    for got, want, bound in ((dA, dYd.T @ used, 2e-5), (dB, dTd.T @ xd, 2e-4)):
        assert float((got.double() - want).norm() / want.norm()) <= bound
    # the same bits whichever results are wanted, and with the intermediate saved or not
    only = ab.ab_layer_backward(x, dY, A, B, T_saved=T, want=("dX",))[0]
    assert torch.equal(only, dX)
    assert torch.equal(ab.ab_layer_forward(x, A, B, save_T=not save)[0], y)
    # a workspace of the status word alone has no room for the intermediate: the fused kernel
    small, _ = ab.ab_layer_forward(x, A, B, ws=ab.workspace(256, "cuda"))
    _close(small, Td @ Ad.T, Td.abs() @ Ad.abs().T)
