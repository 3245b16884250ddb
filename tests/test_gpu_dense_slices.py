"""dW of the dense layer where its rows are cut into one, a few and many slices, against float64 and with dX left out."""
import pytest
import torch

from paper_2405_01067_b200 import binding as ab

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,m,n", [(63, 64, 8), (2049, 136, 264), (4097, 1000, 72), (20011, 64, 72), (50432, 128, 256)])
def test_dense_slices(rows, m, n):
    g = torch.Generator(device="cuda").manual_seed(rows)
    x, dY, W = (torch.randn(s, generator=g, device="cuda").to(torch.bfloat16) for s in ((rows, n), (rows, m), (m, n)))
    dX, dW = ab.ab_dense_backward(x, dY, W)
    ref = dY.double().T @ x.double()
    # products are exact, sums in fp32: roundings of 2^-24 of a partial sum, which add up like the square root of their number.  A
    # slab of 64 rows that got lost would change values by 8, of 50432 rows the bound is 0.5.
    assert bool(((dW.double() - ref).abs() <= rows ** 0.5 * 2.0 ** -24 * (dY.double().abs().T @ x.double().abs())).all())
    refX = dY.double() @ W.double()
    assert bool(((dX.double() - refX).abs() <= 2.0 ** -8 * refX.abs() + m * 2.0 ** -23 * (dY.double().abs() @ W.double().abs())).all())
    assert torch.equal(ab.ab_dense_backward(x, dY, W, want=("dW",))[1], dW)
