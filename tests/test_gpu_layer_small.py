"""The fp32 layer's own kernels at the edges of their row blocks, tiles and splits, against the float64 checker.

Tolerance: sums of 16 products in fp32 and those sums in fp64: about sqrt(16) 2^-24 = 2.4e-7 relative for each of the two
products of a chain, and the rounding of T between them; 2e-6 leaves four times that.
"""
import numpy as np
import pytest
import torch

from oracle import ab_oracle as orc
from paper_2405_01067_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ab():
    from paper_2405_01067_b200 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("save_T", [False, True])
@pytest.mark.parametrize("N,m,n,r", [(1, 16, 16, 1), (3, 33, 31, 7), (149, 64, 512, 32), (300, 40, 1024, 33), (700, 96, 100, 96),
                                     (1100, 200, 64, 64), (2500, 65, 66, 65), (4096, 64, 96, 17), (64, 512, 300, 256), (20, 300, 290, 255)])
def test_small_layer(ab, N, m, n, r, save_T):
    d = synth.chain_case(N + m + r, m, n, r, N, bf16=False)
    x, dY, A, B = (torch.from_numpy(d[k]).cuda() for k in ("x", "dY", "A", "B"))
    y, T = ab.ab_layer_forward(x, A, B, save_T=save_T)
    got = dict(zip(("dX", "dA", "dB"), ab.ab_layer_backward(x, dY, A, B, T_saved=T)))
    again = ab.ab_layer_backward(x, dY, A, B, T_saved=T)
    only_a = ab.ab_layer_backward(x, dY, A, B, T_saved=T, want=("dA",))[1]
    only_b = ab.ab_layer_backward(x, dY, A, B, T_saved=T, want=("dB",))[2]
    torch.cuda.synchronize()
    T_ref, y_ref = orc.forward(d["x"], d["A"], d["B"])
    dX, dA, dB, _ = orc.backward(d["x"], d["dY"], d["A"], d["B"])
    got["y"] = y
    if save_T:
        got["T"] = T
    for k, ref in dict(y=y_ref, T=T_ref, dX=dX, dA=dA, dB=dB).items():
        if k in got:
            assert orc.rel_frob(got[k].cpu().numpy().astype(np.float64), ref) <= 2e-6, k
    assert all(torch.equal(a, got[k]) for k, a in zip(("dX", "dA", "dB"), again))        # fixed order
    assert torch.equal(only_a, got["dA"]) and torch.equal(only_b, got["dB"])
