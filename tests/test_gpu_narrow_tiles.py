"""Products of few tiles run on tiles 32 columns wide: widths around a tile, one row to one more than a row of tiles, ranks around a
16-step of the MMA and a slab of 64, the largest that take them on 148 SMs (116 tiles; 148 of fp32
factors above rank 64) and the next ones (64 columns wide).

Tolerance: fp32 operands as three bf16 pieces lose three products of order 2^-24; the fp32 accumulator rounds once in 16 of the
reduction (r <= 320: 20 roundings of 2^-23, of either sign): below 1e-6 of the 2-norm.  bf16 operands lose only the latter.
"""
import numpy as np
import pytest
import torch

from oracle import ab_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("m,n,r", [(1, 1, 1), (128, 32, 16), (129, 33, 17), (127, 31, 15), (64, 40, 63), (256, 95, 64), (200, 97, 65), (768, 768, 192),
                                   (72, 72, 72), (512, 928, 40), (512, 929, 40), (512, 1184, 66), (512, 1185, 66), (4736, 116, 128), (300, 1000, 320), (3072, 192, 33)])
def test_recombine_of_few_tiles(m, n, r, bf16):
    from paper_2405_01067_b200 import binding as ab
    g = torch.Generator().manual_seed(m * 7 + n * 3 + r)
    td = torch.bfloat16 if bf16 else torch.float32
    A, B = torch.randn((m, r), generator=g).to(td), torch.randn((r, n), generator=g).to(td)
    W = torch.full((m + 1, n), 7.0, device="cuda")             # the row behind stays as it is
    ab.ab_recombine(A.cuda(), B.cuda(), W=W[:m])
    torch.cuda.synchronize()
    assert orc.rel_frob(W[:m].double().cpu().numpy(), orc.recombine(A.float().numpy(), B.float().numpy())) <= 1e-6
    assert torch.all(W[m] == 7.0)


@pytest.mark.parametrize("da,db", [(1, 0), (0, 1), (3, 5)])
def test_strided_factors_of_few_tiles(da, db):
    """Row strides and bases that rule out 16-byte loads."""
    from paper_2405_01067_b200 import binding as ab
    m, n, r = 140, 100, 70
    g = torch.Generator().manual_seed(5)
    a, b = torch.randn((m, r + da), generator=g).cuda(), torch.randn((r, n + db), generator=g).cuda()
    W, ws = torch.empty((m, n), device="cuda"), ab.workspace(256, "cuda")
    A, B = a[:, da:], b[:, db:]
    assert ab.lib().ab_recombine(A.data_ptr(), B.data_ptr(), W.data_ptr(), m, n, r, r + da, n + db, ab.AB_F32, ws.data_ptr(), ws.numel(), None) == 0
    torch.cuda.synchronize()
    assert ab.workspace_status(ws) == 0
    assert orc.rel_frob(W.double().cpu().numpy(), orc.recombine(A.cpu().numpy(), B.cpu().numpy())) <= 1e-6
