"""What is launched behind a backward call that leaves dB out: it may read dX and overwrite the workspace at once, so no
kernel of the call may be running any more.  Compared bit for bit with the full backward, whose dB job waits by itself."""
import pytest
import torch

from paper_2405_01067_b200 import binding as ab

pytestmark = pytest.mark.gpu


# the chain as two products by tiles (one slice of the gradients; several) and as one fused kernel (blocks of two and one)
@pytest.mark.parametrize("rows,m,n,r", [(60, 768, 3072, 192), (2049, 3072, 768, 192), (9472, 3072, 768, 192), (12608, 1000, 776, 120),
                                        (50432, 768, 1536, 64)])
def test_consumer_of_dx_without_db(rows, m, n, r):
    g = torch.Generator(device="cuda").manual_seed(rows)
    x, A, B, dY = (torch.randn(s, generator=g, device="cuda").to(torch.bfloat16) for s in ((rows, n), (m, r), (r, n), (rows, m)))
    _, T = ab.ab_layer_forward(x, A, B, save_T=True)
    dX, dA, _ = ab.ab_layer_backward(x, dY, A, B, T_saved=T)
    want = ab.ab_layer_forward(dX, A, B)[0]
    torch.cuda.synchronize()
    ws = ab.workspace(ab.ab_workspace_bytes(ab.AB_OP_LAYER_BACKWARD, rows, m, n, r, 1, ab.AB_BF16), "cuda")
    got, gotA, y = torch.empty_like(dX), torch.empty_like(dA), torch.empty_like(want)
    for _ in range(10):
        got.fill_(float("nan"))
        ab.ab_layer_backward(x, dY, A, B, T_saved=T, want=("dX", "dA"), dX=got, dA=gotA, ws=ws)
        ab.ab_layer_forward(got, A, B, y=y, ws=ws)
        torch.cuda.synchronize()
        assert torch.equal(got, dX) and torch.equal(gotA, dA) and torch.equal(y, want)
