"""Calls captured into a CUDA graph and launched later on other inputs: the bits of the same calls made directly.  The host
tables of a call are gone by then."""
import pytest
import torch

from paper_2405_01067_b200 import binding as ab

pytestmark = pytest.mark.gpu


def _normal(*shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda")


def _replayed(call, inputs):
    """call() reads `inputs` (tensors) and returns tensors; captured on the first contents, replayed on the second."""
    call()                                         # loads kernels, creates the library's helper stream
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = call()
    junk = [bytes(range(256)) * 64 for _ in range(2000)]      # over whatever the call left on the heap
    for t in inputs:
        t.copy_(_normal(*t.shape, seed=t.numel()).to(t.dtype))
    graph.replay()
    torch.cuda.synchronize()
    got = [t.clone() for t in out]
    want = call()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, want)) and len(junk) == 2000


@pytest.mark.parametrize("m,n", [(300, 257), (400, 768), (768, 768), (1184, 1200), (500, 64), (100, 256), (1300, 1190)])
def test_split(m, n):
    W = _normal(m, n, seed=1)
    r = max(1, min(m, n) // 4)
    ws = ab.workspace(ab.ab_workspace_bytes(ab.AB_OP_SVD_SPLIT, 0, m, n, r, 1, ab.AB_F32), "cuda")
    _replayed(lambda: ab.ab_svd_split(W, r, 0.02, ws=ws), [W])


@pytest.mark.parametrize("path,want_W", [(ab.AB_SYNC_FACTORED, False), (ab.AB_SYNC_FACTORED, True), (ab.AB_SYNC_DENSE, True)])
def test_group_sync(path, want_W):
    A = [_normal(2, 300 + 8 * i, 40, seed=i) for i in range(24)]
    B = [_normal(2, 40, 260, seed=50 + i) for i in range(24)]
    plan = ab.SyncPlan(A, B, 0.1, want_W=want_W)

    def call():
        ab.ab_group_sync(plan, path=path)
        return plan.A_out + plan.B_out + plan.sigma + [plan.r_out, plan.status] + plan.W_out
    _replayed(call, A + B)


@pytest.mark.parametrize("dtype,rows", [(torch.bfloat16, 200), (torch.bfloat16, 20000), (torch.float32, 100), (torch.float32, 5000)])
def test_layer_dense_and_recombination(dtype, rows):
    m, n, r = 264, 200, 40
    x, dY, A, B, W = (_normal(*s, seed=i).to(dtype) for i, s in enumerate([(rows, n), (rows, m), (m, r), (r, n), (m, n)]))

    def call():
        y, T = ab.ab_layer_forward(x, A, B, save_T=True)
        return [y, T, *ab.ab_layer_backward(x, dY, A, B, T_saved=T), ab.ab_dense_forward(x, W), *ab.ab_dense_backward(x, dY, W),
                ab.ab_recombine(A, B)]
    _replayed(call, [x, dY, A, B, W])


def test_convolution():
    x, dY, A, B = (_normal(*s, seed=i).bfloat16() for i, s in enumerate([(9, 7, 7, 72), (9, 7, 7, 64), (64, 24), (24, 648)]))

    def call():
        y, T = ab.ab_conv3x3_forward(x, A, B, save_T=True)
        return [y, T, *ab.ab_conv3x3_backward(x, dY, A, B, T_saved=T)]
    _replayed(call, [x, dY, A, B])
