"""The fp32-accurate tensor-core product behind ab_recombine and the group sync, at the edges of its tiles.

Tolerance: the operands carry 24 bits, products are exact, sums are fp32 over K <= 300 terms plus two accumulators:
2^-24 (1 + sqrt(K)) stays under 1.1e-6; 1e-6 is the library's stated bound and what is held (rms errors add up to far less).
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


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("m,n,r", [(1, 1, 1), (128, 128, 64), (129, 65, 63), (127, 64, 65), (257, 191, 16), (64, 300, 130), (5, 1000, 192),
                                   (1000, 6, 128), (2000, 1600, 40), (1920, 2440, 300), (700, 516, 17)])
def test_recombine_tile_edges(ab, m, n, r, bf16):
    rng = np.random.default_rng(m + 3 * n + 7 * r)
    a, b = rng.standard_normal((m, r)).astype(np.float32), rng.standard_normal((r, n)).astype(np.float32)
    A, B = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    if bf16:
        A, B = A.bfloat16(), B.bfloat16()
        a, b = A.float().cpu().numpy(), B.float().cpu().numpy()
    W = torch.full((m, n), float("nan"), device="cuda")
    ws = ab.workspace(ab.ab_workspace_bytes(ab.AB_OP_RECOMBINE, 0, m, n, r, 1, ab.AB_BF16 if bf16 else ab.AB_F32), "cuda")
    ab.ab_recombine(A, B, W=W, ws=ws)
    again = ab.ab_recombine(A, B, ws=ws)
    torch.cuda.synchronize()
    assert ab.workspace_status(ws) == 0
    assert orc.rel_frob(W.cpu().numpy().astype(np.float64), orc.recombine(a, b)) <= 1e-6
    assert torch.equal(W, again)


def test_recombine_strided_and_misaligned_factors(ab):
    """Row strides and bases that rule out 16-byte loads."""
    rng = np.random.default_rng(5)
    m, n, r = 200, 150, 70
    big_a, big_b = torch.from_numpy(rng.standard_normal((m, r + 3)).astype(np.float32)).cuda(), \
        torch.from_numpy(rng.standard_normal((r, n + 5)).astype(np.float32)).cuda()
    W = torch.empty((m, n), device="cuda")
    ws = ab.workspace(256, "cuda")
    st = ab.lib().ab_recombine(big_a.data_ptr() + 4, big_b.data_ptr() + 8, W.data_ptr(), m, n, r, r + 3, n + 5, ab.AB_F32,
                               ws.data_ptr(), ws.numel(), None)
    assert st == 0
    torch.cuda.synchronize()
    ref = orc.recombine(big_a[:, 1:1 + r].cpu().numpy(), big_b[:, 2:2 + n].cpu().numpy())
    assert orc.rel_frob(W.cpu().numpy().astype(np.float64), ref) <= 1e-6


@pytest.mark.parametrize("m,n,r", [(512, 4608, 64), (200, 2000, 20), (2900, 130, 36)])
def test_lone_layer_gram_slices(ab, m, n, r):
    """A lone matrix: its Gram products are cut into many slices of the long index, none of them empty."""
    a, b = synth.planted_factors(np.random.default_rng(n), m, n, np.linspace(1.0, 0.3, r))
    plan = ab.SyncPlan([torch.from_numpy(a[None].copy()).cuda()], [torch.from_numpy(b[None].copy()).cuda()], 0.1)
    _, _, sigma, r_out, status = ab.ab_group_sync(plan, path=ab.AB_SYNC_FACTORED)
    torch.cuda.synchronize()
    ref = np.linalg.svd(a.astype(np.float64) @ b.astype(np.float64), compute_uv=False)[:r]
    assert int(status[0].item()) == 0 and int(r_out[0].item()) == r
    assert np.max(np.abs(sigma[0].cpu().numpy() - ref) / ref) <= 1e-5      # well conditioned: a few 2^-24 sqrt(n)


@pytest.mark.parametrize("m,n,r", [(1920, 2440, 296), (1921, 2440, 312), (3000, 1992, 200), (300, 20000, 128), (2560, 1024, 2000)])
@pytest.mark.parametrize("shift", [0, 1])
def test_large_bf16_recombine(m, n, r, shift, ab):
    """bf16 factors of many tiles: loaded by TMA where rows and bases allow it, else (shift) through the converters."""
    g = torch.Generator(device="cuda").manual_seed(m + r)
    big_a, big_b = (torch.randn(s, generator=g, device="cuda").bfloat16() for s in ((m * r + 8,), (r * n + 8,)))
    A, B = big_a[shift:shift + m * r].view(m, r), big_b[shift:shift + r * n].view(r, n)
    W = torch.full((m, n), float("nan"), device="cuda")
    ws = ab.workspace(256, "cuda")
    ws[:4] = 255
    ab.ab_recombine(A, B, W=W, ws=ws)
    want = A.double() @ B.double()
    assert ab.workspace_status(ws) == 0
    # products are exact, fp32 sums of up to 2000: sqrt(2000) 2^-24 = 2.7e-6 at worst
    assert float((W.double() - want).norm() / want.norm()) <= 2.7e-6


def test_a_kernel_in_front_may_take_longer_than_a_wait(ab):
    """The waits inside the product are bounded by a second; a kernel in front of it that takes a second (the self-test of
    the chain's waits) and lets it start early is not its own time."""
    rng = np.random.default_rng(9)
    a, b = rng.standard_normal((300, 64)).astype(np.float32), rng.standard_normal((64, 200)).astype(np.float32)
    A, B, W = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), torch.empty((300, 200), device="cuda")
    stall = ab.workspace(int(ab.lib().ab_selftest_chain_stall_workspace_bytes()), "cuda")
    ws = ab.workspace(256, "cuda")
    stream = torch.cuda.current_stream().cuda_stream
    torch.cuda.synchronize()
    assert ab.lib().ab_selftest_chain_stall(stall.data_ptr(), stall.numel(), 1_000_000, stream) == 0
    ab.ab_recombine(A, B, W=W, ws=ws)
    torch.cuda.synchronize()
    assert ab.workspace_status(stall) == ab.AB_ERR_TIMEOUT and ab.workspace_status(ws) == 0
    assert orc.rel_frob(W.cpu().numpy().astype(np.float64), orc.recombine(a, b)) <= 1e-6


def test_records_of_many_tiles(ab):
    """A batch whose CTAs take dozens of tiles each: the tile records go round their ring many times.  Every copy of a
    matrix gives the bits of its first one, in every run."""
    shapes = [(40, 24, 8), (130, 60, 12), (64, 200, 16), (24, 24, 4), (150, 150, 20)]
    rng = np.random.default_rng(2)
    kinds = [synth.planted_factors(rng, m, n, np.linspace(1.0, 0.3, r)) for m, n, r in shapes]
    kinds = [(torch.from_numpy(a[None].copy()).cuda(), torch.from_numpy(b[None].copy()).cuda()) for a, b in kinds]
    order = rng.integers(0, len(kinds), 2500)
    plan = ab.SyncPlan([kinds[k][0] for k in order], [kinds[k][1] for k in order], 0.1, want_W=True)
    for _ in range(3):
        ab.ab_group_sync(plan, path=ab.AB_SYNC_FACTORED)
    torch.cuda.synchronize()
    assert torch.count_nonzero(plan.status) == 0
    for k in range(len(kinds)):
        mine = np.flatnonzero(order == k)
        for out in (plan.A_out, plan.B_out, plan.sigma, plan.W_out):
            assert bool((torch.stack([out[i] for i in mine]) == out[mine[0]]).all())
        W = kinds[k][0][0].double() @ kinds[k][1][0].double()
        got = plan.A_out[mine[0]].double() @ plan.B_out[mine[0]].double()
        assert float((got - W).norm() / W.norm()) <= 1e-5
