"""Calls of different sizes from several host threads at once, each on a stream of its own: none may fail, and each
gives the bits it gives alone.  (A kernel's limit of dynamic shared memory is one for all threads.)"""
import threading

import pytest
import torch

from paper_2405_01067_b200 import binding as ab

pytestmark = pytest.mark.gpu


def _normal(*shape, seed, dtype):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda").to(dtype)


def _layer(dtype, rows, m, n, r):
    x, dY, A, B = (_normal(*s, seed=i, dtype=dtype) for i, s in enumerate([(rows, n), (rows, m), (m, r), (r, n)]))
    dt = ab.AB_BF16 if dtype == torch.bfloat16 else ab.AB_F32
    ws_f, ws_b = (ab.workspace(ab.ab_workspace_bytes(op, rows, m, n, r, 1, dt), "cuda") for op in (ab.AB_OP_LAYER_FORWARD, ab.AB_OP_LAYER_BACKWARD))
    y, T = torch.empty((rows, m), dtype=dtype, device="cuda"), torch.empty((rows, r), dtype=dtype, device="cuda")
    dX, dA, dB = torch.empty_like(x), torch.empty((m, r), device="cuda"), torch.empty((r, n), device="cuda")

    def call(stream):
        ab.ab_layer_forward(x, A, B, y=y, T_save=T, ws=ws_f, stream=stream)
        ab.ab_layer_backward(x, dY, A, B, T_saved=T, dX=dX, dA=dA, dB=dB, ws=ws_b, stream=stream)
        return y, dX, dA, dB
    return call


def _sync(r):
    plan = ab.SyncPlan([_normal(2, 300, r, seed=r, dtype=torch.float32)], [_normal(2, r, 260, seed=r + 1, dtype=torch.float32)], 0.1)

    def call(stream):
        ab.ab_group_sync(plan, stream=stream)
        return plan.A_out[0], plan.B_out[0], plan.sigma[0]
    return call


@pytest.mark.parametrize("kind", ["few_rows", "fused", "fp32", "sync"])
def test_threads_with_calls_of_their_own(kind):
    bf, f = torch.bfloat16, torch.float32
    calls = {"few_rows": lambda: [_layer(bf, 200, 256, 256, 16), _layer(bf, 200, 768, 512, 256), _layer(bf, 90, 512, 768, 64)],
             "fused": lambda: [_layer(bf, 300, 64, 64, 8), _layer(bf, 1000, 256, 256, 32), _layer(bf, 20000, 256, 256, 128)],
             "fp32": lambda: [_layer(f, 2000, 1024, 900, 8), _layer(f, 2300, 400, 500, 8), _layer(f, 2300, 1024, 64, 16)],
             "sync": lambda: [_sync(r) for r in (16, 120, 228)]}[kind]()
    torch.cuda.synchronize()
    alone = []
    for c in calls:
        out = c(torch.cuda.current_stream())
        torch.cuda.synchronize()
        alone.append([t.clone() for t in out])
    failed = []

    def work(i):
        try:
            torch.cuda.set_device(0)
            stream = torch.cuda.Stream()
            for _ in range(400 if kind != "sync" else 60):
                out = calls[i](stream)
            stream.synchronize()
            if not all(torch.equal(a, b) for a, b in zip(out, alone[i])):
                failed.append((i, "other bits"))
        except Exception as e:
            failed.append((i, repr(e)))
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
