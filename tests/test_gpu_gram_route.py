"""Which kernel forms the Gram matrix of a dense split: the one whose reduction goes in parts only where its CTAs are half as many as
the SMs (short side above 384 on 148), since three parts of a few tiles leave the device idle over a long side of any length."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def launches(call):
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    return [e.key for e in prof.key_averages() for _ in range(e.count)]


@pytest.mark.parametrize("m,n,parts", [(100000, 64, 0), (64, 100000, 0), (25000, 128, 0), (20000, 256, 0), (3000, 384, 0), (2700, 385, 1), (385, 2700, 1),
                                       (1000, 640, 1)])
def test_route(m, n, parts):
    from paper_2405_01067_b200 import binding as ab
    W = torch.randn((m, n), generator=torch.Generator(device="cuda").manual_seed(m + n), device="cuda")
    ab.ab_svd_split(W, 8, 0.0)
    names = launches(lambda: ab.ab_svd_split(W, 8, 0.0))
    assert any("tri_values_kernel" in k for k in names)          # the list is not empty
    assert sum("gemm_parts_kernel" in k for k in names) == parts
