"""Which kernels a step launches where the better way changes with the sizes (``-m gpu``)."""
import pytest
import torch

from paper_2601_17818_b200 import binding as vb

pytestmark = pytest.mark.gpu

DEV = "cuda"


def _kernels(B, n, H, d, D=64, metric=0):
    g = torch.Generator(device=DEV).manual_seed(n)
    rand = lambda *s: torch.randn(s, generator=g, device=DEV).to(torch.bfloat16)
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)
    K, budget = rand(B, H, n, d), n // 4
    K_out, score = torch.zeros((B, H, budget, d), dtype=torch.bfloat16, device=DEV), torch.zeros((B, n), device=DEV)
    ws = vb.alloc_workspace(vb.OP_COLLAB_STEP, B=B, Nv=n, D=D)
    vb.vitcop_kernel_timing_begin()
    vb.vitcop_collaborative_step(rand(B, n, D), None, None, K, K, 0, budget, None, K_out, torch.zeros_like(K_out), i32(B), i32(B, n), i32(B), ws,
                                 metric=metric, d_c=0.5 if metric == 0 else 0.5 * D ** 0.5,
                                 n_centers=n // 20, score_out=score)
    kernels = vb.vitcop_kernel_timing_end()
    assert vb.vitcop_poll_status(ws) == vb.OK
    want = K.float().square().sum((1, 3)).sqrt()
    assert bool(((score - want).abs() <= 1e-5 * want).all())
    return kernels


# Norms in the one-kernel sweep or in a kernel of their own: few CTAs with many keys each against either side of that line (the
# batch that is large enough, shorter rows, more CTAs).
@pytest.mark.parametrize("B,n,H,d,apart", [(1, 182, 32, 128, True), (2, 192, 32, 128, True), (1, 256, 48, 128, True), (1, 192, 32, 64, True),
                                           (16, 182, 32, 128, False), (1, 182, 16, 128, False), (1, 300, 32, 128, False), (1, 576, 32, 128, False)])
def test_norms_of_short_samples(B, n, H, d, apart):
    kernels = _kernels(B, n, H, d)
    assert ("knorm_kernel" in kernels) == apart and ("select_quota_kernel" in kernels) == apart


# Norms in the density sweep or in a kernel of their own: with few features the sweep is slower by them than that kernel takes.
@pytest.mark.parametrize("B,n,H,d,D,metric,apart", [(1, 4581, 16, 64, 256, 0, False), (1, 4581, 16, 64, 256, 1, True), (19, 1517, 4, 64, 128, 0, True),
                                                    (19, 1517, 32, 64, 1024, 1, False)])
def test_norms_beside_the_density_sweep(B, n, H, d, D, metric, apart):
    kernels = _kernels(B, n, H, d, D, metric)
    assert "density_sweep_kernel" in kernels and ("knorm_kernel" in kernels) == apart
