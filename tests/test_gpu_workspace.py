"""What a call finds in its workspace does not matter, and the K-norm computed beside a sweep has the bits of the
stand-alone one (``-m gpu``).

The filter and the key projection are not preceded by a memset: their kernels clear what they need themselves, so a workspace full of
anything must give the results and the status of a fresh one, also right behind a call of another size in the same memory.
"""
import pytest
import torch

from paper_2601_17818_b200 import binding as vb

pytestmark = pytest.mark.gpu

DEV = "cuda"


def _randn(seed, *shape):
    return torch.randn(shape, generator=torch.Generator(device=DEV).manual_seed(seed), device=DEV)


def _filter(feat, n_centers, ws):
    B, n, _ = feat.shape
    o = [torch.zeros((B, n), dtype=t, device=DEV) for t in (torch.int32, torch.float32, torch.float32, torch.int32)]
    vb.vitcop_redundancy_filter(feat, None, o[0], torch.zeros(B, dtype=torch.int32, device=DEV), ws, n_centers=n_centers, rho=o[1],
                                delta2=o[2], parent=o[3])
    return vb.vitcop_poll_status(ws), o


# units of 64, 128 and 256 columns; the diagonal, the density sweep and the search (fewer and more diagonal tiles than SMs)
@pytest.mark.parametrize("B,n,D", [(1, 65, 64), (1, 576, 128), (3, 600, 1024), (12, 576, 64), (6, 1700, 256), (80, 300, 128)])
@pytest.mark.parametrize("fill", [0x00, 0x01, 0x3F, 0xFF])
def test_filter_whatever_the_workspace_holds(B, n, D, fill):
    feat = _randn(n, B, n, D).to(torch.bfloat16)
    clean = torch.zeros(vb.vitcop_workspace_bytes(vb.OP_FILTER, B=B, Nv=n, D=D), dtype=torch.uint8, device=DEV)
    status, ref = _filter(feat, n // 20 + 1, clean)
    assert status == vb.OK
    ws = torch.full_like(clean, fill)
    for _ in range(2):                                     # the second call finds what the first one left
        status, got = _filter(feat, n // 20 + 1, ws)
        assert status == vb.OK and all(torch.equal(a, b) for a, b in zip(got, ref))
    m = n // 2 + 1                                         # a smaller problem's words lie elsewhere in the same memory
    half = feat[:1, :m].contiguous()
    status, small = _filter(half, m // 20 + 1, ws)
    ref_small = _filter(half, m // 20 + 1, torch.zeros_like(clean))[1]
    assert status == vb.OK and all(torch.equal(a, b) for a, b in zip(small, ref_small))


# pairs of CTAs and CTAs apart; with and without a score to compute
@pytest.mark.parametrize("N", [10300, 700])
@pytest.mark.parametrize("fill", [0x01, 0xFF])
def test_kproj_whatever_the_workspace_holds(N, fill):
    H, d, Dh = 4, 128, 256
    hidden, W = _randn(1, 1, N, Dh).to(torch.bfloat16), _randn(2, H * d, Dh).to(torch.bfloat16)
    out = []
    for value, scored in ((0, True), (fill, True), (fill, False)):
        ws = torch.full((vb.vitcop_workspace_bytes(vb.OP_KPROJ, B=1, H=H, N=N, d=d),), value, dtype=torch.uint8, device=DEV)
        K = torch.zeros((1, H, N, d), dtype=torch.bfloat16, device=DEV)
        score = torch.zeros((1, N - 64), dtype=torch.float32, device=DEV) if scored else None
        vb.vitcop_kproj_knorm(hidden, W, H, d, K, ws, vis_start=64, score=score)
        assert vb.vitcop_poll_status(ws) == vb.OK
        out.append((K, score))
    assert torch.equal(out[0][0].view(torch.int16), out[1][0].view(torch.int16)) and torch.equal(out[0][1], out[1][1])
    assert torch.equal(out[0][0].view(torch.int16), out[2][0].view(torch.int16))


# Chunks of eight tokens, eight or sixteen lanes a token, boxes that reach past the sequence; head counts that fill the buffers
# once, twice and three times; row lengths that the sweep leaves to the stand-alone kernel (96, 512).
@pytest.mark.parametrize("H,d", [(1, 64), (5, 64), (32, 128), (3, 128), (40, 136), (17, 256), (48, 256), (6, 96), (2, 512)])
@pytest.mark.parametrize("B,n,T", [(1, 1, 1), (2, 9, 0), (3, 129, 9), (1, 577, 3), (16, 200, 2)])
def test_norms_beside_the_sweep_are_the_stand_alone_ones(B, n, T, H, d):
    _compare_norms(B, n, T, H, d, 64)


def _compare_norms(B, n, T, H, d, D):
    N, budget, nc = n + T, max(1, n // 2), max(1, n // 20)
    feat = _randn(n, B, n, D).to(torch.bfloat16)
    K = (_randn(d, B, H, N, d) * torch.exp(0.5 * _randn(H, B, 1, N, 1))).to(torch.bfloat16)
    vis_start = T // 2
    ref = torch.zeros((B, n), dtype=torch.float32, device=DEV)
    vb.vitcop_knorm_score(K, vis_start, n, ref)
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)
    score, cap = torch.zeros_like(ref), T + budget
    hidden, hidden_out = torch.zeros((B, N, 8), dtype=torch.bfloat16, device=DEV), torch.zeros((B, cap, 8), dtype=torch.bfloat16, device=DEV)
    K_out, V_out = (torch.zeros((B, H, cap, d), dtype=torch.bfloat16, device=DEV) for _ in range(2))
    ws = vb.alloc_workspace(vb.OP_COLLAB_STEP, B=B, Nv=n, D=D)
    vb.vitcop_collaborative_step(feat, None, hidden, K, K, vis_start, budget, hidden_out, K_out, V_out, i32(B), i32(B, n), i32(B), ws,
                                 n_centers=nc, score_out=score)
    torch.cuda.synchronize()
    assert torch.equal(score, ref)


# Beside the density sweep: all of the samples or, where the sweep is over before, the first ones of them; units of four and eight
# tokens that end inside a copy, heads that end inside one.
@pytest.mark.parametrize("B,n,T,H,d,D", [(8, 2881, 3, 31, 128, 1024), (9, 2879, 0, 62, 64, 1024), (20, 1501, 1, 32, 128, 1024),
                                         (4, 4606, 2, 33, 128, 1024)])
def test_norms_beside_the_density_sweep_are_the_stand_alone_ones(B, n, T, H, d, D):
    _compare_norms(B, n, T, H, d, D)
