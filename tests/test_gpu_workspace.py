"""What a call finds in its workspace does not matter, and the K-norm computed beside a sweep has the bits of the
stand-alone one (``-m gpu``).

The filter and the key projection are not preceded by a memset: their kernels clear what they need themselves, so a workspace full of
anything must give the results and the status of a fresh one, also right behind a call of another size in the same memory.  Their first
kernels are launched ahead of time and wait on the device for what precedes them.
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


def _compare_norms(B, n, T, H, d, D, metric=0, spatial=False, ws=None):
    """Scores of the one-call step against the stand-alone K-norm; returns its labels and cluster counts, and the step itself."""
    N, budget, nc = n + T, max(1, n // 2), max(1, n // 20)
    feat = _randn(n, B, n, D).to(torch.bfloat16)
    pos = torch.rand((B, n, 2), generator=torch.Generator(device=DEV).manual_seed(n), device=DEV) if spatial else None
    K = (_randn(d, B, H, N, d) * torch.exp(0.5 * _randn(H, B, 1, N, 1))).to(torch.bfloat16)
    vis_start = T // 2
    ref = torch.zeros((B, n), dtype=torch.float32, device=DEV)
    vb.vitcop_knorm_score(K, vis_start, n, ref)
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)
    score, cap = torch.zeros_like(ref), T + budget
    hidden, hidden_out = torch.zeros((B, N, 8), dtype=torch.bfloat16, device=DEV), torch.zeros((B, cap, 8), dtype=torch.bfloat16, device=DEV)
    K_out, V_out = (torch.zeros((B, H, cap, d), dtype=torch.bfloat16, device=DEV) for _ in range(2))
    if ws is None:
        ws = vb.alloc_workspace(vb.OP_COLLAB_STEP, B=B, Nv=n, D=D)
    label, ncl, olen = i32(B, n), i32(B), i32(B)
    how = dict(metric=metric, d_c=0.5 if metric == 0 else 16.0, n_centers=nc)

    def step(ws=ws):
        vb.vitcop_collaborative_step(feat, pos, hidden, K, K, vis_start, budget, hidden_out, K_out, V_out, olen, label, ncl, ws,
                                     score_out=score, **how)
        return vb.vitcop_poll_status(ws)

    assert step() == vb.OK
    assert torch.equal(score, ref)
    got = label.clone(), ncl.clone()
    if D > 64:                                             # the sweep that has keys on the side is another one
        fws = vb.alloc_workspace(vb.OP_FILTER, B=B, Nv=n, D=D)
        vb.vitcop_redundancy_filter(feat, pos, label, ncl, fws, **how)
        assert vb.vitcop_poll_status(fws) == vb.OK and torch.equal(got[0], label) and torch.equal(got[1], ncl)
    return step, (K_out, V_out, olen, label, ncl, score)


def _kernels(step):
    vb.vitcop_kernel_timing_begin()
    assert step() == vb.OK
    return vb.vitcop_kernel_timing_end()


# Beside the density sweep: all of the samples or, where the sweep is over before, the first ones of them; units of four and eight
# tokens that end inside a copy, heads that end inside one (also before its first four).
@pytest.mark.parametrize("B,n,T,H,d,D,alone", [(8, 2881, 3, 31, 128, 1024, False), (9, 2879, 0, 62, 64, 1024, False),
                                               (20, 1501, 1, 32, 128, 1024, True), (4, 4606, 2, 33, 128, 1024, False),
                                               (340, 1000, 1, 1, 128, 256, False), (340, 1000, 1, 2, 64, 256, False),
                                               (115, 999, 2, 3, 128, 512, False)])
def test_norms_beside_the_density_sweep_are_the_stand_alone_ones(B, n, T, H, d, D, alone):
    step, _ = _compare_norms(B, n, T, H, d, D)
    names = _kernels(step)
    assert "density_sweep_kernel" in names and ("knorm_kernel" in names) == alone


# Keys of all samples beside a sweep, on either side of the lines: one and two row tiles, 24 chunks to a CTA, a single buffer; 8 MB.
@pytest.mark.parametrize("B,n,T,H,d,D,alone", [(1, 128, 1, 3, 128, 128, True), (1, 129, 1, 3, 128, 128, False),
                                               (147, 249, 2, 1, 64, 64, True), (147, 249, 0, 16, 64, 64, False),
                                               (32, 576, 3, 3, 256, 64, False), (8, 577, 0, 48, 256, 64, True),
                                               (7, 1921, 5, 32, 64, 768, False), (7, 1921, 0, 4, 64, 768, True)])
def test_norms_of_all_samples_beside_a_sweep(B, n, T, H, d, D, alone):
    step, _ = _compare_norms(B, n, T, H, d, D)
    assert ("knorm_kernel" in _kernels(step)) == alone


@pytest.mark.parametrize("metric,spatial", [(0, True), (1, False), (1, True)])
@pytest.mark.parametrize("B,n,T,H,d,D", [(8, 2881, 3, 31, 128, 512), (9, 2879, 0, 62, 64, 512)])
def test_norms_beside_the_density_sweep_with_either_metric(B, n, T, H, d, D, metric, spatial):
    _compare_norms(B, n, T, H, d, D, metric, spatial)


def test_norms_beside_the_density_sweep_of_a_group():
    """With the least workspace that is taken the samples go through one by one; the first sweep takes norms of others along."""
    B, n, T, H, d, D = 30, 5000, 4, 4, 128, 1024
    full = vb.alloc_workspace(vb.OP_COLLAB_STEP, B=B, Nv=n, D=D)
    step, _ = _compare_norms(B, n, T, H, d, D, ws=full)

    def taken(units):
        try:
            return step(full[:256 * units]) == vb.OK
        except RuntimeError:
            return False

    lo, hi = 1, full.numel() // 256                        # lo is refused
    assert not taken(lo)
    while hi - lo > 1:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if taken(mid) else (mid, hi)
    step, _ = _compare_norms(B, n, T, H, d, D, ws=full[:256 * hi])
    names = _kernels(step)
    assert names["density_sweep_kernel"][0] == B and names["knorm_kernel"][0] == 1


@pytest.mark.parametrize("metric", [0, 1])
@pytest.mark.parametrize("roles", [1, 2, 4])
def test_density_sweep_with_keys_reports_timeout_and_recovers(roles, metric):
    """A role of the sweep's pairs of CTAs gives up while copies of keys are in flight (8: the kernels on pairs alone)."""
    step, outputs = _compare_norms(8, 2881, 3, 31, 128, 512, metric)
    assert step() == vb.OK
    ref = [t.clone() for t in outputs]
    try:
        vb.vitcop_set_wait_limit(0, 8 * roles)
        assert step() == vb.ERR_TIMEOUT
    finally:
        vb.vitcop_set_wait_limit(0, 0)
    assert step() == vb.OK and all(torch.equal(a, b) for a, b in zip(outputs, ref))


# The first kernels of these calls are launched before what precedes them ends: keys that the projection has just written, without a
# synchronisation in between (one-kernel sweep; diagonal and density sweep).
@pytest.mark.parametrize("B,n", [(1, 576), (4, 1800)])
def test_step_right_behind_the_projection_of_its_keys(B, n):
    H, d, Dh, D, T, budget, times = 4, 128, 256, 256, 16, n // 3, 6
    N, cap = n + T, T + n // 3
    W = _randn(1, H * d, Dh).to(torch.bfloat16)
    hidden = [_randn(10 + i, B, N, Dh).to(torch.bfloat16) for i in range(times)]
    feat = [_randn(30 + i, B, n, D).to(torch.bfloat16) for i in range(times)]
    z = lambda *s, dt=torch.bfloat16: torch.zeros(s, dtype=dt, device=DEV)
    i32 = lambda *s: z(*s, dt=torch.int32)

    def run(wait):
        K, out = z(B, H, N, d), []
        wk, ws = vb.alloc_workspace(vb.OP_KPROJ, B=B, H=H, N=N, d=d), vb.alloc_workspace(vb.OP_COLLAB_STEP, B=B, Nv=n, D=D)
        wp = vb.alloc_workspace(vb.OP_PRUNE_STEP, B=B, Nv=n)
        for h, f in zip(hidden, feat):
            o = [z(B, cap, Dh), z(B, H, cap, d), z(B, H, cap, d), i32(B), i32(B, n), i32(B), z(B, n, dt=torch.float32)]
            q = [z(B, cap, Dh), z(B, H, cap, d), z(B, H, cap, d), i32(B), z(B, n, dt=torch.float32)]
            mid = z(B, n, dt=torch.float32)
            vb.vitcop_kproj_knorm(h, W, H, d, K, wk, vis_start=5, score=mid)
            if wait:
                torch.cuda.synchronize()
            vb.vitcop_collaborative_step(f, None, h, K, K, 5, budget, *o[:6], ws, n_centers=n // 20, score_out=o[6])
            if wait:
                torch.cuda.synchronize()
            vb.vitcop_kproj_knorm(o[0][:, :1].expand(B, N, Dh).contiguous(), W, H, d, K, wk, vis_start=5, score=mid)
            if wait:
                torch.cuda.synchronize()
            vb.vitcop_prune_step(h, K, K, 5, n, n, budget, *q[:4], wp, score_out=q[4])
            if wait:
                torch.cuda.synchronize()
            out += o + q
        torch.cuda.synchronize()
        return out

    assert all(torch.equal(a, b) for a, b in zip(run(False), run(True)))
