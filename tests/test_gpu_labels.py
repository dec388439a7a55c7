"""Centres, labels and the selection behind them, at the sizes where their kernels change form (``-m gpu``).

Up to 2048 tokens whose scores a sweep has left, labels and cluster-quota selection are one kernel; beyond 8192 tokens eight CTAs share the labels
of a sample and follow long parent chains together.  The references are the oracle's selection on the GPU's own scores and labels, and
Algorithm 2, steps 3-4, on the GPU's own densities, distances and parents: no tolerance in either.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_17818_b200 import binding as vb
from gpu_helpers import gpu_filter

pytestmark = pytest.mark.gpu

DEV = "cuda"


def _bits(x):
    return vb.bf16_bits(torch.from_numpy(np.ascontiguousarray(x, dtype=np.float32)).to(DEV).to(torch.bfloat16))


def _step(n, budget, n_centers, same, B, H=2, d=64, D=64):
    """One-call step on keys whose norms tie often; `same`: share of the tokens that are copies of token 0 (one large cluster)."""
    g = torch.Generator(device=DEV).manual_seed(n)
    feat = torch.randn((B, n, D), generator=g, device=DEV)
    feat[:, : int(same * n)] = feat[:, :1]
    K = (torch.rand((B, H, n, d), generator=g, device=DEV) < 0.02).to(torch.bfloat16)
    hid = torch.zeros((B, n, 8), dtype=torch.bfloat16, device=DEV)
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)
    cap = max(1, min(budget, n))
    label, ncl, olen, kidx, nk = i32(B, n), i32(B), i32(B), i32(B, n), i32(B)
    score = torch.zeros((B, n), dtype=torch.float32, device=DEV)
    ws = vb.alloc_workspace(vb.OP_COLLAB_STEP, B=B, Nv=n, D=D)
    vb.vitcop_kernel_timing_begin()
    vb.vitcop_collaborative_step(feat.to(torch.bfloat16), None, hid, K, K, 0, budget, torch.zeros((B, cap, 8), dtype=torch.bfloat16, device=DEV),
                                 torch.zeros((B, H, cap, d), dtype=torch.bfloat16, device=DEV),
                                 torch.zeros((B, H, cap, d), dtype=torch.bfloat16, device=DEV), olen, label, ncl, ws, n_centers=n_centers,
                                 score_out=score, keep_idx_out=kidx, n_keep_out=nk)
    kernels = vb.vitcop_kernel_timing_end()
    return vb.vitcop_poll_status(ws), kernels, score.cpu().numpy(), label.cpu().numpy(), kidx.cpu().numpy(), nk.cpu().numpy()


@pytest.mark.parametrize("same", [0.0, 0.6])
@pytest.mark.parametrize("n", [1, 2, 9, 24, 1023, 1024, 1025, 2047, 2048])
def test_selection_right_behind_the_labels(n, same):
    n_centers, B = n // 20 + 1, 2 if n <= 1025 else 1      # (the sweep takes all norms)
    for budget in (n_centers, n // 3 + n_centers, n + n_centers, 2 * n + 7):
        status, kernels, score, label, kidx, nk = _step(n, budget, n_centers, same, B)
        assert status == vb.OK and "select_quota_kernel" not in kernels
        for b in range(B):
            want, _, _ = oracle.select_quota(score[b].astype(np.float64), label[b], budget)
            assert nk[b] == len(want) and np.array_equal(kidx[b, : nk[b]], want), (budget, b)
    if n_centers > 1:
        status, _, _, _, _, nk = _step(n, n_centers - 1, n_centers, same, B)
        assert status == vb.ERR_BUDGET and not nk.any()


def _labels(r, b, n_centers, feat):
    """Algorithm 2, steps 3-4, on what the GPU found; returns labels and the longest chain."""
    rho, d2, par = r.rho[b], r.delta2[b], r.parent[b].astype(np.int64)
    n = len(rho)
    gamma = np.where(par < 0, np.float32(np.inf), rho * np.sqrt(np.where(par < 0, 0, d2).astype(np.float32)))
    centre = np.zeros(n, bool)
    centre[np.lexsort((np.arange(n), -rho, -gamma))[:n_centers]] = True
    nxt = np.where(centre | (par < 0), np.arange(n), par)
    depth, at = 0, nxt
    while True:
        to = nxt[at]
        if np.array_equal(to, at):
            break
        at, depth = to, depth + 1
    surplus = np.flatnonzero((nxt == np.arange(n)) & ~centre)
    if len(surplus):
        c = np.flatnonzero(centre)
        f = torch.from_numpy(feat.astype(np.float64))
        f /= f.norm(dim=1, keepdim=True)
        nxt = np.arange(n)
        nxt[surplus] = c[torch.argmax(f[surplus] @ f[c].T, 1).numpy()]
        at = nxt[at]
    return at, depth


# The tokens left in the cut's bin are ranked on as many lanes each as there are for all of them, four to 32.  The densest token has no
# parent, so the first histogram is a coarse one, and tokens that are much alike all fall into one bin.
@pytest.mark.parametrize("n", [2, 31, 32, 33, 34, 64, 65, 66, 127, 129, 130, 200, 255, 256, 257, 300])
def test_centres_among_few_candidates(n):
    feat = torch.randn((2, n, 64), generator=torch.Generator(device=DEV).manual_seed(n), device=DEV).to(torch.bfloat16)
    for n_centers in {1, n // 2, n - 1}:
        r = gpu_filter(vb.bf16_bits(feat), None, 0, 0.5, -1.0, n_centers)
        for b in range(2):
            assert r.status == vb.OK and np.array_equal(r.label[b], _labels(r, b, n_centers, None)[0])


# every token an orphan (radius zero): all but the centres join the nearest one; a few centres, many, all of them
@pytest.mark.parametrize("n,n_centers", [(8193, 3), (8200, 411), (16384, 820), (8193, 8193)])
@pytest.mark.parametrize("tau", [-1.0, 0.0])
def test_labels_of_long_samples(n, n_centers, tau):
    rng = np.random.default_rng(n)
    bits = _bits(rng.standard_normal((1, n, 64)))
    pos = np.stack([np.arange(n) / n, np.zeros(n)], -1)[None].astype(np.float32)
    r = gpu_filter(bits, pos, 0, 0.5, tau, n_centers)
    assert r.status == vb.OK and r.n_clusters[0] == n_centers
    feat = (bits[0].astype(np.uint32) << 16).view(np.float32)
    assert np.array_equal(r.label[0], _labels(r, 0, n_centers, feat)[0])


def test_long_chains_of_parents():
    """Tokens along a curve whose density falls towards its ends: each one's nearest denser token is its neighbour, so chains are
    hundreds of tokens long."""
    n = 9000
    walk = np.cumsum(np.random.default_rng(1).standard_normal((n, 64)), 0)
    bits = _bits(walk[None])
    r = gpu_filter(bits, None, 1, 400.0, -1.0, 2)
    want, depth = _labels(r, 0, 2, None)
    assert r.status == vb.OK and depth > 256
    assert np.array_equal(r.label[0], want)


# More samples than the device runs clusters of eight for have one CTA each, with sixteen tokens a thread; and a few samples on clusters.
# Ordinary parents, and every token an orphan; single calls (clusters) have the same labels.
@pytest.mark.parametrize("B,n,n_centers", [(20, 8200, 411), (40, 8193, 3), (2, 9001, 450), (3, 16384, 819)])
@pytest.mark.parametrize("tau", [-1.0, 0.0])
def test_labels_of_many_long_samples(B, n, n_centers, tau):
    rng = np.random.default_rng(B)
    bits = _bits(rng.standard_normal((B, n, 64), dtype=np.float32))
    pos = np.repeat(np.stack([np.arange(n) / n, np.zeros(n)], -1)[None].astype(np.float32), B, 0)
    r = gpu_filter(bits, pos, 0, 0.5, tau, n_centers)
    assert r.status == vb.OK and (r.n_clusters == n_centers).all()
    for b in {0, B // 2, B - 1}:
        feat = (bits[b].astype(np.uint32) << 16).view(np.float32)
        assert np.array_equal(r.label[b], _labels(r, b, n_centers, feat)[0])
        one = gpu_filter(bits[b: b + 1], pos[b: b + 1], 0, 0.5, tau, n_centers)
        assert np.array_equal(one.rho[0], r.rho[b]) and np.array_equal(one.parent[0], r.parent[b]) and np.array_equal(one.label[0], r.label[b])
