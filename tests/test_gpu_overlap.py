"""Calls queued one behind the other without a synchronisation, against the same calls waited for (``-m gpu``).

Kernel timing takes programmatic launches away, so tests that ask for the kernels' names see a call in plain stream order.  Here nothing is
timed: a copy that selects has moved rows in front of and behind the span before the scores are there, its lengths are what the
call before has just written, and labels and selection follow a sweep that is still running.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_17818_b200 import binding as vb

pytestmark = pytest.mark.gpu

DEV = "cuda"
TIMES = 5


def _randn(seed, *shape):
    return torch.randn(shape, generator=torch.Generator(device=DEV).manual_seed(seed), device=DEV).to(torch.bfloat16)


def _i32(*s):
    return torch.full(s, -7, dtype=torch.int32, device=DEV)


def _zeros(*s, dtype=torch.bfloat16):
    return torch.zeros(s, dtype=dtype, device=DEV)


def _outputs(B, H, cap, d, Dh, n):
    return dict(hid=_zeros(B, cap, Dh), K=_zeros(B, H, cap, d), V=_zeros(B, H, cap, d), olen=_i32(B), pos=_i32(B, cap), nk=_i32(B),
                keep=_i32(B, n), score=_zeros(B, n, dtype=torch.float32))


def _same(a, b):
    return torch.equal(a.view(torch.int32 if a.element_size() == 4 else torch.int16), b.view(torch.int32 if b.element_size() == 4 else torch.int16))


# The projection of the keys, a pruning step on lengths of its own for every sample, and another one on what that left: rows, lengths and
# kept counts, with text behind the span; then the projection for the next pass into the same keys.
@pytest.mark.parametrize("B,H,d,Dh", [(3, 4, 128, 256), (2, 2, 64, 64)])
@pytest.mark.parametrize("n", [1, 31, 33, 64, 128, 129, 255, 256])
def test_pruning_steps_behind_one_another(n, B, H, d, Dh):
    T, tail, first, second = 5, 9, max(1, 2 * n // 3), max(1, n // 3)
    N, cap1, cap2 = T + n + tail, T + first + tail, T + second + tail
    W = _randn(1, H * d, Dh)
    hidden = [_randn(10 + i, B, N, Dh) for i in range(TIMES)]
    lens = [torch.tensor([max(0, n - 3 * b - i) for b in range(B)], dtype=torch.int32, device=DEV) for i in range(TIMES)]
    seqs = [(x + T + tail - i % 3).to(torch.int32) for i, x in enumerate(lens)]

    def run(wait, apart):
        sync = torch.cuda.synchronize if wait else (lambda: None)
        K, out = _zeros(B, H, N, d), []
        ws = [vb.alloc_workspace(vb.OP_KPROJ, B=B, H=H, N=N, d=d), vb.alloc_workspace(vb.OP_PRUNE_STEP, B=B, Nv=n),
              vb.alloc_workspace(vb.OP_SELECT, B=B, Nv=n)]
        steps = [(_outputs(B, H, cap1, d, Dh, n), _outputs(B, H, cap2, d, Dh, first)) for _ in range(TIMES)]
        torch.cuda.synchronize()

        def step(hid, k, v, vis, seq, cap_v, budget, o):
            if apart:
                vb.vitcop_knorm_score(k, T, vis, o["score"])
                sync()
                vb.vitcop_select(o["score"], vis, budget, o["keep"], o["nk"], ws[2])
                sync()
                vb.vitcop_compact_kv(hid, k, v, T, vis, o["keep"], o["nk"], o["hid"], o["K"], o["V"], o["olen"], kept_pos=o["pos"], seq_len=seq)
            else:
                vb.vitcop_prune_step(hid, k, v, T, vis, cap_v, budget, o["hid"], o["K"], o["V"], o["olen"], ws[1], kept_pos=o["pos"],
                                     seq_len=seq, score_out=o["score"], keep_idx_out=o["keep"], n_keep_out=o["nk"])
            sync()

        for i, (a, b) in enumerate(steps):
            vb.vitcop_kproj_knorm(hidden[i], W, H, d, K, ws[0])
            sync()
            step(hidden[i], K, K, lens[i], seqs[i], n, first, a)
            step(a["hid"], a["K"], a["V"], a["nk"], a["olen"], first, second, b)
        torch.cuda.synchronize()
        return steps

    queued, waited, apart = run(False, False), run(True, False), run(True, True)
    for i in range(TIMES):
        for s in range(2):
            for k, x in queued[i][s].items():
                assert _same(x, waited[i][s][k]) and _same(x, apart[i][s][k]), (i, s, k)


# Labels and selection in one kernel right behind the sweep, and the copy behind both; keys that the projection has just written.
@pytest.mark.parametrize("n", [1, 2, 24, 129, 576, 1023, 1025, 2048])
def test_selection_behind_the_labels_while_the_sweep_runs(n):
    B, H, d, Dh, D, T = 2 if n <= 1025 else 1, 2, 64, 64, 64, 3
    N, n_centers = T + n, n // 20 + 1
    budget = n_centers + n // 3
    cap = T + min(budget, n)
    W = _randn(1, H * d, Dh)
    hidden, feat = [_randn(10 + i, B, N, Dh) for i in range(TIMES)], [_randn(30 + i, B, n, D) for i in range(TIMES)]
    K = _zeros(B, H, N, d)
    wk, ws = vb.alloc_workspace(vb.OP_KPROJ, B=B, H=H, N=N, d=d), vb.alloc_workspace(vb.OP_COLLAB_STEP, B=B, Nv=n, D=D)
    out = [dict(_outputs(B, H, cap, d, Dh, n), label=_i32(B, n), ncl=_i32(B), keys=_zeros(B, H, N, d)) for _ in range(TIMES)]
    torch.cuda.synchronize()
    for h, f, o in zip(hidden, feat, out):
        vb.vitcop_kproj_knorm(h, W, H, d, K, wk)
        vb.vitcop_collaborative_step(f, None, h, K, K, T, budget, o["hid"], o["K"], o["V"], o["olen"], o["label"], o["ncl"], ws,
                                     n_centers=n_centers, kept_pos=o["pos"], score_out=o["score"], keep_idx_out=o["keep"], n_keep_out=o["nk"])
        o["keys"].copy_(K)
    assert vb.vitcop_poll_status(ws) == vb.OK
    for h, o in zip(hidden, out):
        score = torch.empty_like(o["score"])
        vb.vitcop_knorm_score(o["keys"], T, n, score)
        assert _same(score, o["score"])
        for b in range(B):
            want, _, _ = oracle.select_quota(score[b].cpu().numpy().astype(np.float64), o["label"][b].cpu().numpy(), budget)
            assert int(o["nk"][b]) == len(want) and np.array_equal(o["keep"][b, : len(want)].cpu().numpy(), want)
            rows = torch.cat([torch.arange(T), T + torch.from_numpy(np.asarray(want, dtype=np.int64))]).to(DEV)
            L = len(rows)
            assert int(o["olen"][b]) == L and torch.equal(o["pos"][b, :L].long(), rows) and bool((o["pos"][b, L:] == -1).all())
            assert _same(o["hid"][b, :L].contiguous(), h[b, rows]) and _same(o["K"][b, :, :L].contiguous(), o["keys"][b][:, rows])
