"""Selection inside the copy (small ``vitcop_prune_step`` calls without labels) against the three separate calls (``-m gpu``).

The separate K-norm, selection and copy have kernels of their own, which other tests check against the oracle; every output has to have
their bits: rows, lengths, kept positions, scores and the kept list.
"""
import pytest
import torch

from paper_2601_17818_b200 import binding as vb

pytestmark = pytest.mark.gpu

DEV = "cuda"


def _step(B, n, T, tail, budget, H, d, Dh, ties, lengths=False, V=True, spare=3):
    g = torch.Generator(device=DEV).manual_seed(97 * n + budget)
    N = T + n + tail
    rand = lambda *s: torch.randn(s, generator=g, device=DEV).to(torch.bfloat16)
    K, Vt, hid = rand(B, H, N, d), rand(B, H, N, d) if V else None, rand(B, N, Dh) if Dh else None
    if ties:                                               # few different norms
        K = (torch.randint(0, 3, (B, 1, N, 1), generator=g, device=DEV).float() * torch.ones(1, H, 1, d, device=DEV)).to(torch.bfloat16)
    if ties and n > 2:
        K[:, 0, T + n // 2, 0] = float("nan")
    vis, seq = n, None
    if lengths:
        vis = torch.tensor([max(0, n - 5 * b) for b in range(B)], dtype=torch.int32, device=DEV)
        seq = torch.tensor([T + max(0, n - 5 * b) + max(0, tail - b) for b in range(B)], dtype=torch.int32, device=DEV)
    Ncap = T + min(budget, n) + tail + spare
    out = []
    for fused in (True, False):
        i32 = lambda *s: torch.full(s, -7, dtype=torch.int32, device=DEV)
        o = dict(K=torch.zeros((B, H, Ncap, d), dtype=torch.bfloat16, device=DEV), olen=i32(B), pos=i32(B, Ncap), keep=i32(B, n), nk=i32(B),
                 score=torch.zeros((B, n), device=DEV))
        o["V"] = torch.zeros_like(o["K"]) if V else None
        o["hid"] = torch.zeros((B, Ncap, Dh), dtype=torch.bfloat16, device=DEV) if Dh else None
        if fused:
            ws = vb.alloc_workspace(vb.OP_PRUNE_STEP, B=B, Nv=n)
            vb.vitcop_kernel_timing_begin()
            vb.vitcop_prune_step(hid, K, Vt, T, vis, n, budget, o["hid"], o["K"], o["V"], o["olen"], ws, kept_pos=o["pos"], seq_len=seq,
                                 score_out=o["score"], keep_idx_out=o["keep"], n_keep_out=o["nk"])
            kernels = vb.vitcop_kernel_timing_end()
        else:
            ws = vb.alloc_workspace(vb.OP_SELECT, B=B, Nv=n)
            vb.vitcop_knorm_score(K, T, vis, o["score"])
            vb.vitcop_select(o["score"], vis, budget, o["keep"], o["nk"], ws)
            vb.vitcop_compact_kv(hid, K, Vt, T, vis, o["keep"], o["nk"], o["hid"], o["K"], o["V"], o["olen"], kept_pos=o["pos"], seq_len=seq)
        assert vb.vitcop_poll_status(ws) == vb.OK
        out.append(o)
    for k, a in out[0].items():
        if a is not None:
            same = a.view(torch.int32) == out[1][k].view(torch.int32) if a.dtype == torch.float32 else a.view(torch.int16) == out[1][k].view(torch.int16)
            assert bool(same.all()), k
    return kernels


# 1, 32, 128 and 256 tokens and their neighbours; nothing, one, all and more than all of them kept
@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 127, 128, 129, 255, 256])
def test_selection_inside_the_copy(n, ties):
    for budget in sorted({0, 1, n // 2, n - 1, n, n + 9}):
        kernels = _step(2, n, 5, 7, budget, 2, 64, 512, ties)
        assert "select_plain_kernel" not in kernels and "compact_kernel" in kernels


# groups of 256, 128, 64 and 32 threads a row; the span at the front and at the end; lengths on the device; a tensor left out
@pytest.mark.parametrize("H,d,Dh,V", [(8, 128, 4096, True), (8, 128, 0, True), (4, 64, 512, False), (1, 8, 8, True), (1, 8, 0, False)])
@pytest.mark.parametrize("T,tail", [(0, 0), (0, 9), (40, 0), (13, 21)])
def test_selection_inside_the_copy_of_any_row(H, d, Dh, V, T, tail):
    for lengths in (False, True):
        assert "select_plain_kernel" not in _step(3, 130, T, tail, 50, H, d, Dh, False, lengths, V)


# one wave of CTAs, 256 tokens: beyond either line the selection is a kernel again
@pytest.mark.parametrize("B,n", [(1, 257), (60, 100)])
def test_selection_of_larger_calls_is_a_kernel(B, n):
    assert "select_plain_kernel" in _step(B, n, 4, 4, 50, 8, 128, 4096, False)
