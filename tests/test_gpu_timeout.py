"""The give-up path of the Gram kernels' bounded waits, through the C ABI (``-m gpu``).

Every device-side wait of the library is bounded; when one runs out the CTA abandons its work, lets what it has in
flight finish, frees its tensor memory, and the call reports VITCOP_ERR_TIMEOUT through the status word.  No wait
runs out in normal operation, so these tests send one role of every CTA down that path (vitcop_set_wait_limit with
``expire_roles``) while the other roles have copies and tensor-core work in flight, and check that the call
returns, reports the timeout, and that the same workspace gives correct results on the next normal call.
"""
import numpy as np
import pytest
import torch

from paper_2601_17818_b200 import binding as vb
from paper_2601_17818_b200 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_helpers import DEV

ROLE_LOAD, ROLE_MMA, ROLE_EPILOGUE = 1, 2, 4


@pytest.fixture(autouse=True)
def _restore_default_limit():
    yield
    vb.vitcop_set_wait_limit(0, 0)


def _filter_call(feat, pos, w, ws, out):
    vb.vitcop_redundancy_filter(feat, pos, out["label"], out["ncl"], ws, metric=0, d_c=w.d_c, tau=w.tau,
                                n_centers=out["nc"], rho=out["rho"], delta2=out["d2"], parent=out["par"])
    return vb.vitcop_poll_status(ws)


# B = 2 runs the one-kernel sweep (accumulators resident in tensor memory, cooperative launch, flags between CTAs);
# B = 80 exceeds what one wave of CTAs can keep resident and runs the diagonal, the density sweep and the search.
@pytest.mark.parametrize("B,n", [(2, 200), (80, 300)])
@pytest.mark.parametrize("roles", [ROLE_EPILOGUE, ROLE_MMA, ROLE_LOAD])
def test_filter_reports_timeout_and_recovers(B, n, roles):
    w = W.workload("tiny")
    f = W.make_features(w, n=n, B=B)
    feat = vb.bf16_tensor(f)
    pos = torch.from_numpy(np.tile(W.make_positions(w, n)[:1], (B, 1, 1)).copy()).to(DEV)
    nc = max(1, n // 20)

    def outputs():
        z = lambda *s, dt: torch.zeros(s, dtype=dt, device=DEV)
        return dict(label=z(B, n, dt=torch.int32), ncl=z(B, dt=torch.int32), rho=z(B, n, dt=torch.float32),
                    d2=z(B, n, dt=torch.float32), par=z(B, n, dt=torch.int32), nc=nc)

    ws = vb.alloc_workspace(vb.OP_FILTER, B=B, Nv=n, D=w.D)
    ref = outputs()
    assert _filter_call(feat, pos, w, ws, ref) == vb.OK
    vb.vitcop_set_wait_limit(0, roles)
    bad = outputs()
    assert _filter_call(feat, pos, w, ws, bad) == vb.ERR_TIMEOUT           # the call returned and says so
    vb.vitcop_set_wait_limit(0, 0)
    got = outputs()
    assert _filter_call(feat, pos, w, ws, got) == vb.OK                    # same workspace, next call is clean
    for key in ("label", "ncl", "rho", "d2", "par"):
        assert torch.equal(got[key], ref[key]), key


# The density sweep's pairs of CTAs give up by themselves: the diagonal in front of them has its normal limit.
@pytest.mark.parametrize("B,n", [(80, 300), (6, 1700)])
@pytest.mark.parametrize("roles", [ROLE_EPILOGUE, ROLE_MMA, ROLE_LOAD])
def test_density_sweep_reports_timeout_and_recovers(B, n, roles):
    feat = torch.randn((B, n, 256), generator=torch.Generator(device=DEV).manual_seed(n), device=DEV).to(torch.bfloat16)
    ws = vb.alloc_workspace(vb.OP_FILTER, B=B, Nv=n, D=256)

    def run():
        o = [torch.zeros((B, n), dtype=t, device=DEV) for t in (torch.int32, torch.float32, torch.float32, torch.int32)]
        vb.vitcop_redundancy_filter(feat, None, o[0], torch.zeros(B, dtype=torch.int32, device=DEV), ws, n_centers=n // 20,
                                    rho=o[1], delta2=o[2], parent=o[3])
        return vb.vitcop_poll_status(ws), o

    status, ref = run()
    assert status == vb.OK
    vb.vitcop_set_wait_limit(0, roles * 8)
    assert run()[0] == vb.ERR_TIMEOUT
    small = vb.alloc_workspace(vb.OP_FILTER, B=1, Nv=200, D=256)          # the one-kernel sweep is no pair kernel
    vb.vitcop_redundancy_filter(feat[:1, :200].contiguous(), None, torch.zeros((1, 200), dtype=torch.int32, device=DEV),
                                torch.zeros(1, dtype=torch.int32, device=DEV), small, n_centers=10)
    assert vb.vitcop_poll_status(small) == vb.OK
    vb.vitcop_set_wait_limit(0, 0)
    status, got = run()
    assert status == vb.OK and all(torch.equal(a, b) for a, b in zip(got, ref))


# Beyond 8192 tokens the labels follow the parents in rounds.  The sweep gives up in a workspace that holds 0.5 and -1.5 by turns: every
# other token has the same negative density, the blocks' minima let the search look at them, and they are one another's parents.
@pytest.mark.parametrize("roles", [ROLE_EPILOGUE, ROLE_LOAD])
def test_long_samples_report_timeout_and_recover(roles):
    B, n = 2, 9000
    feat = torch.randn((B, n, 64), generator=torch.Generator(device=DEV).manual_seed(n), device=DEV).to(torch.bfloat16)
    ws = vb.alloc_workspace(vb.OP_FILTER, B=B, Nv=n, D=64)

    def run():
        label = torch.full((B, n), -1, dtype=torch.int32, device=DEV)
        ws.view(torch.float32)[0::2] = 0.5
        ws.view(torch.float32)[1::2] = -1.5
        vb.vitcop_redundancy_filter(feat, None, label, torch.zeros(B, dtype=torch.int32, device=DEV), ws, n_centers=n // 20)
        return vb.vitcop_poll_status(ws), label

    status, ref = run()
    assert status == vb.OK
    vb.vitcop_set_wait_limit(0, roles * 8)
    status, label = run()
    assert status == vb.ERR_TIMEOUT and int(label.min()) >= 0 and int(label.max()) < n
    vb.vitcop_set_wait_limit(0, 0)
    status, got = run()
    assert status == vb.OK and torch.equal(got, ref)


def test_sweeps_of_several_streams_end_together():
    """One-kernel sweeps that each want every SM, from three streams of two priorities at once: the CTAs of each wait for one
    another, so they may not keep one another from starting."""
    B, n, D, calls = 16, 576, 256, 12                      # 208 units: 148 CTAs with one or two
    feat = torch.randn((B, n, D), generator=torch.Generator(device=DEV).manual_seed(5), device=DEV).to(torch.bfloat16)
    streams = [torch.cuda.Stream(priority=p) for p in (0, -1, 0)]
    ws = [[vb.alloc_workspace(vb.OP_FILTER, B=B, Nv=n, D=D) for _ in range(calls)] for _ in range(4)]
    z = lambda *s: torch.zeros(s, dtype=torch.int32, device=DEV)
    label, ncl = [[z(B, n) for _ in range(calls)] for _ in range(4)], z(B)

    def call(s, i):
        vb.vitcop_redundancy_filter(feat, None, label[s][i], ncl, ws[s][i], n_centers=29)

    call(3, 0)
    torch.cuda.synchronize()
    for i in range(calls):
        for s, stream in enumerate(streams):
            with torch.cuda.stream(stream):
                call(s, i)
    torch.cuda.synchronize()
    for s in range(3):
        for i in range(calls):
            assert vb.vitcop_poll_status(ws[s][i]) == vb.OK
            assert torch.equal(label[s][i], label[3][0])


def test_similarity_rows_reports_timeout_and_recovers():
    w = W.workload("tiny")
    f = W.make_features(w)
    feat = vb.bf16_tensor(f)
    B, n, D = feat.shape
    ws = vb.alloc_workspace(vb.OP_SIMILARITY, B=B, Nv=n, D=D)
    ref = torch.zeros((B, n, n), dtype=torch.float32, device=DEV)
    vb.vitcop_similarity_rows(feat, 0, 0, n, ref, ws)
    assert vb.vitcop_poll_status(ws) == vb.OK
    vb.vitcop_set_wait_limit(0, ROLE_EPILOGUE)
    vb.vitcop_similarity_rows(feat, 0, 0, n, torch.zeros_like(ref), ws)
    assert vb.vitcop_poll_status(ws) == vb.ERR_TIMEOUT
    vb.vitcop_set_wait_limit(0, 0)
    got = torch.zeros_like(ref)
    vb.vitcop_similarity_rows(feat, 0, 0, n, got, ws)
    assert vb.vitcop_poll_status(ws) == vb.OK and torch.equal(got, ref)


def test_one_call_step_reports_timeout_and_recovers():
    """The one-kernel sweep with its K-norm side work (tensor copies streamed by the warps beside the epilogue)."""
    w = W.workload("tiny")
    B, n = w.B, w.Nv
    feat = vb.bf16_tensor(W.make_features(w))
    pos = torch.from_numpy(W.make_positions(w).copy()).to(DEV)
    K_b, V_b = W.make_kv(w, 0, n)
    tK, tV, th = vb.bf16_tensor(K_b), vb.bf16_tensor(V_b), vb.bf16_tensor(W.make_hidden(w))
    budget, Ncap = w.budgets[0], w.T + w.budgets[0]

    def run(ws):
        z = lambda *s, dt: torch.zeros(s, dtype=dt, device=DEV)
        o = dict(ho=z(B, Ncap, w.Dh, dt=torch.bfloat16), Ko=z(B, w.H, Ncap, w.d, dt=torch.bfloat16),
                 Vo=z(B, w.H, Ncap, w.d, dt=torch.bfloat16), olen=z(B, dt=torch.int32), label=z(B, n, dt=torch.int32),
                 ncl=z(B, dt=torch.int32), score=z(B, n, dt=torch.float32))
        vb.vitcop_collaborative_step(feat, pos, th, tK, tV, w.vis_start, budget, o["ho"], o["Ko"], o["Vo"], o["olen"],
                                     o["label"], o["ncl"], ws, metric=0, d_c=w.d_c, tau=w.tau, n_centers=w.n_centers,
                                     score_out=o["score"])
        return vb.vitcop_poll_status(ws), o

    ws = vb.alloc_workspace(vb.OP_COLLAB_STEP, B=B, Nv=n, D=w.D)
    st, ref = run(ws)
    assert st == vb.OK
    for roles in (ROLE_EPILOGUE, ROLE_MMA):
        vb.vitcop_set_wait_limit(0, roles)
        st, _ = run(ws)
        assert st == vb.ERR_TIMEOUT
        vb.vitcop_set_wait_limit(0, 0)
        st, got = run(ws)
        assert st == vb.OK
        for key in ("label", "olen", "score"):
            assert torch.equal(got[key], ref[key]), key
        for key in ("ho", "Ko", "Vo"):
            assert torch.equal(got[key].view(torch.int16), ref[key].view(torch.int16)), key


@pytest.mark.parametrize("N", [10300, 5000])
@pytest.mark.parametrize("roles", [ROLE_EPILOGUE, ROLE_MMA, ROLE_LOAD])
def test_kproj_reports_timeout_and_recovers(roles, N):
    """The key projection's pairs of CTAs (10300 tokens; 5000 on CTAs apart): whichever role gives up, all CTAs leave."""
    B, H, d, Dh = 1, 4, 128, 512
    g = torch.Generator(device=DEV).manual_seed(3)
    hid = torch.randn((B, N, Dh), generator=g, device=DEV).to(torch.bfloat16)
    Wk = torch.randn((H * d, Dh), generator=g, device=DEV).to(torch.bfloat16)
    ws = vb.alloc_workspace(vb.OP_KPROJ, B=B, H=H, N=N, d=d)

    def run():
        K = torch.zeros((B, H, N, d), dtype=torch.bfloat16, device=DEV)
        score = torch.zeros((B, N), dtype=torch.float32, device=DEV)
        vb.vitcop_kproj_knorm(hid, Wk, H, d, K, ws, score=score)
        return vb.vitcop_poll_status(ws), K, score

    st, K0, s0 = run()
    assert st == vb.OK
    vb.vitcop_set_wait_limit(0, roles)
    assert run()[0] == vb.ERR_TIMEOUT
    vb.vitcop_set_wait_limit(0, 0)
    st, K1, s1 = run()
    assert st == vb.OK and torch.equal(K0.view(torch.int16), K1.view(torch.int16)) and torch.equal(s0, s1)
