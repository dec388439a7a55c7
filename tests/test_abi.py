"""Host-only checks of the C ABI: the library loads, exports what the header declares, and rejects bad
arguments before touching the device.  No compute call is made here."""
import ctypes as C
import os
import re

import pytest
import torch

from paper_2601_17818_b200 import binding as vb
from paper_2601_17818_b200.build import build_library

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def L():
    build_library()
    return vb.lib()


def test_header_symbols_are_exported(L):
    text = open(os.path.join(ROOT, "include", "vitcop.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    declared = sorted(set(re.findall(r"\b(vitcop_[a-z_]+)\s*\(", text)))
    assert len(declared) >= 10
    for name in declared:
        assert hasattr(L, name), name
    assert sorted(vb.EXPORTS) == declared


def test_status_strings(L):
    seen = set()
    for s in range(7):
        msg = L.vitcop_status_string(s).decode()
        assert msg and msg != "unknown status"
        seen.add(msg)
    assert len(seen) == 7
    assert L.vitcop_status_string(99).decode() == "unknown status"


def test_workspace_sizes():
    assert vb.vitcop_workspace_bytes(vb.OP_KNORM, B=4, Nv=100) == 0
    assert vb.vitcop_workspace_bytes(vb.OP_COMPACT, B=4, Nv=100) == 0
    assert vb.vitcop_workspace_bytes(vb.OP_SELECT, B=4, Nv=100) >= 4
    s1 = vb.vitcop_workspace_bytes(vb.OP_PRUNE_STEP, B=16, Nv=576)
    assert s1 >= 16 * 576 * 8 + 16 * 4
    f1 = vb.vitcop_workspace_bytes(vb.OP_FILTER, B=2, Nv=1000, D=128)
    f2 = vb.vitcop_workspace_bytes(vb.OP_FILTER, B=4, Nv=1000, D=128)
    assert f2 > f1 > 2 * 1000 * 20
    with pytest.raises(vb.VitcopError) as e:
        vb.vitcop_workspace_bytes(77)
    assert e.value.status == vb.ERR_INVALID_ARG
    with pytest.raises(vb.VitcopError):
        vb.vitcop_workspace_bytes(vb.OP_SELECT, B=-1)


@pytest.mark.parametrize("arg,error", [(torch.zeros(4), ValueError), ("text", TypeError), (1.5, TypeError),
                                       (2 ** 70, OverflowError)])
def test_native_caller_rejects_what_it_cannot_pass(L, arg, error):
    """A tensor that is not on the device, and whatever is neither a tensor nor an integer, never reaches the library."""
    with pytest.raises(error):
        vb._native(vb._address["vitcop_select"], 0.0, arg)
    with pytest.raises(TypeError):
        vb._native(vb._address["vitcop_select"], 0.0, *[0] * 40)


def test_native_caller_calls_every_entry_point_by_its_type(L):
    """Each with as many words as it has parameters (the float of the saliency travels apart), neither more nor fewer, and
    whatever the host's calling convention."""
    text = open(os.path.join(ROOT, "include", "vitcop.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    for name in vb.NATIVE:
        params = re.search(r"\bint\s+" + name + r"\s*\(([^)]*)\)", text).group(1).split(",")
        words = sum(not p.strip().startswith("float scale") for p in params)
        refused = (vb.ERR_INVALID_ARG, vb.ERR_CUDA) if name == "vitcop_prune_step_static" else (vb.ERR_INVALID_ARG,)
        assert vb._native(vb._address[name], 0.5, *[0] * words) in refused, name       # (the static step looks its scratch up first)
        for wrong in (words - 1, words + 1):
            with pytest.raises(TypeError):
                vb._native(vb._address[name], 0.5, *[0] * wrong)
    source = open(os.path.join(ROOT, "paper_2601_17818_b200", "csrc", "call.cpp")).read()
    assert "__x86_64__" not in source and "#error" not in source
    with pytest.raises(ValueError):
        vb._native(len(vb.NATIVE), 0.0)


@pytest.mark.parametrize("op", [vb.OP_FILTER, vb.OP_COLLAB_STEP])
def test_a_workspace_of_a_larger_problem_serves_a_smaller_one(L, op):
    sizes = [1, 64, 127, 128, 129, 576, 577, 1408, 1409, 1536, 2048, 2880, 4608, 8191, 8192, 12000, 16384]
    batches = [1, 2, 3, 5, 8, 11, 12, 16, 40, 149, 300, 6144, 6145]
    need = [[vb.vitcop_workspace_bytes(op, B=B, Nv=n, D=64) for n in sizes] for B in batches]
    for i in range(len(batches)):
        for j in range(len(sizes)):
            assert i == 0 or need[i][j] >= need[i - 1][j], (batches[i], sizes[j])
            assert j == 0 or need[i][j] >= need[i][j - 1], (batches[i], sizes[j])


@pytest.mark.parametrize("values", [(0, 0.5, 0.6, 0.05, 29), (1, 8.0, 1e300, 0.05, 0), (0, 1e39, -1e39, 2.0, 2 ** 31),
                                    (0, float("inf"), float("nan"), 1e300, -2 ** 40)])
def test_parameters_are_converted_as_c_does(values):
    """Whatever the struct of the ABI takes, the binding passes: out of a field's range too."""
    assert vb._filter_params(*values) == bytes(vb.FilterParams(*values))
    ints = (0, 1, values[-1])
    assert vb._select_params(*ints) == bytes(vb.SelectParams(*ints))


def test_argument_validation_happens_on_the_host(L):
    """Every call below must return before any CUDA work (there may be no device at all)."""
    fake = C.c_void_p(0x1000)                       # 16-byte aligned, never dereferenced by the checks
    odd = C.c_void_p(0x1008)
    ws = C.c_void_p(0x10000)
    null = None
    # knorm
    assert L.vitcop_knorm_score(null, 1, 1, 8, 8, 64, 64, 8, 0, null, 4, fake, 4, null) == vb.ERR_INVALID_ARG
    assert L.vitcop_knorm_score(fake, 1, 1, 8, 8, 64, 64, 8, 6, null, 4, fake, 4, null) == vb.ERR_INVALID_ARG  # span > N
    assert L.vitcop_knorm_score(fake, 1, 1, 8, 8, 64, 64, 8, 0, null, 5, fake, 4, null) == vb.ERR_INVALID_ARG  # len > cap
    assert L.vitcop_knorm_score(fake, -1, 1, 8, 8, 64, 64, 8, 0, null, 4, fake, 4, null) == vb.ERR_INVALID_ARG
    assert L.vitcop_knorm_score(fake, 1, 1, 8, 12, 96, 96, 12, 0, null, 4, fake, 4, null) == vb.ERR_UNSUPPORTED  # d % 8
    assert L.vitcop_knorm_score(odd, 1, 1, 8, 8, 64, 64, 8, 0, null, 4, fake, 4, null) == vb.ERR_UNSUPPORTED   # alignment
    # select
    p = vb.SelectParams(0, 0, 3)
    assert L.vitcop_select(null, null, 1, null, 4, 4, C.byref(p), fake, 4, fake, null, ws, 256, null) == vb.ERR_INVALID_ARG
    assert L.vitcop_select(fake, null, 1, null, 4, 4, C.byref(p), fake, 2, fake, null, ws, 256, null) == vb.ERR_INVALID_ARG  # keep_stride < budget
    assert L.vitcop_select(fake, null, 1, null, 4, 4, C.byref(p), fake, 4, fake, null, null, 0, null) == vb.ERR_WORKSPACE
    assert L.vitcop_select(fake, null, 1, null, 4, 4, C.byref(p), fake, 4, fake, null, ws, 8, null) == vb.ERR_WORKSPACE
    q = vb.SelectParams(1, 0, 3)
    assert L.vitcop_select(fake, null, 1, null, 4, 4, C.byref(q), fake, 4, fake, null, ws, 256, null) == vb.ERR_INVALID_ARG  # quota needs labels
    neg = vb.SelectParams(0, 0, -1)
    assert L.vitcop_select(fake, null, 1, null, 4, 4, C.byref(neg), fake, 4, fake, null, ws, 256, null) == vb.ERR_INVALID_ARG
    big = vb.SelectParams(0, 0, 3)
    assert L.vitcop_select(fake, null, 1, null, 4, 20000, C.byref(big), fake, 4, fake, null, ws, 256, null) == vb.ERR_UNSUPPORTED
    # compact: missing output for a given input, aliasing, bad span
    a, b = C.c_void_p(0x100000), C.c_void_p(0x900000)
    assert L.vitcop_compact_kv(a, null, null, 1, 1, 8, 8, 8, null, 0, null, 4, fake, 4, fake, null, null, null, 8, null, fake, null) == vb.ERR_INVALID_ARG
    assert L.vitcop_compact_kv(a, null, null, 1, 1, 8, 8, 8, null, 0, null, 4, fake, 4, fake, a, null, null, 8, null, fake, null) == vb.ERR_INVALID_ARG
    assert L.vitcop_compact_kv(a, null, null, 1, 1, 8, 8, 8, null, 6, null, 4, fake, 4, fake, b, null, null, 8, null, fake, null) == vb.ERR_INVALID_ARG
    assert L.vitcop_compact_kv(a, null, null, 1, 1, 8, 8, 12, null, 0, null, 4, fake, 4, fake, b, null, null, 8, null, fake, null) == vb.ERR_UNSUPPORTED
    # filter
    fp = vb.FilterParams(0, 0.5, 0.6, 0.05, 0)
    assert L.vitcop_redundancy_filter(null, null, 1, 8, 64, C.byref(fp), fake, fake, null, null, null, ws, 1 << 20, null) == vb.ERR_INVALID_ARG
    assert L.vitcop_redundancy_filter(fake, null, 1, 8, 72, C.byref(fp), fake, fake, null, null, null, ws, 1 << 20, null) == vb.ERR_UNSUPPORTED
    assert L.vitcop_redundancy_filter(fake, null, 1, 8, 64, C.byref(fp), fake, fake, null, null, null, ws, 16, null) == vb.ERR_WORKSPACE
    bad = vb.FilterParams(0, 0.0, 0.6, 0.05, 0)
    assert L.vitcop_redundancy_filter(fake, null, 1, 8, 64, C.byref(bad), fake, fake, null, null, null, ws, 1 << 20, null) == vb.ERR_INVALID_ARG
    bad = vb.FilterParams(3, 0.5, 0.6, 0.05, 0)
    assert L.vitcop_redundancy_filter(fake, null, 1, 8, 64, C.byref(bad), fake, fake, null, null, null, ws, 1 << 20, null) == vb.ERR_INVALID_ARG
    assert L.vitcop_similarity_rows(fake, 1, 8, 64, 0, 4, 2, fake, ws, 1 << 20, null) == vb.ERR_INVALID_ARG
    # prune step
    assert L.vitcop_prune_step(null, null, null, 1, 1, 8, 8, 8, null, 0, null, 4, 4, null, 2, null, null, null, 8, null, fake, null, null, null, ws, 1 << 20, null) == vb.ERR_INVALID_ARG
    assert L.vitcop_prune_step(null, a, null, 1, 1, 8, 8, 8, null, 0, null, 4, 4, null, 2, null, b, null, 8, null, fake, null, null, null, null, 0, null) == vb.ERR_WORKSPACE


def test_argument_validation_of_the_wider_entry_points(L):
    fake, odd, ws, null = C.c_void_p(0x1000), C.c_void_p(0x1008), C.c_void_p(0x10000), None
    a, b = C.c_void_p(0x100000), C.c_void_p(0x900000)
    fp = vb.FilterParams(0, 0.5, 0.6, 0.05, 0)
    # merge: required pointers, Dh % 8, workspace
    assert L.vitcop_merge_clusters(null, 1, 8, 8, 0, null, 4, 4, fake, fake, null, null, fake, fake, fake, 4, ws, 1 << 20, null) == vb.ERR_INVALID_ARG
    assert L.vitcop_merge_clusters(a, 1, 8, 12, 0, null, 4, 4, fake, fake, null, null, fake, fake, fake, 4, ws, 1 << 20, null) == vb.ERR_UNSUPPORTED
    assert L.vitcop_merge_clusters(a, 1, 8, 8, 6, null, 4, 4, fake, fake, null, null, fake, fake, fake, 4, ws, 1 << 20, null) == vb.ERR_INVALID_ARG   # span > N
    assert L.vitcop_merge_clusters(a, 1, 8, 8, 0, null, 4, 4, fake, fake, null, null, fake, fake, fake, 4, ws, 8, null) == vb.ERR_WORKSPACE
    # saliency
    assert L.vitcop_cls_saliency(null, fake, 1, 1, 4, 8, 0.5, fake, null, ws, 1 << 20, null) == vb.ERR_INVALID_ARG
    assert L.vitcop_cls_saliency(fake, fake, 1, 1, 4, 12, 0.5, fake, null, ws, 1 << 20, null) == vb.ERR_UNSUPPORTED
    assert L.vitcop_cls_saliency(fake, odd, 1, 1, 4, 8, 0.5, fake, null, ws, 1 << 20, null) == vb.ERR_UNSUPPORTED
    assert L.vitcop_cls_saliency(fake, fake, 1, 1, 4, 8, 0.5, fake, null, ws, 16, null) == vb.ERR_WORKSPACE
    # one-call Stage II: needs labels out, a valid metric / cutoff, D % 64, a workspace
    args = lambda feat=fake, D=64, f=fp, lab=fake, wsb=1 << 24, B=1: (feat, null, D, C.byref(f), null, a, null, B, 1, 8, 8, 8, 0, 4, 2, null, b, null, 8, null, fake, lab, fake, null, null, null, null, null, null, ws, wsb, null)
    assert L.vitcop_collaborative_step(*args(lab=null)) == vb.ERR_INVALID_ARG
    assert L.vitcop_collaborative_step(*args(f=vb.FilterParams(0, 0.0, 0.6, 0.05, 0))) == vb.ERR_INVALID_ARG
    assert L.vitcop_collaborative_step(*args(D=72)) == vb.ERR_UNSUPPORTED
    assert L.vitcop_collaborative_step(*args(wsb=64)) == vb.ERR_WORKSPACE
    assert L.vitcop_collaborative_step(*args(B=65536, wsb=1 << 40)) == vb.ERR_UNSUPPORTED      # as its sibling calls
    # K projection: weights required, cos and sin together, rotation only for head sizes whose halves are chunk-aligned
    kp = lambda hid=fake, W=fake, Dh=64, d=64, cos=null, sin=null, npos=0, wsb=1 << 24: (hid, W, 1, 8, Dh, 2, d, cos, sin, null, npos, b, 0, 4, fake, ws, wsb, null)
    assert L.vitcop_kproj_knorm(*kp(W=null)) == vb.ERR_INVALID_ARG
    assert L.vitcop_kproj_knorm(*kp(cos=fake)) == vb.ERR_INVALID_ARG
    assert L.vitcop_kproj_knorm(*kp(Dh=72)) == vb.ERR_UNSUPPORTED
    assert L.vitcop_kproj_knorm(*kp(d=32, cos=fake, sin=fake, npos=8)) == vb.ERR_UNSUPPORTED
    assert L.vitcop_kproj_knorm(*kp(wsb=64)) == vb.ERR_WORKSPACE
    assert vb.vitcop_workspace_bytes(vb.OP_KPROJ, B=2, H=4, N=100, d=128) >= 2 * 2 * 100 * 4
    assert vb.vitcop_workspace_bytes(vb.OP_COLLAB_STEP, B=2, Nv=100, D=64) > vb.vitcop_workspace_bytes(vb.OP_FILTER, B=2, Nv=100, D=64)
    assert vb.vitcop_workspace_bytes(vb.OP_MERGE, B=2, Nv=100, N=10) >= 256 + 2 * 100 * 2
    assert vb.vitcop_workspace_bytes(vb.OP_SALIENCY, B=2, H=4, N=33) >= 2 * 4 * 33 * 4


def test_the_caller_belongs_to_one_torch_and_one_interpreter(monkeypatch):
    """The extension is compiled against torch's and Python's headers: with another version of either it is neither taken for
    up to date nor found."""
    from paper_2601_17818_b200 import build
    path, digest = build.caller_path(), build._caller_digest()
    monkeypatch.setattr(torch, "__version__", "9.9.9")
    assert build.caller_path() != path and build._caller_digest() != digest
    monkeypatch.setattr(vb, "_lib", None)
    with pytest.raises(ImportError):
        vb.lib()
    monkeypatch.undo()
    assert build.caller_path() == path and os.path.exists(path)


def test_host_only_calls_need_no_cuda_in_torch():
    import subprocess
    import sys
    code = ("import torch\nfor name in ('_cuda_getCurrentRawStream', '_cuda_getDevice'):\n    delattr(torch._C, name)\n"
            "from paper_2601_17818_b200 import binding as vb\nassert vb.vitcop_stage_count(576, 0.5) == 288\n")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-800:]


def test_missing_library_fails_loudly(tmp_path, monkeypatch):
    monkeypatch.setattr(vb, "_lib", None)
    monkeypatch.setattr(vb, "LIB_PATH", str(tmp_path / "nope.so"))
    with pytest.raises(ImportError):
        vb.lib()
