"""The work that is timed: one pass of each call that a user of this framework makes, over the range of sizes it is used at.

A model that prunes its visual tokens with this library makes one call per pruning layer: Stage I behind the vision
encoder ("stage1": [CLS] saliency, selection, compaction of the features), Stage II at the first pruning layer of the
LLM ("stage2": clustering, K-norm, quota selection and compaction in one call), Stage III at the later ones ("stage3":
K-norm, top-k and compaction, the lengths taken from the device where the call before left them).  Beside them stand the
clustering by itself ("filter"), the merge of the dropped tokens ("merge") and the key projection that yields K and its
norms in one pass ("kproj").  Shapes are those of LLaVA-1.5-like images (576 tokens), AnyRes images (2880), clips of 32
frames (4608) and long videos with grouped-query attention (16384), and ragged sizes between them; all tensors are bf16
as the calls take them.
"""
import math

import torch

from paper_2601_17818_b200 import binding as vb


# ---------------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # one image, first pruning layer: the latency a single chat request sees
        _stage2("stage2_image_b1", 1, 576, 32, 128, 4096, 1024, 64, 192, "grid"),
        # a serving batch of images pruned hard (64 of 576)
        _stage2("stage2_image_b16", 16, 576, 32, 128, 4096, 1024, 64, 64, "grid"),
        # high-resolution images cut into five crops
        _stage2("stage2_anyres_b8", 8, 2880, 32, 128, 4096, 1024, 64, 640, "anyres"),
        # clips of 32 frames: neighbouring frames nearly repeat each other
        _stage2("stage2_video_b4", 4, 4608, 32, 128, 4096, 1024, 64, 1152, "video"),
        # the longest sequence the calls take, few K/V heads
        _stage2("stage2_long_b2", 2, 16384, 4, 128, 3584, 1280, 128, 2048, "long"),
        # clustering alone, Euclidean metric, no positions, a ragged token count and a narrow feature
        dict(name="filter_ragged_b3", kind="filter", B=3, n=1477, D=768, layout="grid", metric=1, spatial=False),
        # the last pruning layer of a single image: the smallest call there is
        _stage3("stage3_image_b1", 1, 128, 32, 128, 4096, 64, 64),
        # a pruning layer over a batch of high-resolution images: the largest plain step
        _stage3("stage3_anyres_b8", 8, 2880, 32, 128, 4096, 64, 640),
        # behind the vision encoder of a batch of images: half of the tokens go on
        dict(name="stage1_image_b16", kind="stage1", B=16, n=576, H=16, d=64, D=1024, budget=288),
        # tokens dropped from clips are averaged into one row per cluster
        dict(name="merge_video_b4", kind="merge", B=4, n=4608, Dh=4096, T=64, clusters=231),
        # keys of a batch of images with rotary embedding, all heads
        dict(name="kproj_image_b16", kind="kproj", B=16, N=640, n=576, T=64, Dh=4096, H=32, d=128, rope=True),
        # keys of two long videos, four heads, no rotation
        dict(name="kproj_long_b2", kind="kproj", B=2, N=16512, n=16384, T=128, Dh=3584, H=4, d=128, rope=False),
    ]


def draw(rng):
    while True:
        kind = rng.choice(["stage2", "stage2", "stage2", "stage2", "filter", "stage3", "stage3", "stage1", "merge", "kproj"])
        B = int(_log_uniform(rng, 1, 16))
        n = int(_log_uniform(rng, 64, 16384))
        T = rng.randint(9, 128)
        H, d = rng.choice([4, 8, 16, 32]), rng.choice([64, 128])
        Dh = rng.choice([1024, 2048, 3584, 4096])
        D = rng.choice([256, 768, 1024, 1280])
        layout = rng.choice(["grid", "anyres", "video", "long"])
        if kind == "stage2":
            case = _stage2("", B, n, H, d, Dh, D, T, max(1, int(n * rng.uniform(0.11, 0.5))), layout,
                           metric=rng.choice([0, 0, 0, 1]), spatial=rng.random() < 0.8)
        elif kind == "filter":
            case = dict(kind="filter", B=B, n=n, D=D, layout=layout, metric=rng.choice([0, 1]), spatial=rng.random() < 0.5)
        elif kind == "stage3":
            case = _stage3("", B, n, H, d, Dh, T, max(1, int(n * rng.uniform(0.06, 0.6))))
        elif kind == "stage1":
            n = int(_log_uniform(rng, 144, 2048))
            case = dict(kind="stage1", B=B, n=n, H=rng.choice([12, 16]), d=64, D=D, budget=max(1, int(n * rng.uniform(0.25, 0.5))))
        elif kind == "merge":
            case = dict(kind="merge", B=B, n=n, Dh=Dh, T=T, clusters=max(1, n // 20))
        else:
            case = dict(kind="kproj", B=B, N=n + T, n=n, T=T, Dh=Dh, H=H, d=d, rope=rng.random() < 0.6)
        case.pop("name", None)
        if "n" in case and case["B"] * case["n"] > 32768:
            continue
        # no dearer than the longest videos of the list
        w = work(case)
        if w["flops"] <= 6.8e11 and w["bytes"] <= 6e8:
            return case


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi + 0.999)))


def _stage2(name, B, n, H, d, Dh, D, T, budget, layout, metric=0, spatial=True):
    return dict(name=name, kind="stage2", B=B, n=n, H=H, d=d, Dh=Dh, D=D, T=T, budget=budget, layout=layout, metric=metric,
                spatial=spatial)


def _stage3(name, B, n, H, d, Dh, T, budget):
    return dict(name=name, kind="stage3", B=B, n=n, H=H, d=d, Dh=Dh, T=T, budget=budget)


# ---------------------------------------------------------------------------------------------- inputs
def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _features(g, c):
    """bf16 [B, n, D]: what a vision encoder yields -- patches of a few themes, each with a spread of its own, and the
    redundancy of the layout.  (Independent patches would all be equally dense, and every decision of the clustering a tie
    in the last bits.)"""
    B, n, D, layout = c["B"], c["n"], c["D"], c["layout"]
    m = 144 if layout == "video" else n                    # tokens of a frame
    themes = max(1, m // 20)
    # runs of neighbouring patches share a theme; a patch's own part is half to twice as long as the theme's, mostly less
    run = (torch.rand(B, m, generator=g, device="cuda") < 0.125).long().cumsum(1)
    theme = torch.randint(0, themes, (B, m + 1), generator=g, device="cuda").gather(1, run)
    f = _randn(g, B, themes, D).gather(1, theme[..., None].expand(-1, -1, D))
    f += 0.5 * torch.exp(0.5 * _randn(g, B, m, 1)) * _randn(g, B, m, D)
    if layout == "video":                                  # frame t + 1 is frame t plus N(0, 0.05) on the whole: some patches
        frames = -(-n // 144)                              # move, others rest
        cur = f.bfloat16()
        out = [cur]
        for _ in range(1, frames):
            cur = (cur.float() + 0.05 * torch.exp(_randn(g, B, 144, 1)) * _randn(g, B, 144, D)).bfloat16()
            out.append(cur)
        return torch.cat(out, 1)[:, :n].contiguous()
    share = {"grid": 0.2, "anyres": 0.3, "long": 0.4}[layout]
    n_dup = int(share * n)
    if n_dup:                                              # near-duplicates: a clean token close by, plus N(0, 0.01)
        order = torch.rand(B, n, generator=g, device="cuda").argsort(1)
        dup, clean = order[:, :n_dup].contiguous(), order[:, n_dup:].sort(1).values
        if layout == "anyres":                             # crops repeat the overview, anywhere in the sequence
            at = torch.randint(0, clean.shape[1], (B, n_dup), generator=g, device="cuda")
        else:                                              # the next clean tokens in reading order
            at = torch.searchsorted(clean, dup) + torch.randint(0, 4, (B, n_dup), generator=g, device="cuda")
            at = at.clamp_(max=clean.shape[1] - 1)
        src = clean.gather(1, at)
        rows = f.gather(1, src[..., None].expand(-1, -1, D))
        rows += 0.01 * torch.exp(_randn(g, B, n_dup, 1)) * _randn(g, B, n_dup, D)
        f.scatter_(1, dup[..., None].expand(-1, -1, D), rows)
    if layout == "long":                                   # a few outliers, ten times as long
        f.mul_(1.0 + 9.0 * (torch.rand(B, n, 1, generator=g, device="cuda") < 0.01))
    return f.bfloat16()


def _positions(c):
    """fp32 [B, n, 2]: coordinates in the unit square."""
    n, layout = c["n"], c["layout"]
    side = {"grid": 24, "anyres": 24, "video": 12, "long": 128}[layout]
    i = torch.arange(n, device="cuda")
    x = ((i % side).float() + 0.5) / side
    y = (((i // side) % side).float() + 0.5) / side
    if layout == "anyres":                                 # the overview covers the image, the crops a quarter each
        t = i // (side * side)
        q = (t - 1) % 4
        x = torch.where(t == 0, x, (x + (q % 2)) * 0.5)
        y = torch.where(t == 0, y, (y + (q // 2)) * 0.5)
    return torch.stack([x, y], -1)[None].expand(c["B"], n, 2).contiguous()


def _keys(g, B, H, N, d):
    """bf16 [B, H, N, d]: N(0, 1) with one log-normal scale per token."""
    return (_randn(g, B, H, N, d) * torch.exp(0.5 * _randn(g, B, 1, N, 1))).bfloat16()


def _clusters(c):
    return math.ceil(c["n"] * 0.05)


def _i32(*shape):
    return torch.zeros(*shape, dtype=torch.int32, device="cuda")


def _bf16(*shape):
    return torch.zeros(*shape, dtype=torch.bfloat16, device="cuda")


def _fp32(*shape):
    return torch.zeros(*shape, dtype=torch.float32, device="cuda")


def _filter_options(c):
    # the cutoff distance on the scale of the metric: unit vectors, or vectors of length sqrt(D)
    return dict(metric=c["metric"], d_c=0.5 if c["metric"] == 0 else 0.5 * math.sqrt(c["D"]), tau=0.6, n_centers=_clusters(c))


def _cache(s, g, c):
    """Hidden states, K and V of a layer, and the shortened ones."""
    B, H, d, Dh, N, cap = c["B"], c["H"], c["d"], c["Dh"], c["n"] + c["T"], c["T"] + min(c["budget"], c["n"])
    s["hidden"], s["K"], s["V"] = _randn(g, B, N, Dh).bfloat16(), _keys(g, B, H, N, d), _randn(g, B, H, N, d).bfloat16()
    s["hidden_out"], s["K_out"], s["V_out"] = _bf16(B, cap, Dh), _bf16(B, H, cap, d), _bf16(B, H, cap, d)
    s["kept_pos"], s["out_len"], s["n_keep"] = _i32(B, cap), _i32(B), _i32(B)


def prepare(case, seed):
    c, s = case, {"case": case}
    g = torch.Generator(device="cuda").manual_seed(seed)
    kind, B, n = c["kind"], c["B"], c["n"]
    if kind in ("stage2", "filter"):
        s["feat"] = _features(g, c)
        s["pos"] = _positions(c) if c["spatial"] else None
        s["label"], s["n_clusters"], s["options"] = _i32(B, n), _i32(B), _filter_options(c)
    if kind == "stage2":
        _cache(s, g, c)
        s["workspace"] = vb.alloc_workspace(vb.OP_COLLAB_STEP, B=B, Nv=n, D=c["D"])
    elif kind == "filter":
        s["rho"], s["delta2"], s["parent"] = _fp32(B, n), _fp32(B, n), _i32(B, n)
        s["workspace"] = vb.alloc_workspace(vb.OP_FILTER, B=B, Nv=n, D=c["D"])
    elif kind == "stage3":
        _cache(s, g, c)
        # as the call before left them on the device: every sample its own visual length (at most n)
        less = torch.randint(0, n // 16 + 1, (B,), generator=g, device="cuda", dtype=torch.int32)
        s["vis_len"] = (n - less).contiguous()
        s["seq_len"] = (s["vis_len"] + c["T"]).contiguous()
        s["workspace"] = vb.alloc_workspace(vb.OP_PRUNE_STEP, B=B, Nv=n)
    elif kind == "stage1":
        H, d, M, D, keep = c["H"], c["d"], n + 1, c["D"], c["budget"]
        q = _randn(g, B, H, d)
        K = _randn(g, B, H, M, d)
        # a few tokens that the [CLS] query looks at
        seen = (torch.rand(B, 1, M, 1, generator=g, device="cuda") < 0.05) * torch.rand(B, 1, M, 1, generator=g, device="cuda")
        s["q"], s["K"] = q.bfloat16(), (K + seen * 1.5 * q[:, :, None]).bfloat16()
        s["feat"], s["feat_out"] = _randn(g, B, M, D).bfloat16(), _bf16(B, 1 + keep, D)
        s["saliency"], s["keep"], s["n_keep"], s["out_len"] = _fp32(B, n), _i32(B, keep), _i32(B), _i32(B)
        s["ws_saliency"] = vb.alloc_workspace(vb.OP_SALIENCY, B=B, H=H, N=M)
        s["ws_select"] = vb.alloc_workspace(vb.OP_SELECT, B=B, Nv=n)
    elif kind == "merge":
        m = c["clusters"]
        s["hidden"] = _randn(g, B, n + c["T"], c["Dh"]).bfloat16()
        centres = torch.rand(B, n, generator=g, device="cuda").argsort(1)[:, :m].sort(1).values
        # uneven clusters: tokens pick a centre with a log-normal preference; a fifth of the tokens were kept
        pick = torch.multinomial(torch.exp(_randn(g, B, m)), n, replacement=True, generator=g)
        label = centres.gather(1, pick)
        label.scatter_(1, centres, centres)
        s["label"] = label.int().contiguous()
        s["keep_mask"] = (torch.rand(B, n, generator=g, device="cuda") < 0.2).to(torch.uint8)
        s["merged"] = _bf16(B, m, c["Dh"])
        s["merged_label"], s["merged_count"], s["n_merged"] = _i32(B, m), _i32(B, m), _i32(B)
        s["workspace"] = vb.alloc_workspace(vb.OP_MERGE, B=B, Nv=n, N=m)
    else:
        N, Dh, H, d = c["N"], c["Dh"], c["H"], c["d"]
        s["hidden"] = _randn(g, B, N, Dh).bfloat16()
        s["W"] = (_randn(g, H * d, Dh) * Dh ** -0.5).bfloat16()
        s["cos"] = s["sin"] = None
        if c["rope"]:
            freq = 10000.0 ** (-torch.arange(0, d, 2, device="cuda").float() / d)
            angle = torch.arange(N, device="cuda").float()[:, None] * freq[None]
            s["cos"], s["sin"] = angle.cos().contiguous(), angle.sin().contiguous()
        s["K_out"], s["score"] = _bf16(B, H, N, d), _fp32(B, n)
        s["workspace"] = vb.alloc_workspace(vb.OP_KPROJ, B=B, H=H, N=N, d=d)
    return s


# ---------------------------------------------------------------------------------------------- one pass
def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "stage2":
        vb.vitcop_collaborative_step(s["feat"], s["pos"], s["hidden"], s["K"], s["V"], c["T"], c["budget"], s["hidden_out"],
                                     s["K_out"], s["V_out"], s["out_len"], s["label"], s["n_clusters"], s["workspace"],
                                     kept_pos=s["kept_pos"], n_keep_out=s["n_keep"], **s["options"])
        return {k: s[k] for k in ("hidden_out", "K_out", "V_out", "out_len", "kept_pos", "n_keep", "label", "n_clusters")}
    if kind == "filter":
        vb.vitcop_redundancy_filter(s["feat"], s["pos"], s["label"], s["n_clusters"], s["workspace"], rho=s["rho"],
                                    delta2=s["delta2"], parent=s["parent"], **s["options"])
        return {k: s[k] for k in ("label", "n_clusters", "rho", "delta2", "parent")}
    if kind == "stage3":
        vb.vitcop_prune_step(s["hidden"], s["K"], s["V"], c["T"], s["vis_len"], c["n"], c["budget"], s["hidden_out"], s["K_out"],
                             s["V_out"], s["out_len"], s["workspace"], kept_pos=s["kept_pos"], seq_len=s["seq_len"],
                             n_keep_out=s["n_keep"])
        return {k: s[k] for k in ("hidden_out", "K_out", "V_out", "out_len", "kept_pos", "n_keep")}
    if kind == "stage1":
        vb.vitcop_cls_saliency(s["q"], s["K"], c["d"] ** -0.5, s["saliency"], s["ws_saliency"])
        vb.vitcop_select(s["saliency"], c["n"], c["budget"], s["keep"], s["n_keep"], s["ws_select"], largest=True)
        vb.vitcop_compact_kv(s["feat"], None, None, 1, c["n"], s["keep"], s["n_keep"], s["feat_out"], None, None, s["out_len"])
        return {k: s[k] for k in ("saliency", "keep", "n_keep", "feat_out", "out_len")}
    if kind == "merge":
        vb.vitcop_merge_clusters(s["hidden"], c["T"], c["n"], s["label"], s["keep_mask"], s["merged_label"], s["merged_count"],
                                 s["n_merged"], s["workspace"], merged=s["merged"])
        return {k: s[k] for k in ("merged", "merged_label", "merged_count", "n_merged")}
    vb.vitcop_kproj_knorm(s["hidden"], s["W"], c["H"], c["d"], s["K_out"], s["workspace"], vis_start=c["T"], score=s["score"],
                          rope_cos=s["cos"], rope_sin=s["sin"])
    return {"K_out": s["K_out"], "score": s["score"]}


# ---------------------------------------------------------------------------------------------- what a pass cannot do without
def work(case):
    c = case
    kind, B, n = c["kind"], c["B"], c["n"]
    if kind in ("stage2", "stage3"):
        kept = min(c["budget"], n)
        if kind == "stage2":                               # Eq. 5: the quotas sum up to the budget less one per cluster
            kept = max(0, kept - _clusters(c))
        # every visual row of K is read for its norm; only rows that stay are copied, and only those of V and hidden read
        rows = c["T"] + kept
        by = 2 * B * c["H"] * c["d"] * (n + c["T"] + 2 * rows + rows) + 2 * 2 * B * rows * c["Dh"]
        fl = 2 * B * c["H"] * c["d"] * n
        if kind == "stage3":
            return {"bytes": by, "flops": fl}
        by += 2 * B * n * c["D"] + (8 * B * n if c["spatial"] else 0) + 4 * B * n
        return {"bytes": by, "flops": fl + B * n * (n + 1) * c["D"]}      # one product per unordered pair of tokens
    if kind == "filter":
        return {"bytes": 2 * B * n * c["D"] + (8 * B * n if c["spatial"] else 0) + 16 * B * n, "flops": B * n * (n + 1) * c["D"]}
    if kind == "stage1":
        return {"bytes": 2 * B * c["H"] * (n + 2) * c["d"] + 4 * B * n + 2 * 2 * B * (1 + c["budget"]) * c["D"],
                "flops": 2 * B * c["H"] * (n + 1) * c["d"]}
    if kind == "merge":
        return {"bytes": int(0.8 * B * n * c["Dh"] * 2) + 2 * B * c["clusters"] * c["Dh"] + 5 * B * n, "flops": 0.8 * B * n * c["Dh"]}
    rows = B * c["N"]
    return {"bytes": 2 * rows * c["Dh"] + 2 * c["H"] * c["d"] * (c["Dh"] + rows) + 4 * B * n, "flops": 2 * rows * c["Dh"] * c["H"] * c["d"]}


def tolerance(case):
    kind = case["kind"]
    if kind == "kproj":
        # bf16 keys: against sums in 64 bits one value in four hundred rounds to the neighbouring bf16 (rel 1.5e-4; a
        # neighbour is at most 2^-7 of the value away)
        return {"rel": 6e-4, "max": 1e-2}
    if kind == "merge":
        # means rounded to bf16 once: no value fell on the other side against sums in 64 bits; another order may round a
        # few in a hundred thousand
        return {"rel": 1e-4, "max": 1e-2}
    # 32-bit sums (densities: rel 5e-6, max 1e-5 against 64 bits); copied rows are bit for bit, indices differ only where
    # two values tie to the last bits
    return {"rel": 2e-5, "max": 1e-4, "differ": 1e-3}
