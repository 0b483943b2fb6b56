"""The calls whose speed is measured, over the sizes that users of this library run.

A case is a dict of plain values with a "kind" (the entry point) and its sizes. The sizes are those of
the repository's own workloads: LLaVA-1.5 (one tile of 1 + 576 patches x 1024, 64 text tokens), LLaVA-NeXT
(5 crops a request), the Qwen2-style GQA decoder with one image of 256-4096 merged tokens a request, a
serving sweep of 1-64 tiles and sequences, decode steps after the prefill. Inputs follow the synthetic
recipe of the tests (planted feature groups with per-token noise, salient attention, normal weights).
Models of whole calls have all their layers; the cases of a layer's kernels have two to four layers
of the same width.

`exact` is the same mathematics in 64-bit torch without any of the 16-bit roundings in between.
"""
import math

import numpy as np
import torch

from paper_2609_34977_gb300 import _native as N
from paper_2609_34977_gb300.pipeline import SpiderPrefill

BF16 = torch.bfloat16
SHAPES = {
    "llava": dict(d_model=4096, n_heads=32, n_kv_heads=32, head_dim=128, d_ffn=11008, vocab=32000,
                  rope_theta=1e4, rms_eps=1e-5, d_vis=0, d_proj=0),
    "qwen": dict(d_model=3584, n_heads=28, n_kv_heads=4, head_dim=128, d_ffn=18944, vocab=152064,
                 rope_theta=1e6, rms_eps=1e-6, d_vis=0, d_proj=0),
}
EPILOGUES = {"f32": N.EPI_F32, "bf16": N.EPI_BF16, "bias": N.EPI_BIAS_BF16, "gelu": N.EPI_BIAS_GELU_BF16}


def listed():
    return [
        # one projection on its own: a small batch of rows, where the call itself counts
        dict(name="linear", kind="linear", m=77, n=4096, k=1024, epi="gelu"),
        # MSV-Prune of a single request's image: latency of a chain of small kernels
        dict(name="prune_one", kind="prune", form=0, tiles=1, n=576, d=1024, heads=16, keep=192),
        # MSV-Prune of a serving batch of tiles
        dict(name="prune_batch", kind="prune", form=0, tiles=64, n=576, d=1024, heads=16, keep=64),
        # one image of dynamic resolution, encoder without [CLS]: odd token count, wider rows
        dict(name="prune_varres", kind="prune", form=1, tiles=1, n=2739, d=1280, heads=16, keep=685),
        # received attention from the full maps of one large image through the 2 x 2 merger
        dict(name="received", kind="received", maps=16, rows=64, cols=60),
        # the attention of a dense GQA prefill: four requests of different lengths
        dict(name="attention", kind="attention", shape="qwen", lens="2996,3302,2995,1021", active=100),
        # decoder layers of one LLaVA-1.5 request without pruning or skipping
        dict(name="prefill_dense", kind="prefill", shape="llava", layers=2, vis="576", text="64", skip=0),
        # decoder layers of a batch of eight pruned LLaVA-NeXT requests under a skip plan
        dict(name="prefill_batch", kind="prefill", shape="llava", layers=2, vis="320,320,320,320,320,320,320,320",
             text="128,128,128,128,128,128,128,128", skip=45),
        # the online skip plan (logit lens of every candidate in the decision window)
        dict(name="adaptive", kind="adaptive", shape="llava", layers=4, vis=192, text=64, device_plan=1),
        # one generated token of one request, the whole LLaVA-1.5 decoder
        dict(name="decode_one", kind="decode", shape="llava", layers=32, pos="256", max_len=512),
        # one generated token of each of 32 requests at different depths of their contexts
        dict(name="decode_batch", kind="decode", shape="qwen", layers=4,
             pos=",".join(str(300 + 53 * i) for i in range(32)), max_len=2048),
        # the whole step of one LLaVA-1.5 request: prune, projector, 32 layers under a skip plan, logits
        dict(name="step", kind="step", layers=32, tiles="1", text="64", keep=192, skip=90),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _ints(s):
    return [int(v) for v in s.split(",")]


def _join(v):
    return ",".join(str(int(x)) for x in v)


def draw(rng):
    kind = rng.choice(["linear", "prune", "prune", "received", "attention", "prefill", "prefill", "adaptive",
                       "decode", "decode", "step"])
    if kind == "linear":
        return dict(kind=kind, m=_log(rng, 1, 4096), n=128 * _log(rng, 8, 96), k=8 * _log(rng, 32, 1024),
                    epi=rng.choice(sorted(EPILOGUES)))
    if kind == "prune" and rng.random() < 0.6:
        return dict(kind=kind, form=0, tiles=_log(rng, 1, 64), n=576, d=1024, heads=16, keep=rng.randint(32, 320))
    if kind == "prune":
        n = _log(rng, 256, 4096)
        return dict(kind=kind, form=1, tiles=1, n=n, d=1280, heads=16, keep=max(1, round(n * rng.uniform(0.1, 0.4))))
    if kind == "received":
        return dict(kind=kind, maps=_log(rng, 4, 32), rows=2 * rng.randint(8, 32), cols=2 * rng.randint(8, 32))
    if kind == "attention":
        b = _log(rng, 1, 8)
        lens = [_log(rng, 64, 4096 if b <= 4 else 1500) for _ in range(b)]
        return dict(kind=kind, shape=rng.choice(["llava", "qwen"]), lens=_join(lens), active=rng.choice([30, 60, 100]))
    if kind == "prefill":
        b = _log(rng, 1, 8)
        most = 3600 // b
        text = [_log(rng, 16, min(512, most // 2)) for _ in range(b)]
        vis = [_log(rng, 32, most - t) for t in text]
        return dict(kind=kind, shape=rng.choice(["llava", "llava", "qwen"]), layers=2, vis=_join(vis), text=_join(text),
                    skip=rng.choice([0, 25, 50]))
    if kind == "adaptive":
        return dict(kind=kind, shape="llava", layers=4, vis=_log(rng, 48, 640), text=_log(rng, 32, 256),
                    device_plan=rng.choice([0, 1]))
    if kind == "decode":
        shape = rng.choice(["llava", "qwen"])
        b = _log(rng, 1, 64 if shape == "qwen" else 16)
        return dict(kind=kind, shape=shape, layers=4, pos=_join([_log(rng, 100, 2047) for _ in range(b)]), max_len=2048)
    return dict(kind=kind, layers=12, tiles=_join([1] * rng.choice([1, 1, 2])), text="%d" % _log(rng, 32, 256),
                keep=rng.randint(32, 192), skip=rng.choice([0, 50, 90]))


# ---- inputs -----------------------------------------------------------------------------------
def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _randn(shape, g, std=1.0, dtype=torch.float32):
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype).mul_(std)


def _layer(cfg, seed, l):
    """Layer l's weights: N(0, 0.02^2), norm gains 1 + 0.2 N(0, 1)."""
    g = _gen(seed, 100 + l)
    d, f = cfg["d_model"], cfg["d_ffn"]
    q, kv = cfg["n_heads"] * cfg["head_dim"], cfg["n_kv_heads"] * cfg["head_dim"]
    m = lambda o, i: _randn((o, i), g, 0.02, BF16)  # noqa: E731
    gain = lambda: (1 + _randn(d, g, 0.2)).to(BF16)  # noqa: E731
    return dict(attn_norm=gain(), wq=m(q, d), wk=m(kv, d), wv=m(kv, d), wo=m(d, q), ffn_norm=gain(),
                w_gate=m(f, d), w_up=m(f, d), w_down=m(d, f))


def _ends(cfg, seed):
    """Final norm, LM head (std 0.24: vocabulary distributions as peaked as a trained model's), projector."""
    g = _gen(seed, 1)
    d = cfg["d_model"]
    w = dict(final_norm=(1 + _randn(d, g, 0.2)).to(BF16), lm_head=_randn((cfg["vocab"], d), g, 0.24, BF16))
    if cfg["d_proj"]:
        dv, dp = cfg["d_vis"], cfg["d_proj"]
        w.update(proj_w1=_randn((dp, dv), g, dv ** -0.5, BF16), proj_b1=_randn(dp, g, 0.1, BF16),
                 proj_w2=_randn((d, dp), g, dp ** -0.5, BF16), proj_b2=_randn(d, g, 0.1, BF16))
    return w


def _cfg(case):
    if case["kind"] == "step":
        return dict(SHAPES["llava"], n_layers=case["layers"], d_vis=1024, d_proj=4096)
    return dict(SHAPES[case["shape"]], n_layers=case["layers"])


def _model(cfg, seed):
    w = _ends(cfg, seed)
    w["layers"] = [_layer(cfg, seed, l) for l in range(cfg["n_layers"])]
    return N.SpdModel(cfg, w)


def _features(seed, tiles, n, d, cls, layers=2):
    """Tapped layers' features: four planted groups in bands of the patch order, noise U(0.5, 3) a token."""
    z = torch.div(2 * torch.arange(n, device="cuda") * 4 + n, 2 * n, rounding_mode="floor") % 4
    out = []
    for l in range(layers):
        g = _gen(seed, 10 + l)
        f = _randn((tiles, n + cls, d), g)
        mu = _randn((tiles, 4, d), g, 4.0)
        sigma = 0.5 + 2.5 * torch.rand((tiles, n, 1), generator=g, device="cuda")
        f[:, cls:] *= sigma
        f[:, cls:] += mu[:, z]
        out.append(f)
    return out


def _attention_rows(seed, tiles, heads, n, cls):
    """[CLS] rows (or received attention): softmax of N(0, 2^2) logits, a salient quarter raised by 2."""
    g = _gen(seed, 20)
    z = _randn((tiles, heads, n + cls), g, 2.0)
    z[:, :, cls:] += 2.0 * (torch.rand((tiles, 1, n), generator=g, device="cuda") < 0.25)
    return torch.softmax(z, -1)


def _mask(seed, layers, visual, skip):
    """Skip bits [layers][tokens]: `skip` % of the visual tokens enter skip mode (in the first half of the
    layers) and keep one target, attention for most layers and the FFN for one in six."""
    if not skip:
        return None
    r = np.random.default_rng(seed)
    target = np.where(np.arange(layers) % 6 == 2, 2, 1).astype(np.uint8)
    admit = np.where(visual & (r.random(len(visual)) < skip / 100), r.integers(0, max(1, layers // 2), len(visual)), layers)
    mask = np.zeros((layers, len(visual)), np.uint8)
    for l in range(layers):
        on = admit <= l
        mask[l, on] = target[admit[on]]
    if layers == 2:  # too few layers for a plan: targets drawn a token at a time
        both = np.where(r.random(len(visual)) < 1 / 6, 2, 1).astype(np.uint8)
        mask[:] = np.where(admit[None] < layers, both[None], 0)
    return mask


def _sequences(case):
    """(cu_seqlens, which tokens are visual) of packed [visual; text] requests."""
    cu, vis = [0], []
    for v, t in zip(_ints(str(case["vis"])), _ints(str(case["text"]))):
        cu.append(cu[-1] + v + t)
        vis += [True] * v + [False] * t
    return np.array(cu, np.int32), np.array(vis)


def _zeros(n_bytes):
    return torch.zeros(n_bytes, dtype=torch.uint8, device="cuda")


def _cache(case, cfg, seed, l):
    """Layer l's cache rows [seq][max_len][K | V] as a prefill leaves them (zeros past each context)."""
    pos = _ints(case["pos"])
    c = _randn((len(pos), case["max_len"], 2 * cfg["n_kv_heads"] * cfg["head_dim"]), _gen(seed, 1000 + l), 1.0, BF16)
    live = torch.arange(case["max_len"], device="cuda")[None] < torch.tensor(pos, device="cuda")[:, None]
    return c.mul_(live[:, :, None])


def prepare(case, seed):
    k = case["kind"]
    g = _gen(seed, 2)
    if k == "linear":
        m, n, kk = case["m"], case["n"], case["k"]
        return dict(case=case, x=_randn((m, kk), g, 1.0, BF16), w=_randn((n, kk), g, kk ** -0.5, BF16),
                    bias=_randn(n, g, 0.1, BF16), ws=_zeros(N.spd_linear_workspace_size(m, n)),
                    out=torch.empty(m, n, device="cuda", dtype=torch.float32 if case["epi"] == "f32" else BF16))
    if k == "prune":
        cls = 1 - case["form"]
        t, n = case["tiles"], case["n"]
        cfg = N.prune_cfg(t, n + cls, case["d"], 2, 1, case["heads"], case["keep"], has_cls=bool(cls), attn_form=case["form"])
        e = lambda dt, w=n: torch.empty(t, w, dtype=dt, device="cuda")  # noqa: E731
        return dict(case=case, cfg=cfg, feats=_features(seed, t, n, case["d"], cls),
                    attn=_attention_rows(seed, t, case["heads"], n, cls), keep=e(torch.int32, case["keep"]),
                    kind=e(torch.uint8), cluster=e(torch.int8), scores=e(torch.float32),
                    ws=_zeros(N.spd_prune_workspace_size(cfg)))
    if k == "received":
        n = case["rows"] * case["cols"]
        maps = torch.empty(case["maps"], n, n, device="cuda")
        for i in range(case["maps"]):  # a softmax row a query; a few columns draw most of the attention
            maps[i] = torch.softmax(_randn((n, n), g) + _randn((1, n), g, 2.0), -1)
        start, members = _merger(case)
        return dict(case=case, maps=maps, start=start, members=members,
                    out=torch.empty(case["maps"], n // 4, device="cuda"),
                    ws=_zeros(N.spd_received_attention_workspace_size(case["maps"], n, n)))
    if k == "attention":
        c = SHAPES[case["shape"]]
        q, kv, pos, q_cu, cu = _attention_inputs(case, seed)
        return dict(case=case, c=c, q=q, kv=kv, pos=pos.int().contiguous(), q_cu=q_cu, cu=cu, o=torch.empty_like(q),
                    ws=_zeros(N.spd_attention_workspace_size(len(q), len(cu) - 1)))
    cfg = _cfg(case)
    d = cfg["d_model"]
    model = _model(cfg, seed)
    if k == "step":
        tiles, text = _ints(case["tiles"]), _step_text(case)
        pipe = SpiderPrefill(model, n_patch=576, has_cls=True, d_vis=1024, n_feat_layers=2, final_layer=1,
                             n_heads_vis=16, attn_form=0, keep=case["keep"], tiles_per_req=tiles, text_lens=text)
        return dict(case=case, pipe=pipe, feats=_features(seed, sum(tiles), 576, 1024, 1),
                    attn=_attention_rows(seed, sum(tiles), 16, 576, 1), text=_randn((sum(text), d), g, 1.0, BF16),
                    mask=_mask(seed, case["layers"], pipe.token_is_visual, case["skip"]))
    if k == "decode":
        pos = _ints(case["pos"])
        cache = torch.stack([_cache(case, cfg, seed, l) for l in range(cfg["n_layers"])])
        return dict(case=case, model=model, x=_randn((len(pos), d), g, 1.0, BF16), pos=np.array(pos, np.int32), cache=cache,
                    logits=torch.empty(len(pos), cfg["vocab"], device="cuda"),
                    ws=_zeros(N.spd_decode_workspace_size(model, len(pos))))
    cu, vis = _sequences(case)
    t, b = int(cu[-1]), len(cu) - 1
    size = N.spd_prefill_workspace_size if k == "prefill" else N.spd_prefill_adaptive_workspace_size
    return dict(case=case, model=model, x=_randn((t, d), g, 1.0, BF16), cu=cu, vis=vis, t=t,
                mask=_mask(seed, case["layers"], vis, case.get("skip", 0)), h=torch.empty(t, d, device="cuda"),
                logits=torch.empty(b, cfg["vocab"], device="cuda"), ws=_zeros(size(model, t, b)))


def _merger(case):
    """Groups of the 2 x 2 merger over a rows x cols patch grid, as CSR device arrays."""
    i = torch.arange(case["rows"] * case["cols"], device="cuda").view(case["rows"] // 2, 2, case["cols"] // 2, 2)
    members = i.permute(0, 2, 1, 3).reshape(-1).int().contiguous()
    return torch.arange(0, len(members) + 1, 4, device="cuda").int(), members


def _attention_inputs(case, seed):
    c = SHAPES[case["shape"]]
    g, r = _gen(seed, 3), np.random.default_rng(seed)
    lens = _ints(case["lens"])
    at = [np.sort(r.choice(n, max(1, n * case["active"] // 100), replace=False)) for n in lens]
    q_cu = np.cumsum([0] + [len(a) for a in at]).astype(np.int32)
    cu = np.cumsum([0] + lens).astype(np.int32)
    q = _randn((int(q_cu[-1]), c["n_heads"] * c["head_dim"]), g, 1.0, BF16)
    kv = _randn((int(cu[-1]), 2 * c["n_kv_heads"] * c["head_dim"]), g, 1.0, BF16)
    return q, kv, torch.from_numpy(np.concatenate(at)).cuda(), q_cu, cu


def _step_text(case):
    return _ints(case["text"]) * len(_ints(case["tiles"]))


def _policy(case):
    """Layer 0 admits the tokens whose online score is high, layer 1 all others (its SLC term alone reaches T_skip)."""
    n = case["layers"]
    slc = np.full(n, 0.5, np.float32)
    slc[1] = 8.0
    return dict(slc_norm=slc, layer_target=np.array([2] + [1] * (n - 1), np.uint8), t_skip=1.9, w1=3.0, w2=1.0, window=n // 2)


def run(s):
    case = s["case"]
    k = case["kind"]
    if k == "linear":
        N.spd_linear(s["x"], case["m"], case["k"], s["w"], case["n"], EPILOGUES[case["epi"]], s["out"], case["n"], s["ws"],
                     bias=s["bias"])
        return s["out"]
    if k == "prune":
        N.spd_prune(s["cfg"], s["feats"], s["attn"], s["keep"], s["kind"], s["cluster"], s["scores"], ws=s["ws"])
        return dict(keep=s["keep"], kind=s["kind"], cluster=s["cluster"], scores=s["scores"])
    if k == "received":
        N.spd_received_attention(s["maps"], s["out"], s["ws"], s["start"], s["members"])
        return s["out"]
    if k == "attention":
        c = s["c"]
        N.spd_attention(s["q"], s["pos"], s["q_cu"], s["kv"], s["cu"], c["n_heads"], c["n_kv_heads"], c["head_dim"], s["o"], s["ws"])
        return s["o"]
    if k == "step":
        logits = s["pipe"].run(s["feats"], s["attn"], s["text"], s["mask"])
        return dict(logits=logits, h=s["pipe"].h, keep=s["pipe"].keep_idx)
    if k == "decode":
        N.spd_decode(s["model"], s["x"], s["pos"], s["cache"], case["max_len"], s["logits"], s["ws"])
        return dict(logits=s["logits"], cache=s["cache"])
    if k == "prefill":
        N.spd_prefill(s["model"], s["x"], s["t"], s["cu"], s["mask"], s["h"], s["logits"], s["ws"])
        return dict(h=s["h"], logits=s["logits"])
    p = _policy(case)
    admit = N.spd_prefill_adaptive(s["model"], s["x"], s["t"], s["cu"], s["vis"], p["slc_norm"], p["layer_target"], p["t_skip"],
                                   p["w1"], p["w2"], p["window"], s["h"], s["logits"], s["ws"], device_plan=case["device_plan"])
    return dict(h=s["h"], logits=s["logits"], admit=admit)


# ---- work and tolerances ------------------------------------------------------------------------
def _layer_params(cfg):
    d, q, kv = cfg["d_model"], cfg["n_heads"] * cfg["head_dim"], cfg["n_kv_heads"] * cfg["head_dim"]
    return d * (q + 2 * kv), d * q, 3 * d * cfg["d_ffn"]


def _prefill_work(cfg, lens, visual, skip, heads_rows):
    """Bytes and flops of the decoder over sequences of `lens` tokens, `skip` % of the `visual` tokens passing by a
    sub-layer (five in six the attention): weights once, input and residual stream once, logits once."""
    t, d, h = sum(lens), cfg["d_model"], cfg["n_heads"] * cfg["head_dim"]
    qkv, o, ffn = _layer_params(cfg)
    q_share = 1 - visual / t * skip / 100 * 5 / 6
    f_share = 1 - visual / t * skip / 100 / 6
    ctx = sum(n * (n + 1) / 2 for n in lens)
    kv = d * 2 * cfg["n_kv_heads"] * cfg["head_dim"]
    flops = cfg["n_layers"] * (2 * t * (kv + q_share * (qkv - kv + o) + f_share * ffn) + 4 * h * ctx * q_share)
    flops += 2 * heads_rows * cfg["vocab"] * d
    return {"bytes": 2 * cfg["n_layers"] * (qkv + o + ffn) + 2 * cfg["vocab"] * d + 6 * t * d + 4 * heads_rows * cfg["vocab"],
            "flops": flops}


def work(case):
    k = case["kind"]
    if k == "linear":
        m, n, kk = case["m"], case["n"], case["k"]
        return {"bytes": 2 * (m * kk + n * kk + n) + (4 if case["epi"] == "f32" else 2) * m * n, "flops": 2 * m * n * kk}
    if k == "prune":
        cls, t, n, d = 1 - case["form"], case["tiles"], case["n"], case["d"]
        anchors = int(case["keep"] * 0.7 + 0.5)
        return {"bytes": t * (8 * (n + cls) * d + 4 * case["heads"] * (n + cls) + 4 * case["keep"] + 6 * n),
                "flops": t * (n - anchors) * d * (2 * anchors + 2 * 4 * 3 + 16)}
    if k == "received":
        n = case["rows"] * case["cols"]
        return {"bytes": 4 * case["maps"] * (n * n + n // 4), "flops": case["maps"] * n * n}
    if k == "attention":
        c, lens = SHAPES[case["shape"]], _ints(case["lens"])
        nq = sum(max(1, n * case["active"] // 100) for n in lens)
        ctx = sum(n * (n + 1) / 2 for n in lens) * case["active"] / 100
        return {"bytes": 4 * c["head_dim"] * (nq * c["n_heads"] + sum(lens) * c["n_kv_heads"]),
                "flops": 4 * c["head_dim"] * c["n_heads"] * ctx}
    cfg = _cfg(case)
    if k == "decode":
        pos = _ints(case["pos"])
        qkv, o, ffn = _layer_params(cfg)
        rows = sum(p + 1 for p in pos)
        params = cfg["n_layers"] * (qkv + o + ffn) + cfg["vocab"] * cfg["d_model"]
        kv, q = cfg["n_kv_heads"] * cfg["head_dim"], cfg["n_heads"] * cfg["head_dim"]
        return {"bytes": 2 * params + 4 * cfg["n_layers"] * rows * kv + len(pos) * (2 * cfg["d_model"] + 4 * cfg["vocab"]),
                "flops": 2 * len(pos) * params + 4 * cfg["n_layers"] * rows * q}
    if k == "step":
        tiles, text = _ints(case["tiles"]), _step_text(case)
        nv = sum(tiles) * case["keep"]
        p = work(dict(kind="prune", form=0, tiles=sum(tiles), n=576, d=1024, heads=16, keep=case["keep"]))
        w = _prefill_work(cfg, [v * case["keep"] + t for v, t in zip(tiles, text)], nv, 0.75 * case["skip"], len(tiles))
        proj = 1024 * 4096 + 4096 * 4096
        return {"bytes": p["bytes"] + w["bytes"] + 2 * proj, "flops": p["flops"] + w["flops"] + 2 * nv * proj}
    vis, text = _ints(str(case["vis"])), _ints(str(case["text"]))
    w = _prefill_work(cfg, [v + t for v, t in zip(vis, text)], sum(vis), case.get("skip", 50), len(vis))
    if k == "adaptive":  # the logit lens of the candidates in the two decision layers
        w["flops"] += 2 * (case["layers"] // 2) * sum(vis) * cfg["vocab"] * cfg["d_model"]
    return w


def tolerance(case):
    """Largest differences between correct implementations of the same precision: fp32 sums in another order for the
    scores of MSV-Prune and the received attention; bf16 roundings of activations that fall differently
    elsewhere, which travel further through the whole models."""
    k = case["kind"]
    if k == "received":
        return {"rel": 2e-6, "max": 1e-5}
    if k == "prune":  # a selection cut or a cluster border within fp32 rounding of a tie may fall either way
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.01}
    if k == "linear":
        return {"rel": 2e-5, "max": 2e-4} if case["epi"] == "f32" else {"rel": 7e-3, "max": 0.05}
    if k == "attention":
        return {"rel": 8e-3, "max": 0.05}
    if k == "step":
        return {"rel": 0.03, "max": 0.3, "differ": 0.01}
    if k == "prefill":
        return {"rel": 0.01, "max": 0.2}
    return {"rel": 0.025 if case["layers"] > 8 or k == "adaptive" else 0.01, "max": 0.2, "differ": 0.01}


# ---- the same mathematics in 64 bits ------------------------------------------------------------
F64 = torch.float64


def _norm64(h, gain, eps):
    return h * torch.rsqrt((h * h).mean(-1, keepdim=True) + eps) * gain.to(F64)


def _rope64(x, pos, cfg):
    hd = cfg["head_dim"]
    x = x.view(x.shape[0], -1, hd)
    half = hd // 2
    a = pos.to(F64)[:, None, None] * cfg["rope_theta"] ** (-2.0 * torch.arange(half, device="cuda", dtype=F64) / hd)
    c, s = a.cos(), a.sin()
    lo, hi = x[..., :half], x[..., half:]
    return torch.cat([lo * c - hi * s, hi * c + lo * s], -1)


def _attend64(q, k, v, q_pos, groups):
    """q [nq][H][hd] against k, v [nk][Hkv][hd]: keys at positions 0 .. q_pos of the same sequence."""
    out = torch.empty_like(q)
    see = torch.arange(k.shape[0], device="cuda")[None] <= q_pos[:, None]
    for h in range(q.shape[1]):
        z = q[:, h] @ k[:, h // groups].T / math.sqrt(q.shape[2])
        out[:, h] = torch.softmax(z.masked_fill(~see, -math.inf), -1) @ v[:, h // groups]
    return out


def _layer64(cfg, w, h, pos, skip, attend):
    """One decoder layer in place; skip [tokens] bits; attend(q of the active rows, k, v, active rows)."""
    xa = _norm64(h, w["attn_norm"], cfg["rms_eps"])
    t, hd = len(h), cfg["head_dim"]
    k = _rope64(xa @ w["wk"].to(F64).T, pos, cfg)
    v = (xa @ w["wv"].to(F64).T).view(t, -1, hd)
    act = (skip & 1).eq(0).nonzero()[:, 0]
    if len(act):
        q = _rope64(xa[act] @ w["wq"].to(F64).T, pos[act], cfg)
        h[act] += attend(q, k, v, act).reshape(len(act), -1) @ w["wo"].to(F64).T
    act = (skip & 2).eq(0).nonzero()[:, 0]
    if len(act):
        y = _norm64(h[act], w["ffn_norm"], cfg["rms_eps"])
        u = torch.nn.functional.silu(y @ w["w_gate"].to(F64).T) * (y @ w["w_up"].to(F64).T)
        h[act] += u @ w["w_down"].to(F64).T


def _logits64(cfg, ends, h):
    z = _norm64(h, ends["final_norm"], cfg["rms_eps"])
    return torch.cat([z @ w.to(F64).T for w in ends["lm_head"].split(16384)], -1)


def _prefill64(cfg, seed, x, cu, mask, admit=None):
    """(h, logits) of packed sequences; admit(l, h, ends) may give layer l's skip bits instead of the mask."""
    h = x.to(F64)
    cu = [int(c) for c in cu]
    pos = torch.cat([torch.arange(b - a, device="cuda") for a, b in zip(cu, cu[1:])])
    groups = cfg["n_heads"] // cfg["n_kv_heads"]
    ends = _ends(cfg, seed)

    def attend(q, k, v, act):
        out = torch.empty_like(q)
        for a, b in zip(cu, cu[1:]):
            rows = ((act >= a) & (act < b)).nonzero()[:, 0]
            if len(rows):
                out[rows] = _attend64(q[rows], k[a:b], v[a:b], pos[act[rows]], groups)
        return out

    for l in range(cfg["n_layers"]):
        skip = admit(l, h, ends) if admit else torch.zeros(len(h), device="cuda", dtype=torch.int64) if mask is None \
            else torch.from_numpy(mask[l].astype(np.int64)).cuda()
        _layer64(cfg, _layer(cfg, seed, l), h, pos, skip, attend)
    return h, _logits64(cfg, ends, h[torch.tensor(cu[1:], device="cuda") - 1])


def _adaptive64(case, cfg, seed, x, cu, vis):
    p, t = _policy(case), len(vis)
    seen = torch.from_numpy(vis).cuda()
    text = ~seen
    at = torch.full((t,), -1, device="cuda", dtype=torch.int64)
    score = torch.zeros(t, device="cuda", dtype=F64)

    def admit(l, h, ends):
        if l < p["window"]:
            cand = (seen & (at < 0)).nonzero()[:, 0]
            if len(cand):
                lp = torch.log_softmax(_logits64(cfg, ends, h[cand]), -1)
                e = -(lp.exp() * lp).sum(-1) / math.log(cfg["vocab"])
                q = h[text].mean(0)
                f = 0.5 + 0.5 * (h[cand] @ q) / (h[cand].norm(dim=-1) * q.norm())
                score[cand] += p["w1"] * (1 - e - f).clamp(min=0) + p["w2"] * float(p["slc_norm"][l])
                at[cand[score[cand] >= p["t_skip"]]] = l
        tgt = torch.from_numpy(p["layer_target"].astype(np.int64)).cuda()
        return torch.where(at >= 0, tgt[at.clamp(min=0)], 0)

    h, logits = _prefill64(cfg, seed, x, cu, None, admit)
    return dict(h=h, logits=logits, admit=at.to(torch.int16).cpu().numpy())


def _quotas(sizes, n_cmp):
    """Eq. 2 in whole numbers: max(1, round(n_cmp size / total)), mended to add up to n_cmp."""
    total, ids = sum(sizes), range(len(sizes))
    live = [k for k in ids if sizes[k]]
    if n_cmp < len(live):
        first = sorted(live, key=lambda k: (-sizes[k], k))[:max(n_cmp, 0)]
        return [int(k in first) for k in ids]
    q = [min(sizes[k], max(1, (2 * n_cmp * sizes[k] + total) // (2 * total))) if sizes[k] else 0 for k in ids]
    rest = [n_cmp * s % total for s in sizes]
    while sum(q) < n_cmp:
        for k in sorted(ids, key=lambda k: (-rest[k], k)):
            if sum(q) < n_cmp and q[k] < sizes[k]:
                q[k] += 1
    while sum(q) > n_cmp:
        for k in sorted(ids, key=lambda k: (rest[k], -k)):
            if sum(q) > n_cmp and q[k] > 1:
                q[k] -= 1
    return q


def _prune64(feats, attn, keep, cls, n_k=4, iters=10):
    """(kind, cluster, scores, kept indices) of one tile: feats [2][n][d] with the last layer final."""
    n = feats[0].shape[0]
    n_anc = int(math.floor(keep * 0.7 + 0.5))
    order = torch.sort(-attn.to(F64)[:, cls:].mean(0), stable=True).indices
    kind = torch.zeros(n, dtype=torch.uint8, device="cuda")
    kind[order[:n_anc]] = 1
    rest = kind.eq(0).nonzero()[:, 0]
    scores = torch.full((n,), math.inf, dtype=F64, device="cuda")
    cluster = torch.full((n,), -1, dtype=torch.int8, device="cuda")
    m = len(rest)
    if m:
        unit = [f / f.norm(dim=-1, keepdim=True) for f in feats]
        a = (unit[1][rest] @ unit[1][kind.eq(1)].T).amax(-1) if n_anc else torch.zeros(m, dtype=F64, device="cuda")
        x = feats[1][rest]
        c = x[[k * m // n_k for k in range(n_k)]].clone()
        old = None
        for _ in range(iters):
            got = torch.stack([((x - c[k]) ** 2).sum(-1) for k in range(n_k)], -1).argmin(-1)
            if old is not None and torch.equal(got, old):
                break
            old = got
            for k in range(n_k):
                if (got == k).any():
                    c[k] = x[got == k].mean(0)
        sizes = [int((old == k).sum()) for k in range(n_k)]
        for k, q in enumerate(_quotas(sizes, keep - n_anc)):
            at = (old == k).nonzero()[:, 0]
            s = 2 * a[at]
            if sizes[k] > 1:
                s = a[at] + (a[at].sum() - a[at]) / (sizes[k] - 1)
                for f in unit:
                    u = f[rest[at]]
                    s = s + (u * (u.sum(0) - u)).sum(-1) / (sizes[k] - 1)
            scores[rest[at]] = s
            cluster[rest[at]] = k
            kind[rest[at[torch.sort(s, stable=True).indices[:q]]]] = 2
    return kind, cluster, scores, kind.nonzero()[:, 0].int()


def _prune_all64(case, seed, keep):
    cls, t, n = 1 - case["form"], case["tiles"], case["n"]
    feats = _features(seed, t, n, case["d"], cls)
    attn = _attention_rows(seed, t, case["heads"], n, cls)
    got = [_prune64([f[i, cls:].to(F64) for f in feats], attn[i], keep, cls) for i in range(t)]
    return [torch.stack(v) for v in zip(*got)], feats


def exact(case, seed):
    k = case["kind"]
    if k == "linear":
        g = _gen(seed, 2)
        m, n, kk = case["m"], case["n"], case["k"]
        x, w, b = _randn((m, kk), g, 1.0, BF16), _randn((n, kk), g, kk ** -0.5, BF16), _randn(n, g, 0.1, BF16)
        y = x.to(F64) @ w.to(F64).T
        if case["epi"] in ("bias", "gelu"):
            y = y + b.to(F64)
        return 0.5 * y * (1 + torch.erf(y / math.sqrt(2.0))) if case["epi"] == "gelu" else y
    if k == "prune":
        (kind, cluster, scores, keep), _ = _prune_all64(case, seed, case["keep"])
        return dict(keep=keep, kind=kind, cluster=cluster, scores=scores)
    if k == "received":
        n = case["rows"] * case["cols"]
        g = _gen(seed, 2)
        maps = []
        for _ in range(case["maps"]):
            maps.append(torch.softmax(_randn((n, n), g) + _randn((1, n), g, 2.0), -1).to(F64).mean(0))
        return torch.stack(maps)[:, _merger(case)[1].long()].view(case["maps"], -1, 4).sum(-1)
    if k == "attention":
        c = SHAPES[case["shape"]]
        q, kv, pos, q_cu, cu = _attention_inputs(case, seed)
        q, out = q.to(F64).view(len(q), -1, c["head_dim"]), []
        for i in range(len(cu) - 1):
            s, e, a, b = int(cu[i]), int(cu[i + 1]), int(q_cu[i]), int(q_cu[i + 1])
            kk, v = kv[s:e].to(F64).view(e - s, 2, -1, c["head_dim"]).unbind(1)
            out.append(_attend64(q[a:b], kk, v, pos[a:b], c["n_heads"] // c["n_kv_heads"]).reshape(b - a, -1))
        return torch.cat(out)
    cfg = _cfg(case)
    g = _gen(seed, 2)
    d = cfg["d_model"]
    if k == "step":
        tiles, text = _ints(case["tiles"]), _step_text(case)
        p = dict(form=0, tiles=sum(tiles), n=576, d=1024, heads=16)
        (_, _, _, keep), feats = _prune_all64(p, seed, case["keep"])
        words = _randn((sum(text), d), g, 1.0, BF16).to(F64)
        e = _ends(cfg, seed)
        v = torch.cat([feats[1][i, 1 + keep[i].long()].to(F64) for i in range(sum(tiles))])
        v = torch.nn.functional.gelu(v @ e["proj_w1"].to(F64).T + e["proj_b1"].to(F64))
        v = v @ e["proj_w2"].to(F64).T + e["proj_b2"].to(F64)
        rows, cu, vis, at_v, at_t = [], [0], [], 0, 0
        for nt, t in zip(tiles, text):
            nv = nt * case["keep"]
            rows += [v[at_v:at_v + nv], words[at_t:at_t + t]]
            vis += [True] * nv + [False] * t
            at_v, at_t = at_v + nv, at_t + t
            cu.append(cu[-1] + nv + t)
        h, logits = _prefill64(cfg, seed, torch.cat(rows), cu, _mask(seed, case["layers"], np.array(vis), case["skip"]))
        return dict(logits=logits, h=h, keep=keep)
    if k == "decode":
        pos = torch.tensor(_ints(case["pos"]), device="cuda")
        h = _randn((len(pos), d), g, 1.0, BF16).to(F64)
        caches, hd = [], cfg["head_dim"]
        for l in range(cfg["n_layers"]):
            cache = _cache(case, cfg, seed, l)
            new = cache.to(F64) if len(pos) * case["max_len"] <= 8192 else None  # the rest of the cache is unchanged

            def attend(q, kk, v, act):
                out = torch.empty_like(q)
                for b, p in enumerate(pos.tolist()):
                    old_k, old_v = cache[b, :p].to(F64).view(p, 2, -1, hd).unbind(1)
                    out[b] = _attend64(q[b:b + 1], torch.cat([old_k, kk[b:b + 1]]), torch.cat([old_v, v[b:b + 1]]),
                                       pos[b:b + 1], cfg["n_heads"] // cfg["n_kv_heads"])[0]
                    if new is not None:
                        new[b, p] = torch.stack([kk[b], v[b]]).reshape(-1)
                return out

            _layer64(cfg, _layer(cfg, seed, l), h, pos, torch.zeros_like(pos), attend)
            caches.append(new)
        return dict(logits=_logits64(cfg, _ends(cfg, seed), h), cache=torch.stack(caches) if caches[0] is not None else None)
    cu, vis = _sequences(case)
    x = _randn((int(cu[-1]), d), g, 1.0, BF16)
    if k == "adaptive":
        return _adaptive64(case, cfg, seed, x, cu, vis)
    h, logits = _prefill64(cfg, seed, x, cu, _mask(seed, case["layers"], vis, case["skip"]))
    return dict(h=h, logits=logits)
