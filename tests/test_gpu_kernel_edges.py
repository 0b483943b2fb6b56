"""Kernels at the sizes where they can go wrong: edges of tiles and groups, remainders, both ends of
each range, against the oracle's definitions."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import decoder as od  # noqa: E402
from paper_2609_34977_gb300 import _native as N  # noqa: E402
from paper_2609_34977_gb300 import synth  # noqa: E402
from oracle import prune as op  # noqa: E402
from tests.gpu_util import assert_prune_parity, bf16_np, conditioned_vision, gpu_prune, rowwise_rel  # noqa: E402

pytestmark = pytest.mark.gpu


def _bf16(seed, *shape):
    g = torch.Generator().manual_seed(seed)
    return torch.randn(*shape, generator=g).to(torch.bfloat16)


@pytest.mark.parametrize("heads,kv_heads,head_dim,pos,offset", [
    (4, 4, 64, [0, 15, 16], 0),                     # one head a K/V head; key groups of 16 not full
    (4, 4, 128, [17, 63, 64], 4),                   # a cache 8 bytes off a 16-byte boundary
    (28, 4, 128, [65, 127, 128, 129, 500, 7], 0),   # seven heads a K/V head, shares of unequal length
    (18, 2, 64, [31, 260, 511], 0),                 # nine heads a K/V head: a second chunk of one head
    (16, 1, 128, [0, 1, 300, 511, 48, 47, 33, 2], 0),  # two full chunks; clusters of eight CTAs
    (32, 32, 64, list(range(0, 500, 50)), 0),          # more CTAs than two an SM
])
def test_decode_attention_edges(heads, kv_heads, head_dim, pos, offset):
    # one decoder layer over a given cache: logits and the appended K/V rows. Tolerance: every rounding of
    # the path is one bf16 unit (2^-9), as in the prefill's parity tests (2e-2 normwise a row).
    cfg = dict(synth.TINY_DECODER, n_layers=1, n_heads=heads, n_kv_heads=kv_heads, head_dim=head_dim, d_ffn=256)
    B, max_len, D, kvd = len(pos), 512, cfg["d_model"], kv_heads * head_dim
    w = synth.decoder_weights(3, cfg, std=0.05)
    wd = {k: v.cuda() for k, v in w.items() if k != "layers"}
    wd["layers"] = [{k: v.cuda() for k, v in lw.items()} for lw in w["layers"]]
    model = N.SpdModel(cfg, wd)
    c = _bf16(5, B, max_len, 2 * kvd)
    for b, p in enumerate(pos):
        c[b, p:] = 0
    flat = torch.zeros(c.numel() + 8, dtype=torch.bfloat16, device="cuda")
    cache = flat[offset:offset + c.numel()]
    cache.copy_(c.reshape(-1).cuda())
    x = _bf16(6, B, D)
    out = torch.full((B, cfg["vocab"]), float("nan"), device="cuda")
    ws = torch.zeros(N.spd_decode_workspace_size(model, B), dtype=torch.uint8, device="cuda")
    N.spd_decode(model, x.cuda(), np.array(pos), cache, max_len, out, ws)
    torch.cuda.synchronize()
    assert N.spd_workspace_status(ws) == 0
    om = od.model_from_torch(w, cfg)
    lw, rnd = om["layers"][0], od.bf16_round
    h, p = bf16_np(x).astype(np.float64), np.array(pos)
    xa = rnd(od.rmsnorm(h, lw["attn_norm"], cfg["rms_eps"]))
    q, k = (rnd(od.rope(xa @ lw[n].T, p, nh, head_dim, cfg["rope_theta"])) for n, nh in (("wq", heads), ("wk", kv_heads)))
    v = rnd(xa @ lw["wv"].T)
    o = np.zeros((B, heads * head_dim))
    for b in range(B):
        kv = bf16_np(c[b, :p[b]]).astype(np.float64)
        ka, va = np.concatenate([kv[:, :kvd], k[b:b + 1]]), np.concatenate([kv[:, kvd:], v[b:b + 1]])
        o[b] = od.causal_attention(q[b:b + 1], ka, va, p[b:b + 1], np.arange(p[b] + 1), heads, kv_heads, head_dim)
    h += rnd(o) @ lw["wo"].T
    y = rnd(od.rmsnorm(h, lw["ffn_norm"], cfg["rms_eps"]))
    h += rnd(od.silu(y @ lw["w_gate"].T) * (y @ lw["w_up"].T)) @ lw["w_down"].T
    z = rnd(od.rmsnorm(h, om["final_norm"], cfg["rms_eps"]))
    assert rowwise_rel(out.cpu().numpy(), z @ om["lm_head"].T) < 2e-2
    got = bf16_np(cache).reshape(B, max_len, 2 * kvd)
    for b in range(B):
        assert rowwise_rel(got[b, p[b]:p[b] + 1], np.concatenate([k[b:b + 1], v[b:b + 1]], 1)) < 2e-2
        assert not got[b, p[b] + 1:].any()


def test_decode_attention_weights_hold_24_bits():
    # two keys of nearly equal weight (2^-11 apart in one dimension) whose values cancel but for that difference,
    # beside two keys that make the weights uneven and carry no value: the output is about 2^-15 of the weights,
    # so a weight cut to 17 bits shows as tens of percent. Tolerance: the bf16 roundings of q and of the output,
    # as in the other decode tests.
    H, hd, B, max_len = 4, 64, 8, 16
    cfg = dict(synth.TINY_DECODER, n_layers=1)
    w = synth.decoder_weights(5, cfg, std=0.05)
    lw = w["layers"][0]
    for name in ("wk", "wv", "w_down"):
        lw[name].zero_()
    lw["wo"].copy_(64 * torch.eye(H * hd))
    wd = {k: v.cuda() for k, v in w.items() if k != "layers"}
    wd["layers"] = [{k: v.cuda() for k, v in lw.items()}]
    c = torch.zeros(B, max_len, 2, H, hd)
    c[:, 0, 0, :, 1] = 2.0 ** -11
    c[:, 2, 0, :, 0], c[:, 3, 0, :, 0] = 8.0, -8.0
    c[:, 0, 1], c[:, 1, 1] = 256.0, -256.0
    cache = c.to(torch.bfloat16).reshape(B, max_len, -1).cuda()
    x = (_bf16(7, B, H * hd).float() * 1e-3).to(torch.bfloat16)
    out = torch.empty(B, cfg["vocab"], device="cuda")
    model = N.SpdModel(cfg, wd)
    ws = torch.zeros(N.spd_decode_workspace_size(model, B), dtype=torch.uint8, device="cuda")
    N.spd_decode(model, x.cuda(), np.full(B, 4), cache, max_len, out, ws)
    om = od.model_from_torch(w, cfg)
    ow, rnd = om["layers"][0], od.bf16_round
    h = bf16_np(x).astype(np.float64)
    xa = rnd(od.rmsnorm(h, ow["attn_norm"], cfg["rms_eps"]))
    q = rnd(od.rope(xa @ ow["wq"].T, np.full(B, 4), H, hd, cfg["rope_theta"]))
    kv = c.double().numpy().reshape(B, max_len, 2, -1)
    for b in range(B):
        o = od.causal_attention(q[b:b + 1], kv[b, :5, 0], kv[b, :5, 1], np.array([4]), np.arange(5), H, H, hd)
        h[b] += 64 * rnd(o)[0]
    z = rnd(od.rmsnorm(h, om["final_norm"], cfg["rms_eps"]))
    assert rowwise_rel(out.cpu().numpy(), z @ om["lm_head"].T) < 2e-2


# ---- few-token GEMMs: m16n8k16 straight from the weight rows ------------------------------------------
@pytest.mark.parametrize("M", [1, 2, 7, 8, 9, 16, 17])  # one and two sets of token columns, and past them
@pytest.mark.parametrize("K,n", [(256, 1), (512, 40), (2816, 1000), (4096, 128)])
def test_few_token_epilogues(M, K, n):
    # K ranges of one chunk, of unequal shares; output widths that end inside a 16-row half, a 32-row group
    g = torch.Generator().manual_seed(M * K + n)
    X = torch.randn(M, K, generator=g).to(torch.bfloat16)
    W = (torch.randn(n, K, generator=g) * 0.05).to(torch.bfloat16)
    bias = torch.randn(n, generator=g).to(torch.bfloat16)
    acc = bf16_np(X) @ bf16_np(W).T
    ws = torch.zeros(N.spd_linear_workspace_size(M, n), dtype=torch.uint8, device="cuda")
    Xc, Wc, bc = X.cuda(), W.cuda(), bias.cuda()
    ldo = n + 3  # a row stride wider than the row: its padding stays untouched
    for epi, ref, tol in ((N.EPI_F32, acc, 1e-4), (N.EPI_BF16, acc, 2 ** -8), (N.EPI_BIAS_BF16, acc + bf16_np(bias), 2 ** -8),
                          (N.EPI_BIAS_GELU_BF16, od.gelu(acc + bf16_np(bias)), 2 ** -8)):
        # fp32 sums: 1e-4 of the row; bf16 outputs: half a unit (2^-9) and the sums' error below another
        dt = torch.float32 if epi == N.EPI_F32 else torch.bfloat16
        out = torch.full((M, ldo), 7.0, dtype=dt, device="cuda")
        N.spd_linear(Xc, M, K, Wc, n, epi, out, ldo, ws, bias=bc)
        got = out.double().cpu().numpy()
        assert rowwise_rel(got[:, :n], ref) < tol, epi
        assert (got[:, n:] == 7.0).all()
    rows = torch.randperm(M + 3, generator=g)[:M].to(torch.int32)
    h0 = torch.randn(M + 3, n, generator=g)
    h = h0.cuda()
    N.spd_linear(Xc, M, K, Wc, n, N.EPI_ADD_F32, h, n, ws, rows=rows.cuda())
    want = h0.double().numpy()
    want[rows.numpy()] += acc
    assert rowwise_rel(h.cpu().numpy(), want) < 1e-4
    assert N.spd_workspace_status(ws) == 0


@pytest.mark.parametrize("M", [2, 4, 8])
@pytest.mark.parametrize("K", [256, 1024, 4096, 18944])
def test_few_token_sums_are_fp32(M, K):
    # sums of up to eight tokens round like fp32: an output passes about 8 additions and K / 512 more, each
    # half a unit (2^-24) of its sum off at most and, adding up at random, their root of it in all.
    n = 4096
    g = torch.Generator(device="cuda").manual_seed(M + K)
    X = torch.randn(M, K, generator=g, device="cuda").to(torch.bfloat16)
    W = (torch.randn(n, K, generator=g, device="cuda") * K ** -0.5).to(torch.bfloat16)
    ws = torch.zeros(N.spd_linear_workspace_size(M, n), dtype=torch.uint8, device="cuda")
    out = torch.empty(M, n, device="cuda")
    N.spd_linear(X, M, K, W, n, N.EPI_F32, out, n, ws)
    ref = X.double() @ W.double().T
    assert ((out.double() - ref).norm() / ref.norm()).item() < 2.0 ** -24 * (8 + K / 512) ** 0.5
    # infinities stay infinities: one infinite weight
    W[:, 0] = float("inf")
    X[:, 0] = 1.0
    N.spd_linear(X, M, K, W, n, N.EPI_F32, out, n, ws)
    assert torch.isposinf(out).all()


@pytest.mark.parametrize("M", [640, 1000, 1200])  # 48, 64 and 80 pair tiles of 4096 rows for 76 slots
def test_residual_whole_tiles_repeat_exactly(M):
    # between half and all of the slots a residual tile belongs to one work item, which adds each element
    # once: the same bits in every run (80 tiles are more than the slots: split, right within rounding)
    K = n = 4096
    g = torch.Generator().manual_seed(M)
    X = torch.randn(M, K, generator=g).to(torch.bfloat16).cuda()
    W = (torch.randn(n, K, generator=g) * 0.05).to(torch.bfloat16).cuda()
    h0 = torch.randn(M, n, generator=g).cuda()
    ws = torch.zeros(N.spd_linear_workspace_size(M, n), dtype=torch.uint8, device="cuda")
    outs = []
    for _ in range(4):
        h = h0.clone()
        N.spd_linear(X, M, K, W, n, N.EPI_ADD_F32, h, n, ws)
        outs.append(h)
    torch.cuda.synchronize()
    assert N.spd_workspace_status(ws) == 0
    assert rowwise_rel(outs[0].cpu().numpy(), (h0.double() + X.double() @ W.double().T).cpu().numpy()) < 1e-4
    if M < 1200:
        assert all(torch.equal(o, outs[0]) for o in outs)


def test_scratch_cleared_as_a_call_needs_more_of_it():
    # 1250 tokens on 152 SMs: the QKV GEMM leaves 12 tiles over (their sums and counters are cleared), the gate-up
    # GEMM needs more counters, the other layer's GEMMs find all of it clear. The workspace holds garbage before.
    cfg = dict(synth.TINY_DECODER, n_layers=2, d_model=2048, n_heads=32, n_kv_heads=32, head_dim=128, d_ffn=11008)
    w = synth.decoder_weights(4, cfg, device="cuda")
    model = N.SpdModel(cfg, w)
    T = 1250
    x = _bf16(8, T, 2048).cuda()
    cu = np.array([0, 700, T], np.int32)
    got = []
    for fill in (0, 0x7f):
        ws = torch.full((N.spd_prefill_workspace_size(model, T, 2),), fill, dtype=torch.uint8, device="cuda")
        ws[:256] = 0  # the status word
        h, logits = torch.empty(T, 2048, device="cuda"), torch.empty(2, cfg["vocab"], device="cuda")
        N.spd_prefill(model, x, T, cu, None, h, logits, ws)
        torch.cuda.synchronize()
        assert N.spd_workspace_status(ws) == 0
        got.append((h, logits))
    for a, b in zip(*got):  # the same kernels twice: bf16 units that the order of residual sums decides
        assert torch.isfinite(b).all()
        assert rowwise_rel(b.double().cpu().numpy(), a.double().cpu().numpy()) < 2.0 ** -6


# ---- MSV-Prune: K-means over the whole GPU, rankings over several CTAs --------------------------------
def _shuffled_tile(seed0, n, d, keep, **kw):
    # a tile whose planted groups lie scattered over the token order: the seeds fall into any of them, so
    # K-means takes several iterations; first seed with margins above 1e-3 at every decision
    for seed in range(seed0, seed0 + 200):
        v = synth.vision_tiles(seed, 1, n, d, 2, 4, has_cls=False, attn_form=1)
        perm = np.random.default_rng(seed).permutation(n)
        v = dict(feats=[np.ascontiguousarray(f[:, perm]) for f in v["feats"]],
                 attn=np.ascontiguousarray(v["attn"][:, :, perm]))
        res = op.prune(v["feats"], v["attn"], has_cls=False, attn_form=1, final_layer=1, keep=keep, **kw)
        if op.well_conditioned(res[0]):
            return v, res
    raise RuntimeError("no well-conditioned seed found")


@pytest.mark.parametrize("tiles,n,d,keep,kw", [
    (1, 1025, 1280, 200, {}),                       # one CTA more than a ranking block holds
    (1, 1500, 128, 300, dict(n_clusters=8)),        # the run-time number of clusters; many short rows
    (2, 1030, 768, 100, dict(kmeans_iters=1)),      # two tiles; one assignment step
    (8, 600, 2048, 64, {}),                         # rows too wide to stay in shared memory
    (10, 576, 1024, 64, {}),                        # the most tiles of this form, rows resident
    (1, 1100, 1024, 150, dict(sim="mse")),
    (1, 1100, 1024, 150, dict(sim="kl")),
])
def test_whole_gpu_kmeans(tiles, n, d, keep, kw):
    vs, res = [], []
    for i in range(tiles):
        _, v1, r1 = conditioned_vision(20263001 + 101 * i, 1, n, d, 2, 4, keep, 1, has_cls=False, attn_form=1, **kw)
        vs.append(v1)
        res += r1
    v = {"feats": [np.concatenate([x["feats"][l] for x in vs]) for l in range(2)],
         "attn": np.concatenate([x["attn"] for x in vs])}
    assert_prune_parity(gpu_prune(v, keep, 1, has_cls=False, attn_form=1, **kw), res)


@pytest.mark.parametrize("tiles,n,d,keep,layers,final,kw", [
    (12, 200, 2052, 40, 2, 1, {}),                  # rows too wide for the one-sweep ring: re-read from L2
    (12, 200, 32, 40, 2, 1, {}),                    # ... too short for it
    (12, 200, 32, 40, 2, 0, dict(sim="mse")),
    (12, 200, 2052, 40, 1, 0, dict(sim="kl")),
    (11, 333, 512, 50, 1, 0, {}),                   # one sweep: the final layer alone, first, between the others
    (11, 333, 512, 50, 3, 0, {}),
    (11, 333, 512, 50, 3, 1, {}),
    (11, 333, 512, 50, 3, 1, dict(sim="mse")),
    (1, 1100, 1024, 150, 1, 0, {}),                 # the whole GPU: the same
    (1, 1100, 1024, 150, 3, 0, {}),
    (1, 1100, 1024, 150, 3, 1, {}),
])
def test_kmeans_forms_and_layers(tiles, n, d, keep, layers, final, kw):
    vs, res = [], []
    for i in range(tiles):
        _, v1, r1 = conditioned_vision(20266001 + 307 * i, 1, n, d, layers, 4, keep, final, has_cls=False, attn_form=1,
                                       tries=256, **kw)
        vs.append(v1)
        res += r1
    v = {"feats": [np.concatenate([x["feats"][l] for x in vs]) for l in range(layers)],
         "attn": np.concatenate([x["attn"] for x in vs])}
    assert_prune_parity(gpu_prune(v, keep, final, has_cls=False, attn_form=1, **kw), res)


@pytest.mark.parametrize("tiles", [1, 12])
def test_prune_without_other_tokens(tiles):
    # every token is an anchor: nothing to cluster, score or select
    v = synth.vision_tiles(9, tiles, 70, 128, 2, 4, has_cls=False, attn_form=1)
    g = gpu_prune(v, 70, 1, has_cls=False, attn_form=1, anchor_ratio=1.0)
    np.testing.assert_array_equal(g["keep_idx"], np.tile(np.arange(70), (tiles, 1)))
    assert (g["kind"] == 1).all() and (g["cluster"] == -1).all() and np.isposinf(g["scores"]).all()


@pytest.mark.parametrize("tiles,n,d,keep,kw", [
    (11, 333, 1024, 50, {}),                        # eight CTAs a tile, each fewer rows than the ring holds
    (20, 576, 1028, 64, dict(kmeans_iters=1)),      # four CTAs; columns past 1024; one assignment step
    (80, 100, 2048, 20, {}),                        # one CTA a tile
    (12, 300, 256, 40, dict(sim="mse")),
    (12, 300, 256, 40, dict(sim="kl")),
    (12, 576, 1024, 64, dict(n_clusters=2)),        # K other than 4: rows re-read from L2 in clusters of eight
])
def test_many_tiles_kmeans(tiles, n, d, keep, kw):
    test_whole_gpu_kmeans(tiles, n, d, keep, kw)


def _stream_of_few_sms(n_sms):
    # a stream of a green context (a part of the device's SMs) through the driver's interface
    import ctypes as C
    cu = C.CDLL("libcuda.so.1")
    everything, part = (C.c_byte * 144)(), (C.c_byte * 144)()  # CUdevResource
    groups, desc, ctx, stream = C.c_uint(1), C.c_void_p(), C.c_void_p(), C.c_void_p()
    torch.cuda.init()
    torch.zeros(1, device="cuda")  # the primary context is current
    for rc in (lambda: cu.cuDeviceGetDevResource(0, everything, 1),  # 1: SMs
               lambda: cu.cuDevSmResourceSplitByCount(part, C.byref(groups), everything, None, 0, n_sms),
               lambda: cu.cuDevResourceGenerateDesc(C.byref(desc), part, 1),
               lambda: cu.cuGreenCtxCreate(C.byref(ctx), desc, 0, 1),  # 1: default stream, required
               lambda: cu.cuGreenCtxStreamCreate(C.byref(stream), ctx, 1, 0)):  # 1: non-blocking, required
        code = rc()
        if code != 0:
            pytest.skip(f"no green context here (driver error {code})")
    return torch.cuda.ExternalStream(stream.value)


def test_large_tile_in_a_context_of_few_sms():
    # a context that holds a part of the SMs cannot run the cooperative launch over all of them: the shape goes
    # through the clusters instead, with the same result
    _, v, res = conditioned_vision(20265001, 1, 1100, 1024, 2, 4, 150, 1, has_cls=False, attn_form=1)
    with torch.cuda.stream(_stream_of_few_sms(32)):
        assert_prune_parity(gpu_prune(v, 150, 1, has_cls=False, attn_form=1), res)
    assert_prune_parity(gpu_prune(v, 150, 1, has_cls=False, attn_form=1), res)


def test_whole_gpu_kmeans_iterations():
    v, res = _shuffled_tile(20264001, 900, 1280, 180)
    a = gpu_prune(v, 180, 1, has_cls=False, attn_form=1)
    assert_prune_parity(a, res)
    b = gpu_prune(v, 180, 1, has_cls=False, attn_form=1)  # sums in a fixed order: the same bits again
    np.testing.assert_array_equal(a["scores"].view(np.uint32), b["scores"].view(np.uint32))
    # the same tile among 24 (one sweep an iteration, every second one backwards)
    many = dict(feats=[np.repeat(f, 24, 0) for f in v["feats"]], attn=np.repeat(v["attn"], 24, 0))
    assert_prune_parity(gpu_prune(many, 180, 1, has_cls=False, attn_form=1), res * 24)


@pytest.mark.parametrize("n", [1024, 1025, 4096])
def test_anchor_ranking_with_ties(n):
    # equal importances fall to the lower index, on one CTA (up to 1024 tokens) and on several
    v = synth.vision_tiles(5, 1, n, 64, 1, 1, has_cls=False, attn_form=1)
    v["attn"][:] = np.random.default_rng(n).integers(0, 7, v["attn"].shape).astype(np.float32)
    g = gpu_prune(v, n // 2, 0, has_cls=False, attn_form=1, n_clusters=1, anchor_ratio=1.0)
    np.testing.assert_array_equal(g["keep_idx"][0], op.select_anchors(v["attn"][0, 0].astype(np.float64), n // 2))


# ---- prefill attention: 64-key blocks, P in TMEM ---------------------------------------------------------
@pytest.mark.parametrize("lens,H,Hkv,hd,frac,ramp", [
    ([63, 64, 65, 1, 191, 193], 4, 2, 128, 1.0, 0.0),  # lengths at the edges of key blocks
    ([127, 128, 129, 257], 4, 4, 64, 0.6, 0.0),        # ... and of query tiles
    ([700], 7, 1, 128, 0.9, 2.0),                      # maxima that grow a little a block
    ([700], 2, 2, 64, 0.9, 40.0),                      # ... by much at every block
    ([1500, 40], 2, 1, 128, 0.05, 8.0),                # few queries far down a long sequence
    ([2996, 1021], 14, 2, 128, 1.0, 0.0),              # many blocks and CTAs: warps of a CTA run ahead of others
])
def test_attention_edges(lens, H, Hkv, hd, frac, ramp):
    from tests import test_gpu_attention as A
    q, q_pos, q_cu, kv, cu = A.case(lens, H, Hkv, hd, frac, seed=sum(lens) + H, ramp=ramp)
    got = A.run(q, q_pos, q_cu, kv, cu, H, Hkv, hd)
    ref = A.oracle_attention(q, q_pos, q_cu, kv, cu, H, Hkv, hd)
    assert np.isfinite(got).all()
    assert rowwise_rel(got, ref) < A.TOL


@pytest.mark.parametrize("hd,ramp", [(128, 0.0), (128, 2.0), (64, 6.0)])
def test_attention_weights_and_sums(hd, ramp):
    # the arithmetic of the kernel, step by step: weights relative to the running maximum of 64-key blocks
    # (at most 1), rounded to bf16 for the product alone, the row sum over the unrounded ones. fp32
    # sums move an output by about 1e-5 of itself, past one in 250 of bf16's borders: 2 % may differ.
    from tests import test_gpu_attention as A
    n, H = 700, 2
    q, q_pos, q_cu, kv, cu = A.case([n], H, H, hd, 1.0, seed=hd, ramp=ramp)
    got = A.run(q, q_pos, q_cu, kv, cu, H, H, hd)
    qf, kvf = bf16_np(q).reshape(n, H, hd), bf16_np(kv).reshape(n, 2, H, hd)
    want = np.zeros((n, H, hd))
    for h in range(H):
        z = (qf[:, h] @ kvf[:, 0, h].T) * (1.4426950408889634 / np.sqrt(hd))
        z[np.triu_indices(n, 1)] = -np.inf
        m, l, o = np.full((n, 1), -np.inf), np.zeros((n, 1)), np.zeros((n, hd))
        for k in range(0, n, 64):
            mn = np.maximum(m, z[:, k:k + 64].max(1, keepdims=True))
            p, corr = np.exp2(z[:, k:k + 64] - mn), np.exp2(m - mn)
            pb = torch.from_numpy(p).float().to(torch.bfloat16).double().numpy()
            l, o, m = l * corr + p.sum(1, keepdims=True), o * corr + pb @ kvf[k:k + 64, 1, h], mn
        want[:, h] = o / l
    want = torch.from_numpy(want.reshape(n, H * hd)).float().to(torch.bfloat16).double().numpy()
    assert (got.reshape(n, H * hd) == want).mean() > 0.98
