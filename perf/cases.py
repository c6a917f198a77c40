"""Measured workloads of the WbG128 library: what a program that decodes with quantized weights, or
prepares them, has the library do.

A case is a dict of plain values; ``kind`` says which path it takes:

  linear    one eager ``laq_gemm_wxg128`` call on one projection (the smallest call);
  pass      the weight pass of one decode step: every projection of ``layers`` decoder layers
            (q|k|v, o, gate|up, down; distinct weights per layer, so that they stream from HBM),
            launched once per step from a CUDA graph as a decode loop would;
  mlp       the MLP blocks of ``layers`` layers from a CUDA graph: RMSNorm + residual folded into
            the gate|up GEMM, SiLU * up, the down GEMM;
  head      the LM head of one step and its greedy tokens;
  attn      the attention of one step over ``layers`` KV caches, with the q/k norm, rotary
            embedding and cache append fused in (``fused``) or as separate calls;
  quantize  fp16 weight -> packed codes, scales and zeros (``QuantLinear``), as model preparation
            does for every projection;
  codec     quantize, pack and unpack as separate calls (a checkpoint written and read back);
  step      one whole decode step of ``DecodeStep`` from its CUDA graph.

Weights, activations, norm weights, KV caches and embeddings follow the distributions of
``paper_2605_08755_gb300.inputs`` (N(0, 0.02^2) weights, optionally with 1 % outliers x 20, N(0, 1)
activations), drawn here from torch generators.
"""
import math

import numpy as np
import torch

DEV = "cuda"
EPS = 1e-6
THETA = 1e6

# (H, q heads, kv heads, I) of the decoders in the repository's configurations, and one with odd
# sizes (an uneven number of 16-column tiles and of 128-row groups everywhere).
DIMS = {
    "qwen3-4b": (2560, 32, 8, 9728),
    "qwen3-8b": (4096, 32, 8, 12288),
    "ragged": (1408, 15, 5, 3712),
}
VOCAB = 151936
D = 128


def listed():
    return [
        # the smallest call: one small projection called eagerly, as a first port of a model does
        dict(name="linear_1024_w3_m1", kind="linear", K=1024, N=1024, M=1, bits=3),
        # the headline: every weight of a Qwen3-4B-shaped decoder once, batch 1, 3 bits
        dict(name="pass_4b_w3_m1", kind="pass", model="qwen3-4b", layers=36, M=1, bits=3,
             outliers=False),
        # a small serving batch at 4 bits
        dict(name="pass_4b_w4_m4", kind="pass", model="qwen3-4b", layers=36, M=4, bits=4,
             outliers=False),
        # the largest batch on the larger decoder, weights with outliers (16 of its 36 layers)
        dict(name="pass_8b_w3_m16", kind="pass", model="qwen3-8b", layers=16, M=16, bits=3,
             outliers=True),
        # odd tile and group counts and an odd batch
        dict(name="pass_ragged_w4_m7", kind="pass", model="ragged", layers=16, M=7, bits=4,
             outliers=False),
        # MLP blocks with the fused norm at a middle batch
        dict(name="mlp_4b_w3_m8", kind="mlp", model="qwen3-4b", layers=12, M=8, bits=3),
        # the vocabulary projection and the greedy choice of one token
        dict(name="head_4b_w3_m1", kind="head", K=2560, N=VOCAB, M=1, bits=3),
        # attention of a single conversation, 2048 tokens, every layer's cache cold
        dict(name="attn_m1_ctx2048", kind="attn", layers=24, M=1, Hq=32, Hkv=8, L=2048,
             fused=True, full=True),
        # a full batch of long conversations of different lengths, through the separate calls
        dict(name="attn_m16_ctx8192", kind="attn", layers=1, M=16, Hq=32, Hkv=8, L=8192,
             fused=False, full=False),
        # preparing the largest projection of a layer at 4 bits
        dict(name="quantize_4b_gateup_w4", kind="quantize", K=2560, N=19456, bits=4,
             outliers=False),
        # a checkpoint's codes written and read back at 3 bits, outlier weights
        dict(name="codec_8b_down_w3", kind="codec", K=12288, N=4096, bits=3, outliers=True),
        # one whole token of the Qwen3-4B-shaped decoder
        dict(name="step_4b_w3_m1_ctx2048", kind="step", layers=36, M=1, bits=3, context=2048,
             vocab=VOCAB),
    ]


def _log(rng, lo, hi):
    """An integer in lo..hi, spread evenly over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["linear", "pass", "pass", "mlp", "head", "attn", "attn", "quantize",
                       "codec", "step"])
    bits, M = rng.choice([3, 4]), _log(rng, 1, 16)
    if kind == "linear":
        return dict(kind=kind, K=128 * _log(rng, 1, 96), N=16 * _log(rng, 4, 1536), M=M, bits=bits)
    if kind == "pass":
        model = rng.choice(sorted(DIMS))
        return dict(kind=kind, model=model, M=M, bits=bits, outliers=rng.random() < 0.5,
                    layers=_log(rng, 2, 32 if model == "ragged" else 12))
    if kind == "mlp":
        return dict(kind=kind, model=rng.choice(sorted(DIMS)), layers=_log(rng, 2, 12), M=M,
                    bits=bits)
    if kind == "head":
        return dict(kind=kind, K=128 * _log(rng, 8, 32), N=16 * _log(rng, 2000, VOCAB // 16), M=M,
                    bits=bits)
    if kind == "attn":
        Hkv = rng.choice([1, 2, 4, 5, 8])
        G = rng.choice([1, 2, 3, 4, 5, 7, 8])
        L = _log(rng, 64, 8192)
        return dict(kind=kind, layers=_log(rng, 1, 4 if M * L > 16384 else 16), M=M, Hq=G * Hkv,
                    Hkv=Hkv, L=L, fused=rng.random() < 0.5, full=rng.random() < 0.5)
    if kind in ("quantize", "codec"):
        return dict(kind=kind, K=128 * _log(rng, 2, 96), N=16 * _log(rng, 8, 1216), bits=bits,
                    outliers=rng.random() < 0.5)
    return dict(kind="step", layers=_log(rng, 1, 4), M=M, bits=bits, context=_log(rng, 16, 4096),
                vocab=16 * _log(rng, 64, 4096))


# ---- inputs -----------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _weight(g, K, N, outliers=False):
    w = torch.randn((K, N), generator=g, device=DEV) * 0.02
    if outliers:
        w = torch.where(torch.rand((K, N), generator=g, device=DEV) < 0.01, w * 20.0, w)
    return w.to(torch.float16)


def _normal(g, *shape):
    return torch.randn(shape, generator=g, device=DEV).to(torch.float16)


def _norm_weight(g, n):
    return (1.0 + 0.1 * torch.randn(n, generator=g, device=DEV)).to(torch.float16)


def _projections(model):
    """(K, N) of the fused projections of one layer, in launch order."""
    H, Hq, Hkv, I = DIMS[model]
    return [(H, (Hq + 2 * Hkv) * D), (Hq * D, H), (H, 2 * I), (I, H)]


def _pass_inputs(case, seed):
    """(X, W) of every launch of the pass, one at a time."""
    g = _gen(seed)
    for _ in range(case["layers"]):
        for K, N in _projections(case["model"]):
            yield _normal(g, case["M"], K), _weight(g, K, N, case["outliers"])


def _mlp_inputs(case, seed):
    """(x, residual, norm weight, W gate|up, W down) of every block, one at a time."""
    g = _gen(seed)
    H, _, _, I = DIMS[case["model"]]
    for _ in range(case["layers"]):
        yield (_normal(g, case["M"], H), _normal(g, case["M"], H), _norm_weight(g, H),
               _weight(g, H, 2 * I), _weight(g, I, H))


def _lengths(case, seed):
    """Tokens in each row's cache, the new one included."""
    M, L = case["M"], case["L"]
    if case["full"]:
        return np.full(M, L, dtype=np.int32)
    return np.random.default_rng(seed).integers(max(1, L // 4), L + 1, size=M).astype(np.int32)


def _attn_inputs(case, seed):
    """(qkv, q norm, k norm, K cache, V cache) of every layer, one at a time."""
    g = _gen(seed)
    M, Hq, Hkv, L = case["M"], case["Hq"], case["Hkv"], case["L"]
    for _ in range(case["layers"]):
        yield (_normal(g, M, (Hq + 2 * Hkv) * D), _norm_weight(g, D), _norm_weight(g, D),
               _normal(g, M, Hkv, L, D), _normal(g, M, Hkv, L, D))


# ---- what a program keeps, and one pass -------------------------------------------------------

def _linear(W, bits, M):
    """A quantized projection and the launch plan a decode loop uses for it."""
    from paper_2605_08755_gb300 import _lib
    from paper_2605_08755_gb300.weight_pass import QuantLinear
    q = QuantLinear(W, bits)
    sms = torch.cuda.get_device_properties(torch.device(DEV)).multi_processor_count
    cfg = _lib.laq_gemm_plan(M, q.K, q.N, bits, sms)
    cfg.pdl = 1
    return q, cfg


def _capture(launch):
    """Run once (first calls set kernel attributes), then record the launches into a graph."""
    launch(None)
    torch.cuda.synchronize()
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        launch(stream)
    return graph


def prepare(case, seed):
    from paper_2605_08755_gb300 import _lib
    kind, M, bits = case["kind"], case.get("M"), case.get("bits")
    st = dict(kind=kind, bits=bits)
    if kind == "linear":
        g = _gen(seed)
        st["X"] = _normal(g, M, case["K"])
        st["q"], _ = _linear(_weight(g, case["K"], case["N"]), bits, M)
    elif kind == "pass":
        out = [torch.empty((case["layers"], M, N), dtype=torch.float16, device=DEV)
               for _, N in _projections(case["model"])]
        calls = []
        for i, (X, W) in enumerate(_pass_inputs(case, seed)):
            calls.append((X, *_linear(W, bits, M), out[i % 4][i // 4]))

        def launch(stream):
            for X, q, cfg, Y in calls:
                _lib.laq_gemm_wxg128(X, q.packed, q.s, q.z, bits, Y=Y, config=cfg, stream=stream)
        st["keep"], st["out"] = calls, out
        st["graph"] = _capture(launch)
    elif kind == "mlp":
        H, _, _, I = DIMS[case["model"]]
        f16 = dict(dtype=torch.float16, device=DEV)
        res = torch.empty((case["layers"], M, H), **f16)
        out = torch.empty((case["layers"], M, H), **f16)
        ygu, act = torch.empty((M, 2 * I), **f16), torch.empty((M, I), **f16)
        blocks = []
        for i, (x, r, w, Wgu, Wd) in enumerate(_mlp_inputs(case, seed)):
            blocks.append((x, r, w, _linear(Wgu, bits, M), _linear(Wd, bits, M), res[i], out[i]))

        def launch(stream):
            for x, r, w, (gu, gcfg), (dn, dcfg), r_out, y in blocks:
                _lib.laq_gemm_wxg128_prologue(x, gu.packed, gu.s, gu.z, bits,
                                              _lib.PROLOGUE_RMSNORM, Y=ygu, R=r, R_out=r_out, w=w,
                                              eps=EPS, config=gcfg, stream=stream)
                _lib.laq_silu_mul(ygu, h=act, stream=stream)
                _lib.laq_gemm_wxg128(act, dn.packed, dn.s, dn.z, bits, Y=y, config=dcfg,
                                     stream=stream)
        st["keep"], st["out"] = (blocks, ygu, act), (res, out)
        st["graph"] = _capture(launch)
    elif kind == "head":
        g = _gen(seed)
        X = _normal(g, M, case["K"])
        q, cfg = _linear(_weight(g, case["K"], case["N"]), bits, M)
        logits = torch.empty((M, q.N), dtype=torch.float16, device=DEV)
        tok = torch.empty((M,), dtype=torch.int32, device=DEV)

        def launch(stream):
            _lib.laq_gemm_wxg128(X, q.packed, q.s, q.z, bits, Y=logits, config=cfg, stream=stream)
            _lib.laq_argmax(logits, out=tok, stream=stream)
        st["keep"], st["out"] = (X, q), (logits, tok)
        st["graph"] = _capture(launch)
    elif kind == "attn":
        Hq, Hkv, L = case["Hq"], case["Hkv"], case["L"]
        lens = torch.from_numpy(_lengths(case, seed)).to(DEV)
        pos = lens - 1
        n, f16 = case["layers"], dict(dtype=torch.float16, device=DEV)
        out = torch.empty((n, M, Hq, D), **f16)
        kcs, vcs = (torch.empty((n, M, Hkv, L, D), **f16) for _ in range(2))
        layers = []
        for i, (qkv, qw, kw, kc, vc) in enumerate(_attn_inputs(case, seed)):
            kcs[i].copy_(kc)
            vcs[i].copy_(vc)
            layers.append((qkv, qw, kw, kcs[i], vcs[i], out[i]))
        ws = (_lib.attention_qkv_workspace(M, Hq, Hkv, L, DEV) if case["fused"]
              else _lib.attention_workspace(M, Hq, L, DEV))
        qbuf = torch.empty((M, Hq, D), dtype=torch.float16, device=DEV)
        scale = 1.0 / math.sqrt(D)

        def launch(stream):
            for qkv, qw, kw, kc, vc, o in layers:
                if case["fused"]:
                    _lib.laq_attention_qkv(qkv, qw, kw, pos, Hq, Hkv, THETA, EPS, kc, vc, scale,
                                           ws, out=o, stream=stream)
                else:
                    _lib.laq_qk_norm_rope(qkv, qw, kw, pos, Hq, Hkv, THETA, EPS, kc, vc,
                                          q_out=qbuf, stream=stream)
                    _lib.laq_attention_decode(qbuf, kc, vc, lens, scale, ws, out=o,
                                              stream=stream)
        st["keep"], st["out"] = (lens, pos, layers, ws, qbuf), (out, kcs, vcs)
        st["graph"] = _capture(launch)
    elif kind in ("quantize", "codec"):
        st["W"] = _weight(_gen(seed), case["K"], case["N"], case["outliers"])
    else:
        from paper_2605_08755_gb300.decode_step import DecodeStep
        step = DecodeStep("qwen3-4b", bits=bits, M=M, layers=case["layers"],
                          context=case["context"], vocab=case["vocab"], seed=seed, device=DEV)
        kcs, vcs = torch.stack(step.kc), torch.stack(step.vc)  # all layers' caches in one piece
        step.kc, step.vc = list(kcs), list(vcs)
        st["keep"], st["graph"] = step, step.capture()
        st["out"] = (step.logits, kcs, vcs)
    return st


def run(st):
    from paper_2605_08755_gb300 import _lib
    kind = st["kind"]
    if "graph" in st:
        st["graph"].replay()
        return st["out"]
    if kind == "linear":
        q = st["q"]
        return _lib.laq_gemm_wxg128(st["X"], q.packed, q.s, q.z, st["bits"])
    if kind == "quantize":
        from paper_2605_08755_gb300.weight_pass import QuantLinear
        q = QuantLinear(st["W"], st["bits"])
        return q.packed, q.s, q.z
    codes, s, z = _lib.laq_quantize_rtn(st["W"], st["bits"])
    packed = _lib.laq_pack(codes, st["bits"])
    K, N = codes.shape
    return codes, s, z, packed, _lib.laq_unpack(packed, K, N, st["bits"])


# ---- the work a pass cannot do without --------------------------------------------------------

def _gemm_work(M, K, N, bits):
    return K * N * bits // 8 + K // 128 * N * 3 + 2 * M * (K + N), 2 * M * K * N


def _attn_work(M, Hq, Hkv, tokens):
    """tokens: cached tokens read, summed over the rows (the new one included)."""
    return tokens * Hkv * D * 4 + M * (2 * Hq + 4 * Hkv) * D * 2, 4 * tokens * Hq * D


def work(case):
    kind, M, bits = case["kind"], case.get("M"), case.get("bits")
    parts = []
    if kind in ("linear", "head"):
        parts = [_gemm_work(M, case["K"], case["N"], bits)]
        if kind == "head":
            parts.append((4 * M, M * case["N"]))
    elif kind == "pass":
        parts = [_gemm_work(M, K, N, bits) for K, N in _projections(case["model"])] * case["layers"]
    elif kind == "mlp":
        H, _, _, I = DIMS[case["model"]]
        parts = [_gemm_work(M, H, 2 * I, bits), _gemm_work(M, I, H, bits),
                 (4 * M * H + 2 * H, 6 * M * (H + I))] * case["layers"]
    elif kind == "attn":
        # the lengths depend on the seed: their mean
        mean = case["L"] if case["full"] else (max(1, case["L"] // 4) + case["L"]) / 2
        parts = [_attn_work(M, case["Hq"], case["Hkv"], int(M * mean))] * case["layers"]
    elif kind in ("quantize", "codec"):
        KN, GN = case["K"] * case["N"], case["K"] // 128 * case["N"]
        parts = [(2 * KN + KN * bits // 8 + 3 * GN, 4 * KN)]
        if kind == "codec":  # codes written by the quantizer, and by the reader of the packed form
            parts.append((2 * KN, 2 * KN))
    else:
        H, Hq, Hkv, I = DIMS["qwen3-4b"]
        parts = [_gemm_work(M, K, N, bits) for K, N in _projections("qwen3-4b")]
        parts.append(_attn_work(M, Hq, Hkv, M * case["context"]))
        parts = parts * case["layers"] + [_gemm_work(M, H, case["vocab"], bits), (4 * M * H, 0)]
    return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}


def tolerance(case):
    kind = case["kind"]
    if kind in ("quantize", "codec"):
        return "exact"  # codes, scales, zeros and packed bytes are defined bit for bit
    if kind == "step":
        return {"rel": 2e-2, "max": 0.2}  # fp16 rounding differences travel through every layer
    if kind == "mlp":
        return {"rel": 2.5e-3, "max": 2e-2}  # the fp16 roundings of input, gate|up and SiLU * up
    # one fp16 rounding of each output (2.1e-4 relative, measured; 3e-4 after attention's fp16 q)
    return {"rel": 1e-3, "max": 1e-2, "differ": 0.01}


# ---- the same results in 64 bits --------------------------------------------------------------

def _quantize64(W, bits):
    """codes, scales (fp16 values) and zeros of min-max RTN quantization, groups of 128 rows."""
    K, N = W.shape
    qmax = 2 ** bits - 1
    w = W.double().view(K // 128, 128, N)
    lo, hi = w.amin(1), w.amax(1)
    lo0, hi0 = lo.clamp(max=0.0), hi.clamp(min=0.0)
    v = (hi0 - lo0) / qmax
    h = v.to(torch.float16)
    up = (h.view(torch.int16) + 1).view(torch.float16)
    down = (h.view(torch.int16) - 1).clamp(min=0).view(torch.float16)
    h = torch.where(h.double() < v, up, torch.where(down.double() >= v, down, h))
    s = h.double().clamp(min=2.0 ** -14)
    z = torch.round(-lo0 / s)
    const = lo == hi
    s = torch.where(const, torch.where(lo == 0, torch.ones_like(lo), lo.abs()), s)
    z = torch.where(const, (lo < 0).double(), z)
    q = (torch.round(w / s[:, None]) + z[:, None]).clamp(0, qmax)
    return q, s, z


def _dequantized64(W, bits):
    q, s, z = _quantize64(W, bits)
    return (s[:, None] * (q - z[:, None])).view(W.shape)


def _packed(codes, bits):
    """The record layout: 16 columns x 128 rows per record, tile-major; lane l = 4 r + c of a
    record holds columns r, r + 8 and rows 32 c + 4 j + 2 h + e in 16-bit fields (e: which half)."""
    K, N = codes.shape
    T, G = N // 16, K // 128
    # [g, c, j, h, e, t, row, r] -> [t, g, lane (r, c), pair i = 2 j + h, row, e]
    a = codes.to(torch.int64).view(G, 4, 8, 2, 2, T, 2, 8).permute(5, 0, 7, 1, 2, 3, 6, 4)
    a = a.reshape(T, G, 32, 16, 2, 2)
    both = a[..., 0] | a[..., 1] << 16  # [t, g, lane, pair, row]
    if bits == 4:
        words = [both[:, :, :, 2 * j, 0] | both[:, :, :, 2 * j + 1, 0] << 4
                 | both[:, :, :, 2 * j, 1] << 8 | both[:, :, :, 2 * j + 1, 1] << 12
                 for j in range(8)]
        split = 4
    else:
        words = [(both[:, :, :, 15, w // 3] >> w % 3) & 0x10001
                 | both[:, :, :, w, 0] << 1 | both[:, :, :, 6 + w, 0] << 4
                 | both[:, :, :, 12 + w // 2, w % 2] << 7
                 | both[:, :, :, w, 1] << 10 | both[:, :, :, 6 + w, 1] << 13 for w in range(6)]
        split = 4
    first = torch.stack(words[:split], -1).reshape(T, G, -1)   # 4 words per lane
    rest = torch.stack(words[split:], -1).reshape(T, G, -1)    # then the lanes' remaining words
    u = torch.cat([first, rest], -1).reshape(-1)
    u = torch.where(u >= 2 ** 31, u - 2 ** 32, u).to(torch.int32)
    return u.view(torch.uint8)


def _rms64(x, w):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + EPS) * w.double()


def _rope64(x, pos):
    """x [M, heads, D] at positions pos [M]."""
    inv = THETA ** (-torch.arange(D // 2, dtype=torch.float64, device=x.device) * 2 / D)
    a = pos.double()[:, None, None] * inv
    cos, sin = torch.cos(a), torch.sin(a)
    x1, x2 = x[..., :D // 2], x[..., D // 2:]
    return torch.cat([x1 * cos - x2 * sin, x2 * cos + x1 * sin], -1)


def _attention64(qkv, qw, kw, kc, vc, pos, Hq, Hkv):
    """Attention output [M, Hq, D] and the caches with the new token, all in 64 bits."""
    M = qkv.shape[0]
    h = qkv.view(M, Hq + 2 * Hkv, D)
    q = _rope64(_rms64(h[:, :Hq], qw), pos)
    k = _rope64(_rms64(h[:, Hq:Hq + Hkv], kw), pos)
    kc, vc = kc.double(), vc.double()
    rows = torch.arange(M, device=pos.device)
    kc[rows, :, pos.long()] = k
    vc[rows, :, pos.long()] = h[:, Hq + Hkv:]
    out = torch.empty((M, Hq, D), dtype=torch.float64, device=qkv.device)
    for m in range(M):
        n = int(pos[m]) + 1
        sc = torch.einsum("gjd,gtd->gjt", q[m].view(Hkv, Hq // Hkv, D), kc[m, :, :n])
        p = torch.softmax(sc / math.sqrt(D), -1)
        out[m] = torch.einsum("gjt,gtd->gjd", p, vc[m, :, :n]).reshape(Hq, D)
    return out, kc, vc


def _silu_up64(gu):
    g, u = gu.chunk(2, -1)
    return g / (1.0 + torch.exp(-g)) * u


def _step_inputs(case, seed):
    """The synthetic model of ``DecodeStep``: its seeds and distributions, drawn again."""
    H, Hq, Hkv, I = DIMS["qwen3-4b"]
    M, V, ctx = case["M"], case["vocab"], case["context"]
    for l in range(case["layers"]):
        b = seed + 1000 * l
        w = [_weight(_gen(b + i), K, N) for i, (K, N) in enumerate(
            [(H, Hq * D), (H, Hkv * D), (H, Hkv * D), (Hq * D, H), (H, I), (H, I), (I, H)])]
        norms = [_norm_weight(_gen(b + 10 + j + 5_555_555), n) for j, n in enumerate((H, H, D, D))]
        kc = _normal(_gen(b + 20 + 1_111_111), M, Hkv, ctx, D)
        vc = _normal(_gen(b + 21 + 1_111_111), M, Hkv, ctx, D)
        yield w, norms, kc, vc
    final = _norm_weight(_gen(seed + 1000 * case["layers"] + 10 + 5_555_555), H)
    E = (0.05 * torch.randn((V, H), generator=_gen(seed + 3_333_333), device=DEV)).half()
    tok = np.random.default_rng(seed + 9_999_999).integers(0, V, size=M)
    yield final, E, torch.from_numpy(tok).to(DEV)


def _step64(case, seed):
    H, Hq, Hkv, I = DIMS["qwen3-4b"]
    bits, M = case["bits"], case["M"]
    pos = torch.full((M,), case["context"] - 1, device=DEV)
    _, E, tok = next(_step_inputs(dict(case, layers=0), seed))
    r, kcs, vcs = E[tok].double(), [], []
    for item in _step_inputs(case, seed):
        if len(item) == 3:
            final = item[0]
            break
        w, (inw, postw, qw, kw), kc, vc = item
        h = _rms64(r, inw)
        qkv = torch.cat([h @ _dequantized64(w[i], bits) for i in range(3)], -1)
        a, kc, vc = _attention64(qkv, qw, kw, kc, vc, pos, Hq, Hkv)
        r = r + a.view(M, -1) @ _dequantized64(w[3], bits)
        h = _rms64(r, postw)
        gu = torch.cat([h @ _dequantized64(w[i], bits) for i in (4, 5)], -1)
        r = r + _silu_up64(gu) @ _dequantized64(w[6], bits)
        kcs.append(kc)
        vcs.append(vc)
    h = _rms64(r, final)
    logits = torch.cat([h @ _dequantized64(e.t().contiguous(), bits) for e in E.split(16384)], -1)
    return logits, torch.stack(kcs), torch.stack(vcs)


def exact(case, seed):
    kind, bits = case["kind"], case.get("bits")
    if kind in ("linear", "head"):
        g = _gen(seed)
        X = _normal(g, case["M"], case["K"])
        W = _weight(g, case["K"], case["N"])
        Y = torch.cat([X.double() @ _dequantized64(w.contiguous(), bits)
                       for w in W.split(16384, 1)], -1)
        return Y if kind == "linear" else (Y, None)
    if kind == "pass":
        Y = [X.double() @ _dequantized64(W, bits) for X, W in _pass_inputs(case, seed)]
        return [torch.stack(Y[i::4]) for i in range(4)]
    if kind == "mlp":
        out = []
        for x, r, w, Wgu, Wd in _mlp_inputs(case, seed):
            h = x.double() + r.double()
            y = _silu_up64(_rms64(h, w) @ _dequantized64(Wgu, bits)) @ _dequantized64(Wd, bits)
            out.append((h, y))
        return tuple(torch.stack(t) for t in zip(*out))
    if kind == "attn":
        pos = torch.from_numpy(_lengths(case, seed)).to(DEV) - 1
        out = [_attention64(t[0].double(), *t[1:], pos, case["Hq"], case["Hkv"])
               for t in _attn_inputs(case, seed)]
        return tuple(torch.stack(t) for t in zip(*out))
    if kind in ("quantize", "codec"):
        W = _weight(_gen(seed), case["K"], case["N"], case["outliers"])
        q, s, z = _quantize64(W, bits)
        codes = q.to(torch.uint8).view(W.shape)
        s, z = s.half(), z.to(torch.uint8)
        packed = _packed(codes, bits)
        return (packed, s, z) if kind == "quantize" else (codes, s, z, packed, codes)
    return _step64(case, seed)
