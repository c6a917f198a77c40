"""The attention kernel where its split can go wrong: steps of 16 tokens dealt to the warps of a
cluster, several clusters per pair on long caches, every group size, non-finite values."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import decoder as dec  # noqa: E402
from paper_2605_08755_gb300 import _lib, inputs  # noqa: E402

pytestmark = pytest.mark.gpu
D = 128
SCALE = 1 / math.sqrt(D)


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2605_08755_gb300 import build
    build.build()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def attend(q, kc, vc, lens, ws=None):
    M, Hq = q.shape[:2]
    ws = _lib.attention_workspace(M, Hq, kc.shape[2], "cuda") if ws is None else ws
    out = _lib.laq_attention_decode(dev(q), dev(kc), dev(vc), dev(np.array(lens, np.int32)),
                                    SCALE, ws)
    torch.cuda.synchronize()
    return out.cpu().numpy().astype(np.float64)


def check(out, ref):
    # one fp16 rounding on each side (2^-11 of the value each), and fp32 sums (1e-5 of the row)
    assert (np.abs(out - ref) <= 2.0 ** -10 * np.abs(ref)
            + 1e-5 * np.abs(ref).max(-1, keepdims=True) + 2.0 ** -24).all()


@pytest.mark.parametrize("G,Hkv,L,lens", [
    (1, 1, 1, [1]), (1, 8, 17, [16, 17, 1]), (3, 5, 130, [15, 16, 17, 63, 64, 65, 128, 130]),
    (5, 2, 300, [300, 299]), (7, 4, 1000, [1000, 513, 0]), (8, 2, 2048, [2048, 2047, 3]),
    (4, 8, 2100, [2100]), (2, 1, 520, list(range(500, 520))), (8, 1, 9000, [9000, 100]),
    (4, 1, 20000, [20000]), (8, 1, 40000, [39999, 5, 0, -1])])
def test_attention_splits(G, Hkv, L, lens):
    M, rng = len(lens), np.random.default_rng(G * L + Hkv)
    q = rng.standard_normal((M, G * Hkv, D)).astype(np.float16)
    kc = inputs.kv_cache(M, Hkv, L, D, seed=L)
    vc = inputs.kv_cache(M, Hkv, L, D, seed=L + 1)
    if L > 100:  # a few dominant keys, so that late maxima rescale what was summed before
        kc[:, :, L // 3] *= 4
        kc[:, :, -2] *= 6
    # a dirty workspace: nothing in it may be read before it is written
    nb = _lib.attention_workspace(M, G * Hkv, L, "cuda").fill_(float("nan"))
    out = attend(q, kc, vc, lens, nb)
    check(out, dec.attention(q, kc, vc, lens, SCALE).astype(np.float64))
    for m, n in enumerate(lens):
        if n <= 0:
            assert not out[m].any()


@pytest.mark.parametrize("G,Hkv,L,pos", [(1, 1, 40, [0, 15, 16, 39]), (7, 3, 700, [699, 640, 5]),
                                         (8, 1, 20000, [19999, 16, 20000])])
def test_fused_attention_appends_and_attends(G, Hkv, L, pos):
    M, Hq = len(pos), G * Hkv
    rng = np.random.default_rng(L + G)
    qkv = (2 * rng.standard_normal((M, (Hq + 2 * Hkv) * D))).astype(np.float16)
    qw, kw = inputs.norm_weight(D, 1), inputs.norm_weight(D, 2)
    kc0, vc0 = inputs.kv_cache(M, Hkv, L, D, 3), inputs.kv_cache(M, Hkv, L, D, 4)
    kc, vc = dev(kc0), dev(vc0)
    pd = dev(np.array(pos, np.int32))
    # the separate calls give q, the new k and v exactly as the fused call must use them
    kc2, vc2 = kc.clone(), vc.clone()
    q = _lib.laq_qk_norm_rope(dev(qkv), dev(qw), dev(kw), pd, Hq, Hkv, 1e6, 1e-6, kc2, vc2)
    ws = _lib.attention_qkv_workspace(M, Hq, Hkv, L, "cuda").fill_(0xff)
    out = _lib.laq_attention_qkv(dev(qkv), dev(qw), dev(kw), pd, Hq, Hkv, 1e6, 1e-6, kc, vc, SCALE,
                                 ws)
    torch.cuda.synchronize()
    assert torch.equal(kc, kc2) and torch.equal(vc, vc2)
    lens = [min(p + 1, L) for p in pos]
    ref = dec.attention(q.cpu().numpy(), kc2.cpu().numpy(), vc2.cpu().numpy(), lens, SCALE)
    check(out.cpu().numpy().astype(np.float64), np.asarray(ref, np.float64))


def test_attention_non_finite_values():
    """An infinite v gives an infinite output of its sign, a NaN stays in its own head and
    dimension, and neither reaches past the row's length."""
    M, Hkv, G, L = 1, 2, 4, 200
    rng = np.random.default_rng(5)
    q = rng.standard_normal((M, G * Hkv, D)).astype(np.float16)
    kc, vc = inputs.kv_cache(M, Hkv, L, D, 6), inputs.kv_cache(M, Hkv, L, D, 7)
    vc[0, 0, 10, 3], vc[0, 0, 50, 4], vc[0, 1, 20, 5] = np.inf, -np.inf, np.nan
    kc[0, :, 150:], vc[0, :, 150:] = np.nan, np.inf
    out = attend(q, kc, vc, [150])
    assert (out[0, :G, 3] == np.inf).all() and (out[0, :G, 4] == -np.inf).all()
    assert np.isnan(out[0, G:, 5]).all()
    bad = np.zeros((G * Hkv, D), bool)
    bad[:G, 3:5], bad[G:, 5] = True, True
    vc[~np.isfinite(vc)] = 0
    kc[~np.isfinite(kc)] = 0
    ref = dec.attention(q, kc, vc, [150], SCALE).astype(np.float64)
    check(np.where(bad, 0, out[0]), np.where(bad, 0, ref[0]))


@pytest.mark.parametrize("G,M", [(4, 320), (8, 320)])
def test_sums_over_many_steps_stay_exact(G, M):
    """One CTA per row, so a warp adds up 16 steps: of values with mean 1 and nearly equal weights
    every sum grows to the end.  A relative error r rounds about 1500 r of the fp16 outputs apart from
    64 bits (an fp16 step is 2^-10 to 2^-11 of its value); fp32 sums stay within 2^-22 of the result:
    3.6e-4 of them.  (Sums kept inside the tensor core, which truncates: 1e-3 and more.)"""
    L, Hkv = 2048, 1
    g = torch.Generator(device="cuda").manual_seed(G)
    f16 = lambda *shape: torch.randn(shape, generator=g, device="cuda").half()
    q, kc, vc = f16(M, G * Hkv, D), f16(M, Hkv, L, D), (f16(M, Hkv, L, D).float() + 1).half()
    lens = torch.full((M,), L, dtype=torch.int32, device="cuda")
    out = _lib.laq_attention_decode(q, kc, vc, lens, SCALE,
                                    _lib.attention_workspace(M, G * Hkv, L, "cuda"))
    ref = torch.cat([torch.softmax(q[m:m + 1].double() @ kc[m].double().mT * SCALE, -1)
                     @ vc[m].double() for m in range(M)])
    assert (out != ref.half()).double().mean() <= 3.6e-4
