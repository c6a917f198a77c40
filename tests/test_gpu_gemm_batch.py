"""The batch kernel at every launch shape it has, on sizes ragged against its tiles,
teams, clusters and shared-memory phases, and the plan that chooses among them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2605_08755_gb300 as laq  # noqa: E402
from oracle import c_oracle as co  # noqa: E402
from paper_2605_08755_gb300 import _lib, inputs  # noqa: E402

TAG = 0x4c424154


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2605_08755_gb300 import build
    build.build()


def batch_config(tw, slots, cluster, pdl=0):
    c = laq.GemmConfig.make(1, 8, 1, 4, pdl)
    c.reserved[0], c.reserved[1] = TAG, tw | slots << 8 | cluster << 16
    return c


def prepared(K, N, bits, seed):
    W = inputs.weights(K, N, seed=seed)
    codes, s, z = co.quantize_rtn(W, bits)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return ((codes, s, z), dev(co.pack(codes, bits).view(np.uint8)),
            dev(s.view(np.uint16)).view(torch.float16), dev(z))


def check(Y, ref, X, q):
    """One fp16 rounding, and fp32 sums: a group's accumulators are as large as sum |x_k| times the
    largest extraction offset (1024) plus the largest code, rounded about 2^-24 of that per
    addition over 8 MMAs, the sum of the two chains, P and z S (16 allowed), times the group's scale.
    (A bound for gross errors at every shape; how exact the sums are is tested below.)"""
    codes, s, z = q
    G = s.shape[0]
    mag = np.abs(X.astype(np.float64)).reshape(X.shape[0], G, 128).sum(-1) * 1040
    bound = 16 * 2.0 ** -24 * (mag @ s.astype(np.float64)) + 2.0 ** -11 * np.abs(ref) + 2.0 ** -24
    err = np.abs(Y.astype(np.float64) - ref)
    assert np.isfinite(Y).all() and (err <= bound).all(), (err / bound).max()


@pytest.mark.gpu
@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("M", [1, 2, 3, 8, 9, 16])
def test_every_launch_shape(bits, M):
    K, N = 1408, 21 * 16     # 11 groups, 21 tiles
    q, packed, s, z = prepared(K, N, bits, seed=M)
    X = inputs.activations(M, K, seed=M)
    ref, xd = co.gemm(X, *q), torch.from_numpy(X).cuda()
    for tw in (1, 2):
        for slots in (1, 2, 4, 8):
            for cluster in range(1, 9):
                Y = torch.full((M, N), float("nan"), dtype=torch.float16, device="cuda")
                laq.laq_gemm_wxg128(xd, packed, s, z, bits, Y=Y,
                                    config=batch_config(tw, slots, cluster, cluster & 1))
                check(Y.cpu().numpy(), ref, X, q)


@pytest.mark.gpu
@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("K", [1408, 4096])
@pytest.mark.parametrize("outliers", [False, True])
def test_sums_are_as_exact_as_the_general_kernels(bits, K, outliers):
    """What a kernel adds to the final fp16 rounding, over 16 batches: the batch kernel's no more
    than the general kernel's.  A row's groups share their P, so the errors of a row go together:
    256 rows make the root mean square good to about 5 %, two of them to 7; 1.15 is twice that.
    (One accumulator chain started at -P - z S: 1.5 times the general kernel's, 2.1 with outliers.)"""
    M, N = 16, 1024
    q, packed, s, z = prepared(K, N, bits, seed=K)
    own = {}
    for seed in range(16):
        X = inputs.activations(M, K, seed=seed).astype(np.float32)
        if outliers:
            X[np.random.default_rng(seed).random(X.shape) < 0.01] *= 50
        X = X.astype(np.float16)
        ref = co.gemm(X, *q)
        rounded = ref.astype(np.float16)
        for name, cfg in (("batch", batch_config(2, 4, 1)),
                          ("general", laq.GemmConfig.make(8, 8, 1, 4))):
            Y = laq.laq_gemm_wxg128(torch.from_numpy(X).cuda(), packed, s, z, bits, config=cfg)
            d2 = np.square(Y.cpu().numpy().astype(np.float64) - ref)
            own[name] = own.get(name, 0.0) + (
                (d2 - np.square(rounded.astype(np.float64) - ref)).sum() / np.square(ref).sum())
    assert 0 < own["batch"] <= 1.15 ** 2 * own["general"], (own["batch"] / own["general"]) ** 0.5


@pytest.mark.gpu
@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("M,K,N,shape", [
    (16, 128, 16, (2, 8, 1)), (3, 256, 16, (2, 1, 8)),          # fewer groups than CTAs and teams
    (16, 12288, 272, (2, 8, 1)), (16, 9728, 48, (2, 1, 3)),     # several phases of staged X
    (5, 16384, 80, (1, 8, 2)), (8, 1920, 1408, (2, 2, 5))])
def test_phases_and_edges(bits, M, K, N, shape):
    q, packed, s, z = prepared(K, N, bits, seed=K + N)
    X = inputs.activations(M, K, seed=K)
    Y = laq.laq_gemm_wxg128(torch.from_numpy(X).cuda(), packed, s, z, bits,
                            config=batch_config(*shape))
    check(Y.cpu().numpy(), co.gemm(X, *q), X, q)


def check_prologue(Y, Z, xin):
    """Y with the prologue against Z, the plain GEMM of the input rounded from 64 bits.  The
    prologue's input is within 2^-20 of the exact one (fp32 sums and reciprocals), so it rounds apart
    where that is within 2^-20 of a tie: K 2^-9 of the K elements expected, 8 more allowed, each by
    one fp16 step (2^-10 of it) of either sign.  8 standard deviations of their sum through weights of
    root mean square 0.02, one rounding of each output, and the plain kernel's sums in another order
    where the two stage K in phases of other lengths."""
    Y, Z = Y.cpu().numpy().astype(np.float64), Z.cpu().numpy().astype(np.float64)
    K = xin.shape[1]
    rms = np.sqrt(np.square(xin.astype(np.float64)).mean())
    bound = (8 * np.sqrt(8 + K * 2.0 ** -9) * 2.0 ** -10 * rms * 0.02 + 2.0 ** -10 * np.abs(Z)
             + 2.0 ** -12 * np.sqrt(np.square(Z).mean()))
    assert np.isfinite(Y).all() and (np.abs(Y - Z) <= bound).all(), (np.abs(Y - Z) / bound).max()


@pytest.mark.gpu
@pytest.mark.parametrize("M,K", [(1, 1408), (3, 1408), (7, 1408), (8, 256), (16, 1408),
                                 (16, 12288)])   # the last: several phases, two passes over X and R
def test_prologues(M, K):
    bits, N = 3, 336
    q, packed, s, z = prepared(K, N, bits, seed=1)
    dev = lambda a: torch.from_numpy(a).cuda()
    x, r = inputs.activations(M, K, seed=2), inputs.activations(M, K, seed=3)
    w = inputs.norm_weight(K, seed=4)
    h = (x.astype(np.float32) + r.astype(np.float32)).astype(np.float16)  # one fp16 sum: exact
    h64 = h.astype(np.float64)
    xin = (h64 / np.sqrt(np.square(h64).mean(-1, keepdims=True) + 1e-6) * w).astype(np.float16)
    gu = inputs.activations(M, 2 * K, seed=5)
    g64 = gu.astype(np.float64)
    act = (g64[:, :K] / (1 + np.exp(-g64[:, :K])) * g64[:, K:]).astype(np.float16)
    for shape in ((2, 4, 1), (1, 2, 3), (2, 8, 8)):
        cfg = batch_config(*shape)
        hd = torch.empty((M, K), dtype=torch.float16, device="cuda")
        Y = _lib.laq_gemm_wxg128_prologue(dev(x), packed, s, z, bits, _lib.PROLOGUE_RMSNORM,
                                          R=dev(r), R_out=hd, w=dev(w), eps=1e-6, config=cfg)
        check_prologue(Y, laq.laq_gemm_wxg128(dev(xin), packed, s, z, bits, config=cfg), xin)
        assert np.array_equal(hd.cpu().numpy(), h)
        Y = _lib.laq_gemm_wxg128_prologue(dev(gu), packed, s, z, bits, _lib.PROLOGUE_SILU_MUL,
                                          config=cfg)
        check_prologue(Y, laq.laq_gemm_wxg128(dev(act), packed, s, z, bits, config=cfg), act)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(2, 4, 1), (1, 2, 3), (2, 8, 8)])
@pytest.mark.parametrize("kind", ["plain", "norm", "silu"])
def test_non_finite_rows_stay_in_their_rows(shape, kind):
    bits, M, K, N = 4, 8, 1408, 336
    q, packed, s, z = prepared(K, N, bits, seed=1)
    w = torch.from_numpy(inputs.norm_weight(K, seed=4)).cuda()
    x = torch.from_numpy(inputs.activations(M, K * (2 if kind == "silu" else 1), seed=2)).cuda()
    r = torch.from_numpy(inputs.activations(M, K, seed=3)).cuda()

    def run(x):
        if kind == "plain":
            return laq.laq_gemm_wxg128(x, packed, s, z, bits, config=batch_config(*shape))
        if kind == "silu":
            return _lib.laq_gemm_wxg128_prologue(x, packed, s, z, bits, _lib.PROLOGUE_SILU_MUL,
                                                 config=batch_config(*shape))
        return _lib.laq_gemm_wxg128_prologue(x, packed, s, z, bits, _lib.PROLOGUE_RMSNORM, R=r, w=w,
                                             eps=1e-6, config=batch_config(*shape))
    clean, bad = run(x), x.clone()
    bad[1, 5], bad[4, K - 1], bad[6, 700] = float("inf"), float("nan"), -float("inf")
    Y = run(bad)
    keep = [0, 2, 3, 5, 7]
    assert torch.equal(Y[keep], clean[keep])
    assert not torch.isfinite(Y[4]).any()


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(2, 8, 1), (2, 4, 3), (1, 2, 8)])
@pytest.mark.parametrize("M", [3, 16])
def test_dependent_launches_wait(shape, M):
    """Layers of plain, norm and SiLU calls, each reading what the one before it writes (X, R, gate|up),
    overlapped by programmatic dependent launch and not: the same bits."""
    bits, H, I, layers = 3, 1408, 1024, 12
    o, gu, dn = (prepared(K, N, bits, seed=K + N)[1:] for K, N in ((H, H), (H, 2 * I), (I, H)))
    w = torch.from_numpy(inputs.norm_weight(H, seed=4)).cuda()
    x0 = torch.from_numpy(inputs.activations(M, H, seed=2)).cuda()
    f16 = dict(dtype=torch.float16, device="cuda")

    def run(pdl):
        cfg = batch_config(*shape, pdl)
        res = [torch.zeros((M, H), **f16), torch.empty((M, H), **f16)]
        x, a = x0.clone(), torch.empty((M, H), **f16)
        g, out = torch.empty((M, 2 * I), **f16), []
        torch.cuda.synchronize()
        for layer in range(layers):
            laq.laq_gemm_wxg128(x, *o, bits, Y=a, config=cfg)
            _lib.laq_gemm_wxg128_prologue(a, *gu, bits, _lib.PROLOGUE_RMSNORM, Y=g,
                                          R=res[layer % 2], R_out=res[1 - layer % 2], w=w, eps=1e-6,
                                          config=cfg)
            _lib.laq_gemm_wxg128_prologue(g, *dn, bits, _lib.PROLOGUE_SILU_MUL, Y=x, config=cfg)
        torch.cuda.synchronize()
        return x, res[0], res[1]
    want = run(0)
    assert all(torch.isfinite(t).all() and t.any() for t in want)
    for _ in range(5):
        assert all(torch.equal(p, q) for p, q in zip(run(1), want))


@pytest.mark.gpu
@pytest.mark.parametrize("K,shape", [(4096, (2, 8, 4)), (2560, (2, 4, 2)), (1408, (1, 2, 1))])
def test_norm_prologue_sums_squares_as_exactly_as_the_general_kernel(K, shape):
    """The inverse RMS decides the fp16 rounding of every normalised input; a row in which none
    rounds apart from 64 bits equals the plain GEMM of the exactly normalised row bit for bit.  Out
    of 640 rows 75 to 88 % do with fp32 sums (with the sums of squares on the tensor cores, which
    truncate, 40, 38 and 55 % at these three shapes).  The two counts differ by under 4 standard deviations
    of a difference of binomials, 4 sqrt(2 * 640 / 4) = 72."""
    bits, M, N = 3, 16, 256
    q, packed, s, z = prepared(K, N, bits, seed=K)
    dev = lambda a: torch.from_numpy(a).cuda()
    count = {"batch": 0, "general": 0}
    for seed in range(40):
        x, r = inputs.activations(M, K, seed=100 + seed), inputs.activations(M, K, seed=200 + seed)
        w = inputs.norm_weight(K, seed=300 + seed)
        h = (x.astype(np.float32) + r.astype(np.float32)).astype(np.float16).astype(np.float64)
        xn = (h / np.sqrt(np.square(h).mean(-1, keepdims=True) + 1e-6) * w).astype(np.float16)
        for name, cfg in (("batch", batch_config(*shape)), ("general", laq.GemmConfig.make(8, 8, 1, 4))):
            Y = _lib.laq_gemm_wxg128_prologue(dev(x), packed, s, z, bits, _lib.PROLOGUE_RMSNORM,
                                              R=dev(r), w=dev(w), eps=1e-6, config=cfg)
            Z = laq.laq_gemm_wxg128(dev(xn), packed, s, z, bits, config=cfg)
            count[name] += int((Y == Z).all(-1).sum())
    assert count["batch"] >= count["general"] - 72, count


@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("M", [1, 2, 3, 4, 5, 8, 9, 16])
def test_plan_names_a_valid_batch_shape(bits, M):
    for K, N in ((128, 16), (256, 4096), (1408, 7424), (9728, 2560), (4096, 24576), (2560, 151936),
                 (65535 * 128, 16)):
        for sms in (152, 1):
            c = laq.laq_gemm_plan(M, K, N, bits, sms)
            if M >= 5 or N == 151936:
                assert c.reserved[0] == TAG
            if c.reserved[0]:
                tw, slots, cluster = (c.reserved[1] & 255, c.reserved[1] >> 8 & 255,
                                      c.reserved[1] >> 16)
                assert c.reserved[0] == TAG and tw in (1, 2) and slots in (1, 2, 4, 8)
                assert 1 <= cluster <= min(8, K // 128)


@pytest.mark.parametrize("M,K,N,bits,batch", [
    # where chains of calls time the general kernel the faster one, by up to a third ...
    (4, 512, 12288, 4, False), (4, 1024, 12288, 4, False), (4, 2048, 12288, 4, False),
    (2, 256, 32768, 3, False), (2, 1024, 24576, 4, False), (1, 512, 24576, 4, False),
    (1, 4096, 6144, 4, False), (1, 2560, 40960, 3, False), (3, 8192, 1024, 3, False),
    (4, 9728, 512, 4, False), (3, 9728, 2560, 3, False),
    # ... and where the batch kernel is
    (4, 2560, 19456, 4, True), (4, 9728, 2560, 3, True), (3, 9728, 2560, 4, True),
    (2, 4096, 24576, 3, True), (1, 4096, 24576, 4, True), (1, 12288, 4096, 4, True),
    (3, 256, 32768, 3, True), (1, 2560, 151936, 3, True), (5, 128, 16, 3, True)])
def test_plan_takes_the_faster_kernel(M, K, N, bits, batch):
    assert (laq.laq_gemm_plan(M, K, N, bits, 152).batch is not None) == batch


@pytest.mark.parametrize("M,K,N", [(8, 2048, 1152), (16, 2048, 1152), (8, 3072, 1152), (8, 2048, 1024)])
def test_plan_does_not_fill_the_device_with_short_clusters(M, K, N):
    """Two CTAs per SM of 2 or 3 groups each in clusters of 8 (4.3 us a call at 2048 x 1152 W4 M = 8):
    slower than the general kernel (3.35) and than half the CTAs (3.0)."""
    tw, slots, cluster = laq.laq_gemm_plan(M, K, N, 4, 152).batch
    assert cluster < 7 or -(-(N // 16) // (tw * slots)) * cluster <= 152
