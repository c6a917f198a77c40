"""The quantizer's fp32 arithmetic makes the decisions of the exact rule, bit for bit."""
import ctypes

import numpy as np
import pytest

from oracle import c_oracle as co


def _f32(x):
    return np.asarray(x, np.float64).astype(np.float32)


@pytest.mark.parametrize("qmax", [7, 15])
def test_corrected_quotient_rounds_like_the_exact_one(qmax):
    """Every pair of fp16 significands and every exponent difference at which |w| / s lies in
    1/8 .. qmax + 1/2 (below, the quotient rounds to 0 with room to spare): the one-step corrected
    fp32 quotient, rounded half to even, equals the exactly rounded w / s.  Powers of two scale
    both sides alike, so s in [1, 2) stands for every normal s.  The products and residuals are
    exact in fp64, so rounding them to fp32 restates the kernel's single-rounded fma."""
    s = _f32(1 + np.arange(1024) / 1024.0)
    inv = _f32(1.0 / s.astype(np.float64))
    for e in range(-3, 4):
        w = _f32((1 + np.arange(1024) / 1024.0) * 2.0 ** e)
        W, S, I = (a.astype(np.float64) for a in np.broadcast_arrays(w[None], s[:, None],
                                                                     inv[:, None]))
        q = _f32(W * I).astype(np.float64)
        r = _f32(W - q * S).astype(np.float64)
        c = _f32(q + r * I).astype(np.float64)
        ok = 2 * W <= (2 * qmax + 1) * S
        assert np.array_equal(np.rint(c)[ok], np.rint(W / S)[ok])


def _matrix(K, N, seed):
    """fp16 columns of every magnitude: random bit patterns, narrow exponent ranges, one-signed
    and constant columns, and ranges whose end points are far apart."""
    rng = np.random.default_rng(seed)
    W = rng.integers(0, 1 << 16, size=(K, N)).astype(np.uint16)
    exp = rng.integers(0, 31, size=N)
    narrow = rng.random(N) < 0.5
    W[:, narrow] = (W[:, narrow] & 0x83ff) | (exp[narrow] << 10).astype(np.uint16)
    W[(W & 0x7c00) == 0x7c00] &= 0xbbff          # finite only
    W[:, rng.random(N) < 0.1] &= 0x7fff          # one sign
    W[:, rng.random(N) < 0.1] = 0x8001           # a constant, subnormal
    far = rng.random(N) < 0.1
    W[:, far] = 0x7bff
    W[0, far] = 0x8000 | rng.integers(1, 0x400, size=int(far.sum())).astype(np.uint16)
    return W.view(np.float16)


@pytest.mark.gpu
@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("K,N,offset", [(128, 1, 0), (128, 127, 0), (256, 130, 0), (384, 4096, 0),
                                        (256, 132, 1), (128, 160, 2), (256, 272, 4)])
def test_quantizer_at_edges(bits, K, N, offset):
    """Ragged and unaligned matrices (offset: elements past an aligned start) of all magnitudes."""
    import torch
    from paper_2605_08755_gb300 import _lib, build
    build.build()
    W = _matrix(K, N, seed=K + N + offset)
    buf = torch.zeros(K * N + offset, dtype=torch.float16, device="cuda")
    buf[offset:] = torch.from_numpy(W).cuda().flatten()
    G = K // 128
    codes = torch.zeros(K * N + offset, dtype=torch.uint8, device="cuda")
    s = torch.empty((G, N), dtype=torch.float16, device="cuda")
    z = torch.empty((G, N), dtype=torch.uint8, device="cuda")
    st = _lib.lib().laq_quantize_rtn(
        ctypes.c_void_p(buf.data_ptr() + 2 * offset), K, N, bits, 128,
        ctypes.c_void_p(codes.data_ptr() + offset), ctypes.c_void_p(s.data_ptr()),
        ctypes.c_void_p(z.data_ptr()), None)
    assert st == 0
    torch.cuda.synchronize()
    rc, rs, rz = co.quantize_rtn(W, bits)
    assert np.array_equal(s.cpu().numpy().view(np.uint16), rs.view(np.uint16))
    assert np.array_equal(z.cpu().numpy(), rz)
    assert np.array_equal(codes[offset:].view(K, N).cpu().numpy(), rc)


@pytest.mark.gpu
@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("K,N,offset", [(128, 16, 0), (256, 112, 0), (384, 4096, 0), (256, 144, 1),
                                        (128, 272, 2), (256, 1040, 4)])
def test_fused_quantize_pack_at_edges(bits, K, N, offset):
    """The packed records, scales and zeros are those of the quantizer and packer of the oracle."""
    import torch
    from paper_2605_08755_gb300 import _lib, build
    build.build()
    W = _matrix(K, N, seed=K + N + offset)
    buf = torch.zeros(K * N + offset, dtype=torch.float16, device="cuda")
    buf[offset:] = torch.from_numpy(W).cuda().flatten()
    packed, s, z = _lib.laq_quantize_pack(buf[offset:].view(K, N), bits)
    torch.cuda.synchronize()
    rc, rs, rz = co.quantize_rtn(W, bits)
    assert np.array_equal(packed.cpu().numpy().view(np.uint32), co.pack(rc, bits))
    assert np.array_equal(s.cpu().numpy().view(np.uint16), rs.view(np.uint16))
    assert np.array_equal(z.cpu().numpy(), rz)


@pytest.mark.gpu
@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("K,N,offset", [(128, 16, 0), (256, 112, 0), (128, 144, 1), (384, 272, 2),
                                        (256, 1040, 4)])
def test_pack_and_unpack_at_edges(bits, K, N, offset):
    """Ragged column blocks and codes at any address."""
    import torch
    from paper_2605_08755_gb300 import _lib, build
    build.build()
    rng = np.random.default_rng(K * N + bits + offset)
    c = rng.integers(0, 1 << bits, size=(K, N)).astype(np.uint8)
    codes = torch.zeros(K * N + offset, dtype=torch.uint8, device="cuda")
    codes[offset:] = torch.from_numpy(c).cuda().flatten()
    packed = torch.empty(K * N * bits // 8, dtype=torch.uint8, device="cuda")
    L = _lib.lib()
    assert L.laq_pack(ctypes.c_void_p(codes.data_ptr() + offset), K, N, bits,
                      ctypes.c_void_p(packed.data_ptr()), None) == 0
    back = torch.zeros_like(codes)
    assert L.laq_unpack(ctypes.c_void_p(packed.data_ptr()), K, N, bits,
                        ctypes.c_void_p(back.data_ptr() + offset), None) == 0
    torch.cuda.synchronize()
    assert np.array_equal(packed.cpu().numpy().view(np.uint32), co.pack(c, bits))
    assert torch.equal(back, codes)
