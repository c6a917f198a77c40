"""The one-row RMSNorm prologue where its register pass begins and ends: rows of up to one staging
unit per thread (one pass), longer rows and clusters (two passes), one group and ragged units."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2605_08755_gb300 as laq  # noqa: E402
from oracle import c_oracle as co  # noqa: E402
from paper_2605_08755_gb300 import _lib, inputs  # noqa: E402
from tests.test_gpu_gemm_batch import check_prologue  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2605_08755_gb300 import build
    build.build()


@pytest.mark.parametrize("bits", [3, 4])
@pytest.mark.parametrize("K,cfg", [(128, (1, 1, 1, 2)), (1024, (1, 1, 1, 4)), (1152, (1, 1, 1, 4)), (512, (1, 2, 1, 4)), (4096, (1, 8, 1, 3)), (4224, (1, 8, 1, 3)),
                                   (2560, (4, 8, 1, 6)), (2688, (2, 8, 1, 6)), (8192, (1, 8, 1, 3)),
                                   (8320, (1, 8, 1, 3)), (2560, (2, 4, 2, 3)), (256, (1, 2, 8, 3)), (2560, None)])
@pytest.mark.parametrize("with_r", [False, True])
def test_one_row(bits, K, cfg, with_r):
    N = 80
    W = inputs.weights(K, N, seed=K)
    q = co.quantize_rtn(W, bits)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    packed = dev(co.pack(q[0], bits).view(np.uint8))
    s, z = dev(q[1].view(np.uint16)).view(torch.float16), dev(q[2])
    x, r = inputs.activations(1, K, seed=K + 1), inputs.activations(1, K, seed=K + 2)
    w = inputs.norm_weight(K, seed=K + 3)
    h_out = torch.full((1, K), float("nan"), dtype=torch.float16, device="cuda")
    Y = _lib.laq_gemm_wxg128_prologue(dev(x), packed, s, z, bits, _lib.PROLOGUE_RMSNORM,
                                      R=dev(r) if with_r else None, R_out=h_out, w=dev(w),
                                      eps=1e-6, config=cfg and laq.GemmConfig.make(*cfg))
    torch.cuda.synchronize()
    # h is one fp16 sum: exact
    exact = x.astype(np.float32) + (r.astype(np.float32) if with_r else 0)
    assert np.array_equal(h_out.cpu().numpy(), exact.astype(np.float16))
    # against the plain GEMV of the input normalised in 64 bits, same configuration
    xin = (exact.astype(np.float16).astype(np.float64)
           / np.sqrt(np.square(exact.astype(np.float16).astype(np.float64)).mean() + 1e-6)
           * w).astype(np.float16)
    Z = laq.laq_gemm_wxg128(dev(xin), packed, s, z, bits, config=cfg and laq.GemmConfig.make(*cfg))
    check_prologue(Y, Z, xin)
