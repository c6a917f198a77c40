"""The argmax's split of a row over a cluster: every part, its edges, ties across parts."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import decoder as dec  # noqa: E402
from paper_2605_08755_gb300 import _lib  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2605_08755_gb300 import build
    build.build()


@pytest.mark.parametrize("V", [1, 8, 8191, 32768, 32776, 49153, 65537, 98312, 151936, 262144])
@pytest.mark.parametrize("M", [1, 4, 16, 17])
def test_argmax_parts(V, M):
    rng = np.random.default_rng(V + M)
    x = rng.standard_normal((M, V)).astype(np.float16)
    for m in range(M):
        if m % 4 == 0:      # a winner at a part's first or last element
            k = rng.integers(0, 9)
            x[m, min(V - 1, max(0, V * k // 8 - (m // 4) % 2))] = 9.0
        elif m % 4 == 1:    # equal winners in several parts: the smallest index
            x[m, rng.integers(0, V, 5)] = 9.0
        elif m % 4 == 2:    # nothing above -inf, NaN in between
            x[m] = -np.inf
            x[m, rng.integers(0, V)] = np.nan
    got = _lib.laq_argmax(torch.from_numpy(x).cuda())
    assert list(got.cpu().numpy()) == list(dec.argmax(x))
