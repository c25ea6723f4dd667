"""Top-k selection at the edges of its routes: one CTA or a grid, the
threshold from the threads' maxima or the composite radix select, both sorts
(needs a GB300)."""
import numpy as np
import pytest

import oracle.communicability as oc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1409_5000_gb300 import binding

    binding.lib()
    return binding


def _scores(n, kind):
    rng = np.random.default_rng(n)
    if kind == "spread":
        return np.exp(6 * rng.normal(size=n))
    if kind == "ties":  # more equal scores than candidates one CTA sorts
        return rng.integers(0, 3, size=n).astype(np.float64)
    if kind == "equal":
        return np.zeros(n)
    s = rng.normal(size=n)  # signs, both zeros, infinities, NaN and subnormals
    s[rng.integers(0, n, size=n // 8 + 1)] = rng.choice([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324],
                                                        size=n // 8 + 1)
    return s


@pytest.mark.parametrize("kind", ["spread", "ties", "equal", "special"])
@pytest.mark.parametrize("n", [1, 33, 1024, 4096, 4097, 8193, 155_649, 700_001])
def test_matches_full_sort(B, n, kind):
    S = _scores(n, kind)
    d = torch.from_numpy(S).cuda()
    for k in sorted({1, min(n, 20), min(n, 256), min(n, 1025), min(n, 4096)}):
        idx, val = B.topk(d, k)
        key = np.where(np.isnan(S), -np.inf, S)  # NaN after -inf, ties to the smaller index
        ref = np.lexsort((np.arange(n), np.isnan(S), -key))[:k]
        assert np.array_equal(idx.cpu().numpy().astype(np.int64), ref)
        assert np.array_equal(val.cpu().numpy(), S[ref], equal_nan=True)
        if kind in ("spread", "ties"):
            assert np.array_equal(ref, oc.topk(S, k)[0])
