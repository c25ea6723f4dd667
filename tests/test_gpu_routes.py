"""Which route a call takes, where a wrong one costs several times as much:
counted by the launches of one pass, the scores against the per-step kernels
(needs a GB300)."""
import numpy as np
import pytest

from tests import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1409_5000_gb300 import binding

    binding.lib()
    return binding


def _pass(B, gs, m, prec):
    """Scores of one pass and the launches of its recurrence (1: all steps in one)."""
    B.cb_profile_enable(1)
    try:
        ls, S = B.ensemble_scores(gs, m, prec)
        torch.cuda.synchronize()
        return float(ls.item()), S.cpu().numpy(), B.cb_profile_read(B.CB_K_SPMV)[1]
    finally:
        B.cb_profile_enable(0)


@pytest.mark.parametrize("N,n,deg,one", [
    (60, 3000, 40, True),     # columns fit in shared memory: teams
    (140, 1000, 150, True),   # they do not, few entries in all: one CTA each
    (60, 3000, 100, False),   # more: the per-step kernels
    (8, 30_000, 40, False),
    (600, 4000, 12, True),    # fit, whatever the entries of all together
])
def test_columns_beyond_shared_memory(B, N, n, deg, one):
    """FP32 ensembles on both sides of what a CTA can keep.  FP32 parity bars
    against the per-step kernels."""
    m, target = 12, np.array([(0, 1)])
    with B.GraphSet.generate_er([n - q % 5 for q in range(N)], deg, 17, target) as gs:
        ls, S, launches = _pass(B, gs, m, B.CB_FP32)
        B.cb_graph_set_path(gs.h, B.CB_PATH_CSR)
        ls_r, S_r, launches_r = _pass(B, gs, m, B.CB_FP32)
    assert launches_r == m and launches == (1 if one else m)
    parity.assert_scores(ls, S, ls_r, S_r, "fp32")
