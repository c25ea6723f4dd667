"""Sums over many tiles and realisations: the norm's group sums by one lane
per group, the ensemble sum's grid of resident CTAs (needs a GB300)."""
import numpy as np
import pytest

import oracle.communicability as oc
from paper_1409_5000_gb300 import synth
from tests import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(graphs, m, prec):
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    th_o, S_o = oc.ensemble_scores([(g.n, g.row_ptr, g.col) for g in graphs], m)
    with B.GraphSet(graphs) as gs:
        ls, S = B.ensemble_scores(gs, m, prec)
        parity.assert_scores(float(ls.item()), S.cpu().numpy(), th_o, S_o, "fp64" if prec else "fp32")


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("groups", [23, 24, 25, 33])
def test_norm_group_edges(groups, prec):
    """One group of 32 finalize tiles of 2048 nodes more or less than where the
    one-lane-per-group sum starts, the last group of one slot with a ragged tile;
    the suite's parity bars against the oracle."""
    n = (groups - 1) * 32 * 2048 + 5
    rng = np.random.default_rng(groups)
    e = rng.integers(0, n, (n // 2, 2))
    _check([synth.from_edges(n, e[e[:, 0] != e[:, 1]])], 4, prec)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n_inst,n", [(1, 256), (9, 257), (3000, 40), (2, 700_001)])
def test_ensemble_sum_grid(n_inst, n, prec):
    """Fewer nodes than resident CTAs and more, one realisation and many;
    isolated nodes, whose terms FP32 rounds to zero or below its normal range,
    beside the others."""
    graphs = [synth.er(n - (q % 7), 4.0 / n, 50 + q) for q in range(n_inst)]
    _check(graphs, 5, prec)
