"""FP64 tiled-CSR SpMV: batches of short, medium and long rows (needs a GB300)."""
import numpy as np
import pytest

import oracle.communicability as oc
from paper_1409_5000_gb300 import synth
from tests import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lanes", [1, 2, 4, 8, 16, 32])
@pytest.mark.parametrize("n_med,n_long", [(0, 1), (31, 3), (33, 4), (70, 9)])
def test_row_batches_match_oracle(lanes, n_med, n_long):
    """Medium rows are summed four at a time per warp and long ones four at a
    time per CTA, short ones in batches of the group width: counts at and past
    full batches, isolated nodes, a ragged last tile.  FP64 bars."""
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    n = 5001
    rng = np.random.default_rng(n_med + n_long)
    e = [rng.integers(200, n, (3 * n, 2))]
    deg = [int(d) for d in rng.integers(257, 1024, n_med)] + [int(d) for d in rng.integers(1025, 3000, n_long)]
    e += [np.stack([np.full(d, 3 + h), rng.choice(np.arange(300, n), d, replace=False)], axis=1) for h, d in enumerate(deg)]
    e = np.concatenate(e)
    g = synth.from_edges(n, e[e[:, 0] != e[:, 1]])
    with B.GraphSet([g], path=B.CB_PATH_CSR) as gs:
        B.cb_graph_set_lanes(gs.h, lanes)
        ls, y = B.communicability(gs, 0, 12, B.CB_FP64)
        th_o, y_o, _ = oc.krylov_expv(g.n, g.row_ptr, g.col, 12)
        parity.assert_scores(float(ls.item()), y.cpu().numpy(), th_o, y_o, "fp64")
