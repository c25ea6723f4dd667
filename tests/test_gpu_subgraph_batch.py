"""Sub-graph centrality of batches of start nodes: batch edges, rows summed by
a warp and by the CTA, vectors that stop early beside others (needs a GB300)."""
import numpy as np
import pytest

import oracle.communicability as oc
from paper_1409_5000_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("k", [1, 31, 32, 33, 70])
def test_batches_match_oracle(k, prec):
    """Against the oracle's Gauss rule per node: relative error in units of the
    largest value (the accuracy the rule promises), 1e-4 in FP32, 1e-11 in FP64."""
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    rng = np.random.default_rng(k)
    n, m = 4001, 12
    e = [rng.integers(50, n, (2 * n, 2)), [(1, 2), (3, 4), (4, 5), (3, 5)]]  # nodes 0, 6..49 isolated but for hubs
    e += [np.stack([np.full(d, h), rng.choice(np.arange(100, n), d, replace=False)], axis=1)
          for h, d in ((60, 1500), (61, 257), (62, 256))]
    e = np.concatenate([np.asarray(x) for x in e])
    g = synth.from_edges(n, e[e[:, 0] != e[:, 1]])
    nodes = [0, 1, 3, 60, 61, 62][:k] + [int(x) for x in rng.integers(50, n, max(0, k - 6))]
    with B.GraphSet([synth.er(300, 0.02, 1), g]) as gs:
        ls, sc = B.subgraph_centrality(gs, 1, m, nodes, prec)
        th, c0 = oc.subgraph_centrality_krylov(g.n, g.row_ptr, g.col, nodes, m)
        ref = np.exp(th) * c0
        got = sc.cpu().numpy() * np.exp(float(ls.item()))
    assert np.max(np.abs(got - ref)) <= (1e-11 if prec else 1e-4) * ref.max()
