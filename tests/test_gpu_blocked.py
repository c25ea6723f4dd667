"""Column-blocked SpMV: streams of 0 to many rounds, empty column blocks,
realisations that stop early beside others (needs a GB300)."""
import numpy as np
import pytest

import oracle.communicability as oc
from paper_1409_5000_gb300 import synth
from tests import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deg", [0.02, 1.0, 4.0, 9.0, 17.0, 40.0])
@pytest.mark.parametrize("n", [31, 16_384, 40_001])
def test_stream_lengths_match_oracle(n, deg):
    """A warp's stream of a block is cut into rounds of four pairs of steps and
    loaded two rounds ahead across blocks: mean degrees from all but none to
    several rounds, with a ring beside them (its start vector is an eigenvector,
    so it stops after one step) and entries in one corner (every other block
    empty).  FP32 parity bars against the oracle."""
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    g = synth.er(n, min(1.0, deg / n), 5)
    k = 20_000
    corner = synth.er(300, 0.03, 6)
    src = np.repeat(np.arange(300), np.diff(corner.row_ptr.astype(np.int64)))
    far = synth.from_edges(k, [(k - 1 - int(a), k - 1 - int(b)) for a, b in zip(src, corner.col) if a < b])
    ring = synth.from_edges(1000, [(i, (i + 1) % 1000) for i in range(1000)])
    graphs = [ring, g, far]
    th_o, S_o = oc.ensemble_scores([(q.n, q.row_ptr, q.col) for q in graphs], 15)
    with B.GraphSet(graphs, path=B.CB_PATH_FORMATS) as gs:
        ls, S = B.ensemble_scores(gs, 15, B.CB_FP32)
        parity.assert_scores(float(ls.item()), S.cpu().numpy(), th_o, S_o, "fp32")


@pytest.mark.parametrize("d", [9, 30, 31, 250, 511])
def test_rows_as_long_as_their_stream(d):
    """Rows that fill a stream's steps, so that a run goes on from one lane's
    last step to the next lane's first: no step may add twice into one sum.
    Hubs of d entries beside rows of a few, FP32 parity bars against the oracle."""
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    n = 3000
    rng = np.random.default_rng(d)
    e = [rng.integers(0, n, (n // 2, 2))]
    e += [np.stack([np.full(d, h), rng.choice(np.arange(200, n), d, replace=False)], axis=1) for h in (3, 4, 40, 41, 77)]
    e = np.concatenate(e)
    graphs = [synth.from_edges(n, e[e[:, 0] != e[:, 1]]), synth.er(500, 0.02, d)]
    th_o, S_o = oc.ensemble_scores([(q.n, q.row_ptr, q.col) for q in graphs], 15)
    with B.GraphSet(graphs, path=B.CB_PATH_FORMATS) as gs:
        ls, S = B.ensemble_scores(gs, 15, B.CB_FP32)
        parity.assert_scores(float(ls.item()), S.cpu().numpy(), th_o, S_o, "fp32")


@pytest.mark.parametrize("d", [64, 120, 250, 440])
def test_long_runs_without_hubs(d):
    """The same in graphs dense enough that rows of d entries are no hubs, so that
    their streams are dealt out of lane order and ordered by bank: a row's run of
    up to 511 entries goes on over lanes and rounds, and no step may add twice
    into one sum.  FP32 parity bars against the oracle."""
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    n, rng = 3000, np.random.default_rng(d)
    base = synth.er(n, 60.0 / n, d)
    src = np.repeat(np.arange(n), np.diff(base.row_ptr.astype(np.int64)))
    e = [np.stack([src, base.col.astype(np.int64)], axis=1)]
    e += [np.stack([np.full(d, h), rng.choice(np.arange(200, n), d, replace=False)], axis=1) for h in (3, 4, 40, 41, 77)]
    e = np.concatenate(e)
    g = synth.from_edges(n, e[e[:, 0] != e[:, 1]])
    deg = np.diff(g.row_ptr.astype(np.int64))
    assert deg.max() <= min(8 * (deg.sum() // n) + 64, 512)  # no hub, and none too long for the streams
    graphs = [g, synth.er(20_000, 70.0 / 20_000, d + 1)]
    th_o, S_o = oc.ensemble_scores([(q.n, q.row_ptr, q.col) for q in graphs], 15)
    with B.GraphSet(graphs, path=B.CB_PATH_FORMATS) as gs:
        ls, S = B.ensemble_scores(gs, 15, B.CB_FP32)
        parity.assert_scores(float(ls.item()), S.cpu().numpy(), th_o, S_o, "fp32")
