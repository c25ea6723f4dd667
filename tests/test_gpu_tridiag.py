"""The small tridiagonal step at every kind of depth: one step, a breakdown,
the deepest recurrence (needs a GB300)."""
import numpy as np
import pytest

import oracle.communicability as oc
from paper_1409_5000_gb300 import synth
from tests import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 3, 31, 32, 33, 64, 128])
def test_shift_and_scores_at_depth(m):
    """theta is lambda_max of the oracle's T_m to FP64 rounding (1e-13 of its
    size), and the scores meet the FP64 bar.  Reorthogonalised: T_m itself
    agrees only then once the recurrence has converged."""
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    graphs = [synth.er(3001, 9.0 / 3000, 11), synth.ws(700, 8, 0.1, 12), synth.ba(1200, 4, 13),
              synth.from_edges(40, [(i, i + 1) for i in range(39)])]
    with B.GraphSet(graphs) as gs:
        for r, g in enumerate(graphs):
            ls, y = B.communicability(gs, r, m, B.CB_FP64 | B.CB_REORTH)
            th_o, y_o, _ = oc.krylov_expv(g.n, g.row_ptr, g.col, m)
            assert abs(float(ls.item()) - th_o) <= 1e-13 * max(1.0, abs(th_o))
            parity.assert_scores(float(ls.item()), y.cpu().numpy(), th_o, y_o, "fp64")


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("q", [47, 49, 50, 120])
def test_shift_around_the_second_method(q, prec):
    """lambda_max on both sides of where the FP32 recurrences change the method
    for theta: a clique of q nodes (q - 1 and a little) in a sparse graph, whose
    T carries copies of it at this depth.  The suite's parity bars."""
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    rng = np.random.default_rng(q)
    n = 2000
    e = [rng.integers(0, n, (n, 2)), np.array([(a, b) for a in range(q) for b in range(a)])]
    e = np.concatenate(e)
    g = synth.from_edges(n, e[e[:, 0] != e[:, 1]])
    with B.GraphSet([g]) as gs:
        ls, y = B.communicability(gs, 0, 35, prec)
        th_o, y_o, _ = oc.krylov_expv(g.n, g.row_ptr, g.col, 35)
        parity.assert_scores(float(ls.item()), y.cpu().numpy(), th_o, y_o, "fp64" if prec else "fp32")


@pytest.mark.parametrize("graph", [("er", 2001, 0), ("ws", 3500, 8), ("er", 2601, 2), ("ba", 2500, 0)])
def test_shift_is_one_in_both_fp64_modes(graph):
    """While orthogonality holds to rounding T is the same with and without
    reorthogonalisation, so theta and the scaled scores are too: 1e-12 (T's
    rounding, some 1e-15 of lambda_max < 25, through exp(theta) y)."""
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    kind, n, seed = graph
    if kind == "er":
        g = synth.er(n, 9.0 / 2000, seed)
    elif kind == "ba":
        g = synth.ba(n, 5, seed)
    else:
        g = synth.single_background("ws", n, 12, seed).graphs[0]
    with B.GraphSet([g], path=B.CB_PATH_CSR) as gs:
        ls, y = B.communicability(gs, 0, 30, B.CB_FP64)
        ls_r, y_r = B.communicability(gs, 0, 30, B.CB_FP64 | B.CB_REORTH)
    ls, ls_r, y, y_r = float(ls.item()), float(ls_r.item()), y.cpu().numpy(), y_r.cpu().numpy()
    assert abs(ls - ls_r) <= 1e-12 * ls
    assert np.max(np.abs(y - y_r)) <= 1e-12 * y.max()


@pytest.mark.parametrize("q", [20, 30, 40, 47, 49, 50, 80, 120, 200])
def test_fp32_shift_on_both_sides_of_the_methods(q):
    """theta of FP32 recurrences against the oracle's (dense eigensolver on T of a
    reorthogonalised FP64 run), T full of copies of it: within five units of FP32
    roundoff (3e-7, T's own entries) by bracketing, below lambda_max = 48, and
    within the relative step at which the other method's FP32 stage stops (1e-6)
    above."""
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    rng, n = np.random.default_rng(q), 2000
    e = [rng.integers(0, n, (n, 2)), np.array([(a, b) for a in range(q) for b in range(a)])]
    e = np.concatenate(e)
    g = synth.from_edges(n, e[e[:, 0] != e[:, 1]])
    th_o = oc.krylov_expv(g.n, g.row_ptr, g.col, 35)[0]
    with B.GraphSet([g]) as gs:
        th = float(B.communicability(gs, 0, 35, B.CB_FP32)[0].item())
    assert abs(th - th_o) <= (3e-7 if th_o < 47.9 else 1e-6) * th_o
