"""Which route a call takes, where a wrong one costs several times as much:
counted by the launches of one pass, the scores against the per-step kernels
(needs a GB300)."""
import numpy as np
import pytest

import oracle.communicability as oc
from paper_1409_5000_gb300 import synth
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


@pytest.mark.parametrize("k", [1, 2])
def test_centrality_of_a_few_nodes_in_little_memory(B, k):
    """32 vectors of a graph of 2e5 nodes take 77 MB, k copies of graph, format
    and basis about 25 k: with 64 MB left, one node and two still run."""
    n, m = 200_000, 12
    g = synth.er(n, 6.0 / n, 3)
    th, c0 = oc.subgraph_centrality_krylov(g.n, g.row_ptr, g.col, list(range(k)), m)
    with B.GraphSet([g]) as gs:
        torch.cuda.synchronize()
        base = B.cb_memory_in_use()
        try:
            B.cb_set_memory_limit(base + (64 << 20))
            ls, sc = B.subgraph_centrality(gs, 0, m, list(range(k)), B.CB_FP32)
        finally:
            B.cb_set_memory_limit(0)
        assert B.cb_memory_in_use() == base
        got = sc.cpu().numpy() * np.exp(float(ls.item()))
    ref = np.exp(th) * c0
    assert np.max(np.abs(got - ref)) <= 1e-4 * ref.max()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("k,links,copies", [(1, 2, True), (7, 2, True), (64, 2, True), (64, 45, False)])
def test_centrality_beside_a_heavy_row(B, k, links, copies, prec):
    """A row that the SpMV cuts over CTAs (more than 8192 entries): few start
    nodes, or many in a graph of little else, by copies of the graph, whose
    recurrence the profile counts; many by 32 vectors, whose kernels it does not.  Against the oracle's Gauss rule, in
    units of the largest value, 1e-4 in FP32 and 1e-11 in FP64."""
    n, m = 20_000, 10
    rng = np.random.default_rng(4)
    e = np.concatenate([rng.integers(1, n, (links * n, 2)),
                        np.stack([np.zeros(9000, np.int64), rng.choice(np.arange(1, n), 9000, replace=False)], axis=1)])
    g = synth.from_edges(n, e[e[:, 0] != e[:, 1]])
    nodes = [0] + [int(x) for x in rng.choice(np.arange(1, n), k - 1, replace=False)]
    with B.GraphSet([g]) as gs:
        B.cb_profile_enable(1)
        try:
            ls, sc = B.subgraph_centrality(gs, 0, m, nodes, prec)
            launches = B.cb_profile_read(B.CB_K_SPMV)[1]
        finally:
            B.cb_profile_enable(0)
        got = sc.cpu().numpy()
    assert (launches > 0) == copies
    th, c0 = oc.subgraph_centrality_krylov(g.n, g.row_ptr, g.col, nodes, m)
    top = th.max() if hasattr(th, "max") else th
    ref = np.exp(th - top) * c0  # the hub's lambda is 95: no plain exponentials
    got = got * np.exp(float(ls.item()) - top)
    assert np.max(np.abs(got - ref)) <= (1e-11 if prec else 1e-4) * ref.max()


def test_tuning_keeps_the_one_launch(B):
    """Eight graphs of 30 000 nodes run fastest in one launch: the tuner times that
    beside the per-step paths, keeps it, and the path read back and set on
    another handle, as from a cache, is the same."""
    sizes, target = [30_000] * 8, np.array([(0, 1)])
    with B.GraphSet.generate_er(sizes, 12, 5, target) as gs:
        lanes, ms = B.cb_graph_tune(gs.h, B.CB_FP32, 0)
        assert all(x >= 0 for x in ms) and ms[7] == min(ms)
        path = B.cb_graph_path(gs.h)
        ls, S, launches = _pass(B, gs, 10, B.CB_FP32)
        assert launches == 1 and path == B.CB_PATH_AUTO
    with B.GraphSet.generate_er(sizes, 12, 5, target) as gs:
        B.cb_graph_set_lanes(gs.h, lanes)
        B.cb_graph_set_path(gs.h, path)
        ls_2, S_2, launches = _pass(B, gs, 10, B.CB_FP32)
    assert launches == 1 and ls_2 == ls and np.array_equal(S_2, S)


def test_tuning_fp32_leaves_fp64_alone(B):
    """One larger graph: FP32 keeps a per-step path, reorthogonalised FP64 its one
    launch; a path that the caller sets holds for both."""
    with B.GraphSet.generate_er([60_000], 10, 6, np.array([(0, 1)])) as gs:
        p64 = B.CB_FP64 | B.CB_REORTH
        ls, S, launches = _pass(B, gs, 10, p64)
        assert launches == 1
        for _ in range(3):
            B.cb_graph_tune(gs.h, B.CB_FP32, 0)
            assert B.cb_graph_path(gs.h) in (B.CB_PATH_FORMATS, B.CB_PATH_CSR)
            assert _pass(B, gs, 10, B.CB_FP32)[2] == 10
            ls_t, S_t, launches = _pass(B, gs, 10, p64)
            assert launches == 1 and ls_t == ls and np.array_equal(S_t, S)
        B.cb_graph_set_path(gs.h, B.CB_PATH_CSR)
        assert _pass(B, gs, 10, p64)[2] == 10
