"""The one-launch recurrence (teams of CTAs) at its edges, against the oracle:
teams of one and of many, rows for a lane, a warp and the CTA, empty rows,
16- and 32-bit columns, breakdowns, the most realisations (needs a GB300).

Bars: the suite's (parity.py) against the oracle; with reorthogonalisation in
FP64 the per-step kernels run the same scheme in another order of sums, so the
scores of the two agree to 1e-12 (sums of at most 1e4 terms of relative rounding
1.1e-16, and the head's scores are within 1e3 of each other)."""
import numpy as np
import pytest

import oracle.communicability as oc
from paper_1409_5000_gb300 import synth
from tests import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _hubs(n, hubs, seed):
    """An ER graph with a few nodes joined to many others."""
    rng = np.random.default_rng(seed)
    e = [rng.integers(0, n, (3 * n, 2))]
    for h, d in enumerate(hubs):
        e.append(np.stack([np.full(d, h), rng.choice(np.arange(len(hubs), n), d, replace=False)], axis=1))
    e = np.concatenate(e)
    return synth.from_edges(n, e[e[:, 0] != e[:, 1]])


def _sets():
    er = lambda n, d, s: synth.er(n, d / max(n - 1, 1), s)  # noqa: E731
    k7 = synth.from_edges(7, [(i, j) for i in range(7) for j in range(i)])
    return {
        "tiny": [synth.from_edges(1, np.zeros((0, 2))), synth.from_edges(2, [(0, 1)]), k7, er(33, 4, 1)],
        "one": [er(8191, 6, 2)],
        "uneven": [er(n, 9, n) for n in (500, 1023, 1025, 4097, 8192)],
        "hubs": [_hubs(7001, (6000, 2049, 2048, 1025, 600, 300), 3), er(300, 5, 4)],
        "large": [er(30_011, 12, 5), _hubs(20_003, (9000, 3000), 6)],
        "wide": [er(70_001, 8, 7), er(66_000, 3, 8)],
        "most": [er(200 + q, 6, q) for q in range(160)],
        "beyond": [er(150 + q, 6, q) for q in range(161)],
    }


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("name", sorted(_sets()))
def test_matches_oracle(name, prec):
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    graphs = _sets()[name]
    m, p = 15, (B.CB_FP32 if prec == "fp32" else B.CB_FP64 | B.CB_REORTH)
    th_o, S_o = oc.ensemble_scores([(g.n, g.row_ptr, g.col) for g in graphs], m)
    with B.GraphSet(graphs) as gs:
        ls, S, rep = B.ensemble_scores(gs, m, p, report=True)
        parity.assert_scores(float(ls.item()), S.cpu().numpy(), th_o, S_o, prec)
        if prec == "fp64":
            with B.GraphSet(graphs, path=B.CB_PATH_CSR) as ref:
                ls_r, S_r = B.ensemble_scores(ref, m, p)
            e = parity.errors(float(ls.item()), S.cpu().numpy(), float(ls_r.item()), S_r.cpu().numpy())
            assert e["head_rel"] <= 1e-12 and e["norm_rel"] <= 1e-12, e
        if name == "tiny":  # breakdowns: an empty graph, K_2 and K_7 are spanned by 1
            assert [r.m_eff for r in rep[:3]] == [1, 1, 1]
        again = B.ensemble_scores(gs, m, p)[1]
        assert torch.equal(S, again)


@pytest.mark.parametrize("sizes", [(9000, 12000), (2500, 3000)])
def test_ensembles_with_hubs_keep_the_order(sizes):
    """FP32 ensembles whose leading eigenvector sits on a few hubs: above the
    small size the automatic path gives the bits of the per-step kernels; all
    meet the suite's bars against the oracle."""
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    graphs = [synth.ba(n, 10, 3 + q) for q, n in enumerate(sizes)]
    th_o, S_o = oc.ensemble_scores([(g.n, g.row_ptr, g.col) for g in graphs], 17)
    got = []
    for path in (B.CB_PATH_AUTO, B.CB_PATH_CSR):
        with B.GraphSet(graphs, path=path) as gs:
            ls, S = B.ensemble_scores(gs, 17, B.CB_FP32)
            got.append((float(ls.item()), S.cpu().numpy()))
        parity.assert_scores(*got[-1], th_o, S_o, "fp32")
    if min(sizes) > 8192:
        assert got[0][0] == got[1][0] and np.array_equal(got[0][1], got[1][1])


@pytest.mark.parametrize("seed", [1, 2, 3, 4])
def test_beta_to_fp64_rounding(seed):
    """One step on 4^5 nodes of mean degree 8 is exact but for the root: the
    entries of w are (degree - 8) / 32, their squares and sums few bits, so beta is
    the root of a known number, to two units in FP64's last place, also in FP32."""
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    n, rng = 1024, np.random.default_rng(seed)
    u, v = np.triu_indices(n, 1)
    at = rng.choice(len(u), 4 * n, replace=False)
    g = synth.from_edges(n, np.stack([u[at], v[at]], axis=1))
    deg = np.diff(g.row_ptr.astype(np.int64))
    assert deg.sum() == 8 * n
    with B.GraphSet([g]) as gs:
        beta = B.ensemble_scores(gs, 1, B.CB_FP32, report=True)[2][0].beta_last
    ref = np.sqrt(float(((deg - 8) ** 2).sum()) / n)
    assert abs(beta - ref) <= 2 * np.spacing(ref)


def test_small_ensembles_to_fp32_rounding():
    """Scaled scores of ten 500-node graphs against the oracle's, 16 seeds: on
    average within two FP32 units of roundoff (2 x 6e-8), one for theta, which
    shifts them all, and one for the sums."""
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    err = []
    for seed in range(16):
        graphs = [synth.er(500, 8.0 / 499, 100 * seed + q) for q in range(10)]
        _, S_o = oc.ensemble_scores([(g.n, g.row_ptr, g.col) for g in graphs], 20)
        with B.GraphSet(graphs) as gs:
            S = B.ensemble_scores(gs, 20, B.CB_FP32)[1].float().double().cpu().numpy()
        err.append(np.linalg.norm(S - S_o) / np.linalg.norm(S_o))
    assert np.mean(err) <= 1.2e-7, err


def _is_hub(g):
    deg = np.diff(g.row_ptr.astype(np.int64))
    return deg.max() > 8 * (deg.sum() // g.n) + 64


@pytest.mark.parametrize("name", ["warp rows", "cta rows"])
def test_long_rows_in_fp32(name):
    """FP32 graphs without hubs, which the team kernel takes, whose rows are still
    too long for the lanes of a row: 1000 rows a CTA and one lane a row, some of
    them above 32 entries (few enough for the list); a dense graph of teams with
    rows above 1024 and above 2048."""
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    if name == "warp rows":
        graphs = [synth.er(1000, 24.0 / 999, 900 + q) for q in range(160)]  # more than SMs: a CTA each
        over = [int((np.diff(g.row_ptr.astype(np.int64)) > 32).sum()) for g in graphs]
        assert sum(0 < c <= 64 for c in over) > 100
    else:
        rng, n = np.random.default_rng(9), 3000
        base = synth.er(n, 270.0 / n, 31)
        src = np.repeat(np.arange(n), np.diff(base.row_ptr.astype(np.int64)))
        e = [np.stack([src, base.col.astype(np.int64)], axis=1)]
        e += [np.stack([np.full(d, h), rng.choice(np.arange(10, n), d, replace=False)], axis=1)
              for h, d in ((3, 1400), (4, 2100))]
        e = np.concatenate(e)
        graphs = [synth.from_edges(n, e[e[:, 0] != e[:, 1]])]
        deg = np.diff(graphs[0].row_ptr.astype(np.int64))
        assert deg[3] > 1024 and deg[4] > 2048
    assert not any(_is_hub(g) for g in graphs)
    m = 12
    th_o, S_o = oc.ensemble_scores([(g.n, g.row_ptr, g.col) for g in graphs], m)
    with B.GraphSet(graphs) as gs:
        B.cb_profile_enable(1)
        ls, S = B.ensemble_scores(gs, m, B.CB_FP32)
        torch.cuda.synchronize()
        launches = B.cb_profile_read(B.CB_K_SPMV)[1]
        B.cb_profile_enable(0)
        assert launches == 1
        parity.assert_scores(float(ls.item()), S.cpu().numpy(), th_o, S_o, "fp32")
