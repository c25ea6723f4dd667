"""Barriers between the CTAs of a launch that run out (needs a GB300; no GPU
fault, trap or hang): the hook cb_debug_stall_barrier keeps one CTA from
arriving and shortens the wait to 20 ms.  The top-k then selects on one CTA and
returns the same; a realisation of the one-launch recurrence reports
CB_ERR_TIMEOUT; the next calls are as ever."""
import math
import time

import numpy as np
import pytest

from paper_1409_5000_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_1409_5000_gb300 import binding

    binding.lib()
    return binding


@pytest.fixture
def stall(B):
    yield lambda: B.cb_debug_stall_barrier(20)
    B.cb_debug_stall_barrier(0)


@pytest.mark.parametrize("kind", ["spread", "ties"])
@pytest.mark.parametrize("n", [4096, 4097, 155_649, 700_001])
def test_topk_whose_barrier_runs_out(B, stall, n, kind):
    rng = np.random.default_rng(n)
    S = np.exp(6 * rng.normal(size=n)) if kind == "spread" else rng.integers(0, 3, size=n).astype(np.float64)
    d = torch.from_numpy(S).cuda()
    order = np.lexsort((np.arange(n), -S))
    for k in (1, 20, 1025, 4096):
        for on in (False, True, False):
            if on:
                stall()
            idx, val = B.topk(d, k)
            B.cb_debug_stall_barrier(0)
            assert np.array_equal(idx.cpu().numpy().astype(np.int64), order[:k])
            assert np.array_equal(val.cpu().numpy(), S[order[:k]])


@pytest.mark.parametrize("prec", ["fp32", "fp64 reorthogonalised"])
def test_recurrence_whose_barrier_runs_out(B, stall, prec):
    graphs = [synth.er(n, 10.0 / n, n) for n in (30_000, 12_000, 25_000)]
    p = B.CB_FP32 if prec == "fp32" else B.CB_FP64 | B.CB_REORTH
    with B.GraphSet(graphs) as gs:
        def run(report=True):
            S = torch.empty(gs.n_max, dtype=torch.float64, device="cuda")
            ls = torch.empty(1, dtype=torch.float64, device="cuda")
            rep, err = (B.InstReport * 3)() if report else None, None
            try:
                B.cb_ensemble_scores(gs.h, 12, p, gs.n_max, S.data_ptr(), ls.data_ptr(), rep,
                                     torch.cuda.current_stream().cuda_stream)
            except B.CBError as e:
                err = e
            torch.cuda.synchronize()
            return err, float(ls.item()), S.cpu().numpy(), rep

        B.cb_profile_enable(1)
        err, ls_ref, S_ref, _ = run()
        assert err is None and B.cb_profile_read(B.CB_K_SPMV)[1] == 1  # one launch
        B.cb_profile_enable(0)
        run(False), run(False)  # a captured pass
        stall()
        for report in (True, False):
            t0 = time.perf_counter()
            err, ls, S, rep = run(report)
            assert time.perf_counter() - t0 < 2.0
            assert math.isnan(ls) and np.all(np.isnan(S))
            if report:
                assert err is not None and err.code == B.CB_ERR_TIMEOUT and "barrier" in str(err)
                assert [r.status for r in rep] == [B.CB_ERR_TIMEOUT] * 3 and [r.m_eff for r in rep] == [0] * 3
        B.cb_debug_stall_barrier(0)
        for report in (True, False, False):
            err, ls, S, _ = run(report)
            assert err is None and ls == ls_ref and np.array_equal(S, S_ref)


def test_limits(B):
    with pytest.raises(B.CBError):
        B.cb_debug_stall_barrier(4001)
