"""Uploads whose host scans share the helper threads (needs a GB300)."""
import threading
import time

import numpy as np
import pytest

from paper_1409_5000_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pause", [0.0, 2.5])
def test_concurrent_uploads_bit_identical(pause):
    """Four threads upload ensembles at once, before and after the helpers have
    left for want of work: the scores of every handle are those of an upload
    alone, bit for bit."""
    from paper_1409_5000_gb300 import binding as B

    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    sets = [[synth.er(2_000 + 40_000 * (q % 3), 6.0 / (2_000 + 40_000 * (q % 3)), 10 * t + q) for q in range(5)]
            for t in range(4)]

    def scores(graphs):
        with B.GraphSet(graphs) as gs:
            return B.ensemble_scores(gs, 12, B.CB_FP32)[1].cpu().numpy()

    ref = [scores(g) for g in sets]
    time.sleep(pause)
    got = [None] * 4

    def work(t):
        with torch.cuda.stream(torch.cuda.Stream()):
            got[t] = scores(sets[t])

    th = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for x in th:
        x.start()
    for x in th:
        x.join()
    for r, g in zip(ref, got):
        assert g is not None and np.array_equal(r, g)
