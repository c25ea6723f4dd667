"""The path that the bench reports is the one the profile counted (no GPU needed)."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


class _G:
    def __init__(self, n, nnz):
        self.n, self.nnz = n, nnz


class _E:
    def __init__(self, *graphs):
        self.graphs = graphs


def test_one_launch_is_told_from_the_count():
    one, per_step = {"spmv": (1.0, 5)}, {"spmv": (1.0, 5 * 30)}
    ensemble, dense = _E(*[_G(30_000, 360_000)] * 8), _E(*[_G(3000, 300_000)] * 60)
    assert bench.path_run(ensemble, one, 5) == "small"
    assert bench.path_run(ensemble, per_step, 5, prec=1) == "csr"
    assert bench.path_run(dense, per_step, 5, csr_only=True) == "csr"
    assert bench.path_run(_E(_G(10_000_000, 160_000_000)), per_step, 5) == "twophase"
    # forward and backward: two recurrences a step
    assert bench.path_run(dense, {"spmv": (1.0, 10)}, 10) == "small"
