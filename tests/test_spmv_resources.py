"""The SpMV kernels keep their working set in registers at every group width
(compiles one file with nvcc, no GPU needed)."""
import os
import re

from paper_1409_5000_gb300 import _build


def test_spmv_kernels_do_not_spill(tmp_path):
    """Both precisions, group widths 1 to 32: at most 32 bytes a thread (a few
    values used once per tile), where a spilled inner loop takes hundreds."""
    cmd = [_build._nvcc(), "-c", os.path.join(_build.CSRC, "cb_lanczos.cu"), "-o", str(tmp_path / "x.o")]
    log = _build._run(cmd + _build.nvcc_flags(["-Xptxas", "-v"]))
    names = re.findall(r"Function properties for (\S+)\n\s+\d+ bytes stack frame, (\d+) bytes spill stores", log)
    spills = {n: int(b) for n, b in names if re.search(r"\d+spmv_kernelI[fd]Li\d+E", n) and "bspmv" not in n}
    assert len(spills) == 13, log[-2000:]  # FP64 at width 4 in two shapes
    assert max(spills.values()) <= 32, spills
