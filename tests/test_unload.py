"""libcb keeps helper threads for a while after an upload, so it must stay
mapped when a host program closes it (no GPU needed)."""
import os
import subprocess
import sys

import pytest

from paper_1409_5000_gb300 import _build

SCRIPT = """
import _ctypes, ctypes, sys
path = sys.argv[1]
h = ctypes.CDLL(path)._handle
_ctypes.dlclose(h)
sys.exit(0 if any(path in line for line in open("/proc/self/maps")) else 3)
"""


@pytest.mark.parametrize("debug", [False, True])
def test_closed_library_stays_mapped(debug):
    path = _build.cb_lib_path(debug)
    if not os.path.exists(path):
        _build.build_cb(debug=debug)
    assert subprocess.run([sys.executable, "-c", SCRIPT, os.path.realpath(path)]).returncode == 0
