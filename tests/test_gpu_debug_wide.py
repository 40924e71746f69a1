"""The bounds-checked debug build over the kernels of the wide radices, the fused
loss, the three peak passes, the chirp-z rows and the grouped mixed-size kernels (see
_debug_wide_child.py, run in a process of its own): every result matches and no
device index check fires."""
import os
import subprocess
import sys

import pytest

from tests import _gpu

pytestmark = pytest.mark.gpu


def test_debug_build_index_checks_of_the_wide_lengths_stay_clean():
    _gpu.torch_cuda()                                   # the normal library (built if missing)
    from paper_1904_09409_gb300 import funnel as f
    if not os.path.exists(os.path.join(f.PKG, "libfunnel_debug.so")):
        from paper_1904_09409_gb300 import build
        build.build()
    child = os.path.join(os.path.dirname(os.path.abspath(__file__)), "_debug_wide_child.py")
    r = subprocess.run([sys.executable, child], capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.strip().endswith("OK"), r.stdout + r.stderr
