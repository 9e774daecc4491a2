"""The suites that put points and frames at the borders, against the
bounds-checked build in a child process (every test there also asserts that no
access left its buffer), and that build's positive control of the map-point
kernels."""
import os
import re
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
ENV = dict(os.environ, GLT_LIBRARY="checked")


def test_map_point_kernels_flag_what_they_access():
    code = ("import ctypes, paper_2607_16897_gb300 as glt\n"
            "f = ctypes.c_uint(0)\n"
            "rc = glt.glt_debug_checked_probe(ctypes.byref(f))\n"
            "assert rc == 0, glt.glt_last_error()\n"
            "assert glt.glt_debug_checked_flags(ctypes.byref(f)) == 0 and f.value == 0\n"
            "print('probe ok')\n")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=ENV, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "probe ok" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]


def test_border_suites_in_the_checked_build():
    suites = ["test_gpu_patch_tables.py", "test_gpu_pyramid_edges.py", "test_gpu_block_sums.py", "test_gpu_track_image.py"]
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider",
                        *[os.path.join(ROOT, "tests", s) for s in suites]],
                       cwd=ROOT, env=ENV, capture_output=True, text=True, timeout=1800)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
    m = re.search(r"(\d+) passed", r.stdout)
    assert m and int(m.group(1)) >= 100, r.stdout[-2000:]
