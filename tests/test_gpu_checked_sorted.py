"""The bounds-checked build (-DPP_CHECKED) on the particle kernels that sort in
every step, the tile kernel and the row kernel: every index into the windows,
the pairs and quads of the gather and the mesh is tested against its array.  On
the cases of tests/checked_sorted_cases.py (every shape, partly empty last
tiles, blocks of one, two and four planes, walls, an open end with an injector
and a window, several chunks) it must report no violation and give the normal
build's fields."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_checked_build_finds_no_out_of_bounds_index():
    from paper_1211_4575_gb300 import build
    build.build()
    build.build(checked=True)
    from tests import checked_sorted_cases
    plain = checked_sorted_cases.run_cases()
    env = dict(os.environ, PP_GB300_CHECKED="1")
    r = subprocess.run([sys.executable, "-m", "tests.checked_sorted_cases", ROOT], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    checked = json.loads(r.stdout.strip().splitlines()[-1])
    assert set(checked) == set(plain) == set(checked_sorted_cases.CASES)
    for name, (status, launches, fields) in checked.items():
        assert status == 0, (name, status)          # PP_EBOUNDS would be 10
        assert launches == 1 == plain[name][1], name   # one launch for both species: a sorted kernel
        a, b = np.asarray(fields), np.asarray(plain[name][2])
        assert np.abs(a - b).max() <= 1e-4 * max(np.abs(b).max(), 1e-30), name
