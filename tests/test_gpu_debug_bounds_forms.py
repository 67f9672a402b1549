"""The bounds-checked library on the kernel forms of small problems and of many states (tests/_forms.py) and on
the fallback pass's longer ranges: every checked index stays in its range."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_index_leaves_its_range_in_any_form():
    from paper_2507_06300_gb300 import build
    build.build(debug=True)
    r = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "_debug_bounds_forms_run.py")],
                       env=dict(os.environ, LISA_DEBUG_BOUNDS="1"), capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-3000:]
    rep = json.loads(r.stdout.strip().splitlines()[-1])
    assert rep["enabled"] is True and rep["finite"] is True and rep["bounds"]["count"] == 0, rep
