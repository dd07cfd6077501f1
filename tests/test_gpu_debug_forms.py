"""The bounds-checked build over the kernels that the library dispatches by size:
the two-step tiles of 16, 24 and 32 rows, dependent launches or not, and the phases
on chip, in modelling, migration, checkpointed migration and Born modelling.  Any
index outside its array fails the child's tests."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_debug_build_runs_the_dispatched_forms_cleanly():
    from paper_2001_06444_gb300 import build

    build.build(debug=True)
    r = subprocess.run(
        [sys.executable, "-m", "pytest", "-x", "-q", "-m", "gpu", "tests/test_gpu_step2_forms.py",
         "tests/test_gpu_resident.py"],
        cwd=ROOT, env=dict(os.environ, RTM_DEBUG="1"), capture_output=True, text=True, timeout=1800)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-2000:]
    assert " passed" in r.stdout and "skipped" not in r.stdout
