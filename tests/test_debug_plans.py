"""The kernels that run when the plan is left to the library, under the debug build's device-side
index checks (tests/debug_plans.py, in a child process because a process loads one build)."""
import os
import subprocess
import sys

import pytest

from paper_1612_02495_gb300 import build as libbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.gpu
def test_library_plans_clean():
    libbuild.build(debug=True)
    env = dict(os.environ, SWEPT_DEBUG="1", PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, os.path.join("tests", "debug_plans.py")], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "all clean" in r.stdout
