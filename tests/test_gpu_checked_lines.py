"""The bounds-checked build (tests/test_gpu_checked.py) on the suites of the line kernels at every order,
the triangle groups, the allocation-free entry at its size limit, and non-finite kinematic states: run
again in a child process on the checked library, each test also required to leave the process's count of
bounds failures unchanged (tests/conftest.py)."""
import os
import re
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SUITES = ["tests/test_gpu_lines.py", "tests/test_gpu_line_calls.py", "tests/test_gpu_tri_groups.py",
          "tests/test_noalloc_limit.py", "tests/test_gpu_kin_nonfinite.py"]


def test_gpu_suites_on_the_checked_build(dg):
    env = dict(os.environ, DGPF_CHECKED="1")
    cmd = [sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider"] + SUITES
    r = subprocess.run(cmd, cwd=ROOT, env=env, capture_output=True, text=True, timeout=1500)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-2000:]
    m = re.search(r"(\d+) passed", r.stdout)
    assert m and int(m.group(1)) >= 100 and " failed" not in r.stdout and " skipped" not in r.stdout, r.stdout[-2000:]
