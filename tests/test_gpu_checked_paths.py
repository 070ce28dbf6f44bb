"""The plan, join, sort and granularity edge cases on the checked build (libssj_checked.so): list ends,
early flushes, bad offsets, windows beyond the bitmap, forced granularities and stretches of empty lists,
with no index check firing (a fired check turns a call into SSJ_EDEVICE, which fails them)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("suite", ["plan", "join", "sort", "forced", "sparse"])
def test_suite_on_the_checked_build(suite):
    r = subprocess.run([sys.executable, "-m", "pytest", "-q", "-x", "-p", "no:cacheprovider",
                        f"tests/test_gpu_{suite}.py", "-k", "not walked"], cwd=ROOT,
                       env=dict(os.environ, SSJ_LIBRARY="checked"), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-2000:]
