"""The column-list SIMT kernel for fp32 blocks of 16 and 32 rows at each of its token tiles and
several task sizes (forced: by itself it takes only calls it is faster on), and
with both chosen per launch (one product and three then differ in them)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("tile", [0, 1, 2])
def test_xcol_parity_at_tile(tile):
    r = subprocess.run([sys.executable, "-m", "tests.xcol_check"], cwd=ROOT, env=dict(os.environ, BSR_XC_TILE=str(tile)),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]


@pytest.mark.parametrize("env", [{}, {"BSR_XC_G": "1"}, {"BSR_XC_G": "3"}, {"BSR_XC_G": "8"}])
def test_xcol_parity_at_task_size(env):
    r = subprocess.run([sys.executable, "-m", "tests.xcol_check"], cwd=ROOT, env=dict(os.environ, BSR_XC="1", **env),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
