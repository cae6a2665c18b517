"""The tensor-core kernel on fp32 blocks (A operands in tensor memory) at each
task size, so at each number of ring stages and tensor-memory slots."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("g", [1, 2, 4, 8, 16])
def test_tc_f32_parity_at_task_size(g):
    r = subprocess.run([sys.executable, "-m", "tests.tc_f32_check"], cwd=ROOT,
                       env=dict(os.environ, BSR_TC_G=str(g), BSR_TC_F32_R16="1"), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
    assert r.stdout.count(": ok") == r.stdout.count("\n")
