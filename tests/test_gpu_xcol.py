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


ERRORS = """
import torch
import paper_2106_08846_gb300 as bsr
for R, C, M, K, N, sparsity in ((32, 1, 768, 768, 1024, 50), (32, 1, 4096, 4096, 512, 90), (16, 1, 2048, 2048, 1000, 70),
                                (32, 2, 768, 768, 1024, 50), (32, 2, 4096, 4096, 512, 90), (32, 1, 1024, 1024, 4096, 90)):
    total = 0.0
    for seed in range(4):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        keep = torch.rand(M // R, K // C, device="cuda", generator=gen) * 100 >= sparsity
        W = torch.randn(M // R, R, K // C, C, device="cuda", generator=gen) * 0.02
        W = (W * keep[:, None, :, None]).reshape(M, K)
        X = torch.randn(N, K, device="cuda", generator=gen)
        h = bsr.bsr_create(*bsr.bsr_from_dense(W, R, C), R, C, M, K)
        exact = X.double() @ W.double().T
        total += float((h.spmm(X).double() - exact).norm() / exact.norm())
    print(h.call_info(N)["kernel"], total / 4)
"""


def test_xcol_errors_are_no_larger_than_the_per_task_kernels():
    """Relative errors against 64-bit products, mean of four weights (1% for the draws)."""
    runs = []
    for env in ({}, {"BSR_XC": "0"}):
        r = subprocess.run([sys.executable, "-c", ERRORS], cwd=ROOT, env=dict(os.environ, **env), capture_output=True,
                           text=True, timeout=600)
        assert r.returncode == 0, r.stderr[-3000:]
        runs.append([line.split() for line in r.stdout.splitlines()])
    for (kernel, error), (other, bound) in zip(*runs):
        assert (kernel, other) == ("xcol", "xstage") and float(error) <= 1.01 * float(bound), (error, bound)
