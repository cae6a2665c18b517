"""A handle holds device memory for a kernel only if some call would run it."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import sys, torch
import paper_2106_08846_gb300 as bsr
R, C, M, K, dt, keep, uneven = eval(sys.argv[1])
gen = torch.Generator(device="cuda").manual_seed(8700)
MB, KB = M // R, K // C
share = torch.full((MB, 1), keep, device="cuda")
if uneven:
    share[::2], share[1::2] = 0.2 * keep, 1.8 * keep
mask = torch.rand(MB, KB, device="cuda", generator=gen) < share
if uneven == 2:
    mask[0] = True
W = (torch.ones(MB, R, KB, C, device="cuda") * mask[:, None, :, None]).reshape(M, K).to(dt)
arrays = bsr.bsr_from_dense(W, R, C)
small = bsr.bsr_create(*bsr.bsr_from_dense(W[:64, :64].contiguous(), R, C), R, C, 64, 64)
torch.cuda.synchronize()
before = torch.cuda.mem_get_info()[0]
h = bsr.bsr_create(*arrays, R, C, M, K)
torch.cuda.synchronize()
print(before - torch.cuda.mem_get_info()[0], h.schedule()["kernels"])
"""


def held(weight, **env):
    """Device bytes that creating the weight's handle takes, and the kernels it holds operands for."""
    r = subprocess.run([sys.executable, "-c", CODE, weight], cwd=ROOT, env=dict(os.environ, **env), capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    n, kernels = r.stdout.split()
    return int(n), kernels.split(",")


@pytest.mark.parametrize("weight,kernel,off", [
    # column lists: not for unequal rows, a row that fills the ring's stages, few columns a chunk
    ("(32, 1, 4096, 4096, torch.float32, 0.1, 1)", "xcol", "BSR_XC"),
    ("(32, 1, 4096, 4096, torch.float32, 0.1, 2)", "xcol", "BSR_XC"),
    ("(16, 2, 4096, 4096, torch.float32, 0.002, 0)", "xcol", "BSR_XC"),
    # dense tiles: not for wide weights too sparse for them at any token count
    ("(32, 1, 8192, 8192, torch.bfloat16, 0.01, 0)", "dense", "BSR_DENSE"),
    ("(1, 1, 8192, 8192, torch.bfloat16, 0.005, 0)", "dense", "BSR_DENSE"),
    # gathered columns: only for the shapes that are otherwise the generic kernel's
    ("(16, 16, 4096, 4096, torch.bfloat16, 0.1, 0)", "gk", "BSR_GK"),
    ("(32, 1, 4096, 4096, torch.float32, 0.1, 0)", "gk", "BSR_GK"),
])
def test_no_memory_for_a_kernel_that_no_call_runs(weight, kernel, off):
    n, kernels = held(weight)
    assert kernel not in kernels
    assert n == held(weight, **{off: "0"})[0]


def test_operands_of_a_kernel_that_calls_run():
    assert "xcol" in held("(32, 1, 1024, 1024, torch.float32, 0.1, 0)")[1]
    assert "gk" in held("(64, 1, 512, 768, torch.float32, 0.1, 0)")[1]
    assert "dense" in held("(16, 16, 1024, 1024, torch.bfloat16, 0.1, 0)")[1]
