"""The limit of a kernel's waits begins when its inputs can be there: a launch
behind a kernel that runs far longer than the limit computes as usual."""
import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import build_on_gpu, check_product, to_dev, to_host

pytestmark = pytest.mark.gpu

LIMIT_NS = 1_000_000
SHAPES = {   # the kernel; R, C, M, K, dtype, sparsity, N: more chunks than a ring has stages
    "dense": ("dense", 16, 16, 1024, 1536, "bf16", 80, 600),
    "tc_bf16": ("tcgen05", 16, 16, 4096, 4096, "bf16", 97, 2048),
    "tc_f32": ("tcgen05", 32, 32, 512, 1536, "f32", 50, 300),
    "xcol": ("xcol", 32, 1, 1024, 1536, "f32", 50, 3000),
    "xstage": ("xstage", 8, 1, 512, 1536, "f32", 80, 300),
    "gk": ("gk", 64, 1, 512, 1536, "f32", 85, 1000),
}


@pytest.fixture(scope="module")
def slow():
    """A product of one CTA that takes many times the limit."""
    import paper_2106_08846_gb300 as bsr
    mp = pytest.MonkeyPatch()
    mp.setenv("BSR_FORCE_VARIANT", "generic")
    K = 1 << 19
    W = torch.full((32, K), 0.5, device="cuda")
    h = bsr.bsr_create(*bsr.bsr_from_dense(W, 32, 1), 32, 1, 32, K)
    mp.undo()
    X, Y = torch.ones((8, K), device="cuda"), torch.empty((8, 32), device="cuda")
    a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    for _ in range(2):
        a.record()
        bsr.bsr_spmm(h, X, None, Y)
        b.record()
        torch.cuda.synchronize()
    assert a.elapsed_time(b) * 1e6 > 4 * LIMIT_NS, a.elapsed_time(b)
    return lambda: bsr.bsr_spmm(h, X, None, Y)


@pytest.mark.parametrize("kind", list(SHAPES))
def test_a_limit_does_not_run_while_the_previous_kernel_does(slow, kind, monkeypatch):
    import paper_2106_08846_gb300 as bsr
    kernel, R, C, M, K, dt, sp, N = SHAPES[kind]
    w = synth.make_weight("wt", 8400 + R, M, K, R, C, dt, sp)
    gpu = build_on_gpu(w.W, R, C)
    monkeypatch.setenv("BSR_WAIT_LIMIT_NS", str(LIMIT_NS))
    h = bsr.bsr_create(*gpu, R, C, M, K)
    monkeypatch.delenv("BSR_WAIT_LIMIT_NS")
    X = synth.activations(8500, N, K, dt)
    Xd, b = to_dev(X), to_dev(w.bias)
    h.reserve(N)
    assert h.call_info(N)["kernel"] == kernel
    Y = h.spmm(Xd, b)
    torch.cuda.synchronize()
    for _ in range(3):
        slow()
        bsr.bsr_spmm(h, Xd, b, Y)
        torch.cuda.synchronize()
        assert h.check_device_status() == 0
    check_product(to_host(Y), oracle.bsr_from_dense(w.W, R, C), X, w.bias, M, rows=np.arange(0, N, 17))
