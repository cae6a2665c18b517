"""bsr_get_call_info names the kernel that runs a call and counts its launches."""
import ctypes

import numpy as np
import pytest
import torch

import synth
from tests.gpu_util import build_on_gpu

pytestmark = pytest.mark.gpu

CALLS = [  # R, C, M, K, dtype, sparsity, N, the kernel
    (32, 1, 1024, 1024, "f32", 90, 16384, "xcol"), (32, 1, 1024, 1024, "f32", 90, 128, "xstage"),
    (16, 1, 1024, 1024, "f32", 90, 16384, "xcol"), (16, 16, 1024, 1024, "f32", 90, 4096, "tcgen05"),
    (16, 16, 1024, 1024, "bf16", 90, 16384, "dense"), (32, 1, 768, 768, "bf16", 80, 1024, "dense"),
    (32, 1, 1024, 1024, "bf16", 95, 16384, "dense"), (16, 16, 4096, 4096, "bf16", 97, 2048, "tcgen05"),
    (64, 1, 512, 768, "f32", 85, 1000, "gk"), (64, 1, 512, 768, "f32", 85, 300, "generic"),
    (1, 1, 768, 768, "f32", 80, 1024, "xstage"),
]


@pytest.mark.parametrize("R,C,M,K,dtype,sparsity,N,kernel", CALLS)
def test_call_info_names_the_kernel(R, C, M, K, dtype, sparsity, N, kernel):
    import paper_2106_08846_gb300 as bsr
    w = synth.make_weight("ci", 8800 + R, M, K, R, C, dtype, sparsity)
    h = bsr.bsr_create(*build_on_gpu(w.W, R, C), R, C, M, K)
    info = h.call_info(N)
    assert info["kernel"] == kernel
    assert kernel in h.schedule()["kernels"].split(",") and h.schedule()["kernels"].startswith(h.schedule()["variant"])
    X = torch.zeros((N, K), dtype=torch.float32 if dtype == "f32" else torch.bfloat16, device="cuda")
    Y = torch.empty((N, M), dtype=X.dtype, device="cuda")
    plan = bsr.bsr_plan_create([h], [X], [None], [Y])
    assert plan.order()[2] == info["launches"]
    assert h.call_info(0) == {"kernel": "none", "launches": 0}
    buf = ctypes.create_string_buffer(8)
    lib = bsr.load()
    assert lib.bsr_get_call_info(h.ptr, -1, buf, 8) == lib.bsr_get_call_info(None, 1, buf, 8) == 1
    assert lib.bsr_get_call_info(h.ptr, N, buf, 8) == 0 and buf.value == b"kernel="


def test_call_info_counts_the_reduce_pass():
    import paper_2106_08846_gb300 as bsr
    cnt = np.full(40, 3, dtype=np.int64)
    cnt[7] = 512   # split into pieces that a second launch adds up
    w = synth.make_weight("cj", 8801, 40 * 8, 512, 8, 1, "f32", 0, mask=synth.mask_from_row_counts(8801, cnt, 512))
    h = bsr.bsr_create(*build_on_gpu(w.W, 8, 1), 8, 1, 320, 512)
    assert h.schedule()["split_rows"] == 1 and h.call_info(100) == {"kernel": "xstage", "launches": 2}
