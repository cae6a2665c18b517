"""bsr_from_dense at the edges of its segments: blocks of the largest size in
either direction, rows that are not 16-byte aligned, a misaligned W, one and
many segments per block row, a partly filled last one; bit for bit against the
oracle, NaN and threshold rule included."""
import concurrent.futures
import ctypes

import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import assert_structure_equal, dtype_of, to_dev

pytestmark = pytest.mark.gpu

SHAPES = [  # R, C, M, K
    (4096, 1, 8192, 6), (1, 4096, 3, 3 * 4096), (64, 64, 128, 64 * 5), (1, 1, 7, 2049), (1, 1, 3, 5000),
    (2, 3, 10, 3 * 701), (8, 1, 16, 1026), (32, 1, 64, 4100), (5, 7, 15, 7 * 333), (16, 16, 32, 16 * 70),
]


@pytest.mark.parametrize("R,C,M,K", SHAPES)
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("offset", [0, 1])
def test_builder_segments_match_the_oracle(R, C, M, K, dtype, offset):
    import paper_2106_08846_gb300 as bsr
    MB, KB = M // R, K // C
    w = synth.make_weight("be", 8000 + R + C, M, K, R, C, dtype, 0,
                          mask=synth.uniform_block_mask(8000 + R + C, MB, KB, max(1, (MB * KB) // 3)))
    W = w.W.copy()
    W.flat[0] = np.float32("nan") if dtype == "f32" else 0x7fc0
    Wd = to_dev(W).flatten()
    buf = torch.empty(M * K + 8, dtype=Wd.dtype, device="cuda")
    at = buf[offset:offset + M * K].view(M, K)   # offset 1: no 16-byte loads
    at.copy_(Wd.view(M, K))
    for thr in (0.0, 0.03):
        assert_structure_equal(bsr.bsr_from_dense(at, R, C, thr), oracle.bsr_from_dense(W, R, C, thr))
    assert dtype_of(W) == dtype


def test_a_conversion_keeps_no_device_memory():
    """What a call allocates comes from the device's default pool, and all of
    it is back there afterwards."""
    import paper_2106_08846_gb300 as bsr
    W = torch.randn(1024, 4096, device="cuda") * (torch.rand(1024, 4096, device="cuda") < 0.01)
    torch.cuda.synchronize()
    cuda = ctypes.CDLL("libcuda.so.1")
    pool, n = ctypes.c_void_p(), ctypes.c_uint64(0)
    assert cuda.cuDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    used, used_high = 7, 8   # CU_MEMPOOL_ATTR_USED_MEM_CURRENT, _HIGH
    assert cuda.cuMemPoolSetAttribute(pool, used_high, ctypes.byref(n)) == 0
    for R, C in ((1, 1), (32, 1), (16, 16)):
        indptr, indices, data = bsr.bsr_from_dense(W, R, C)
        assert indices.numel() == int(indptr[-1]) > 0
    torch.cuda.synchronize()
    assert cuda.cuMemPoolGetAttribute(pool, used_high, ctypes.byref(n)) == 0 and n.value > 0
    assert cuda.cuMemPoolGetAttribute(pool, used, ctypes.byref(n)) == 0 and n.value == 0


def test_conversions_of_several_threads_and_under_capture():
    """Each call reads its own count: eight threads on streams of their own; and
    a call in a stream capture, whose wait fails, leaves later ones right."""
    import paper_2106_08846_gb300 as bsr
    lib = bsr.load()
    Ws, refs = [], []
    for k in range(8):
        w = synth.make_weight("bt", 8900 + k, 256, 512, 8, 4, "f32", 10 * k)
        Ws.append(to_dev(w.W))
        refs.append(oracle.bsr_from_dense(w.W, 8, 4))
    torch.cuda.synchronize()

    def convert(k):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(50):
                out = bsr.bsr_from_dense(Ws[k], 8, 4, stream=s)
        s.synchronize()
        return out

    def check():
        with concurrent.futures.ThreadPoolExecutor(8) as ex:
            for out, ref in zip(ex.map(convert, range(8)), refs):
                assert_structure_equal(out, ref)

    check()
    indptr, s, graph = torch.empty(33, dtype=torch.int32, device="cuda"), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        graph.capture_begin()
        status = lib.bsr_from_dense(Ws[0].data_ptr(), 256, 512, 8, 4, 0.0, 0, indptr.data_ptr(), None, None, 0, None,
                                    s.cuda_stream)
        with pytest.raises(RuntimeError):
            graph.capture_end()
    assert status != 0
    assert_structure_equal(bsr.bsr_from_dense(Ws[0], 8, 4), refs[0])   # (this thread finds no error of that call)
    check()
