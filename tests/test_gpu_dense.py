"""The dense-tile tensor-core kernel for bf16 weights: task sizes at the edges
of its range, ragged tokens, rows and columns, unequal and empty rows, X with
infinities and NaN, and a fused batch of different shapes."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
import synth
from tests.gpu_util import as_f64, build_on_gpu, check_product, to_dev, to_host

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("g", [None, "own", 1, 3, 7, 16, 34, 38, 48])   # 32 + g: pairs of CTAs
def test_dense_parity_at_task_size(g):
    env = dict(os.environ, **({} if g is None else {"BSR_DENSE": "1"} if g == "own" else {"BSR_DENSE_G": str(g)}))
    r = subprocess.run([sys.executable, "-m", "tests.dense_check"], cwd=ROOT, env=env, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]


@pytest.mark.parametrize("g", [4, 48])
def test_dense_bounded_wait_times_out_and_reports(g):
    """A chunk that is never loaded: both CTAs of a pair give up, complete each
    other's loads and return; a later call computes correctly."""
    code = """
import os, numpy as np, oracle, synth, torch
import paper_2106_08846_gb300 as bsr
from paper_2106_08846_gb300 import bsrlib as b
from tests.gpu_util import as_f64, build_on_gpu, check_product, to_dev, to_host
w = synth.make_weight("ds", 7700, 512, 1536, 16, 16, "bf16", 80)
gpu = build_on_gpu(w.W, 16, 16)
os.environ.update(BSR_WAIT_LIMIT_NS="2000000", BSR_TEST_STALL_CHUNK="9")
h = bsr.bsr_create(*gpu, 16, 16, 512, 1536)
del os.environ["BSR_WAIT_LIMIT_NS"], os.environ["BSR_TEST_STALL_CHUNK"]
X = synth.activations(7701, 3000, 1536, "bf16")
h.spmm(to_dev(X), to_dev(w.bias))
assert h.check_device_status() == b.BSR_ERR_TIMEOUT
h2 = bsr.bsr_create(*gpu, 16, 16, 512, 1536)
Y = to_host(h2.spmm(to_dev(X), to_dev(w.bias)))
assert h2.check_device_status() == b.BSR_OK
check_product(Y, oracle.bsr_from_dense(w.W, 16, 16), X, w.bias, 512, rows=np.arange(0, 3000, 37))
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, BSR_DENSE_G=str(g)),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-3000:]


def test_dense_batch_of_different_shapes_is_bitwise_the_single_calls():
    import paper_2106_08846_gb300 as bsr
    N, K = 333, 384
    ws = [synth.make_weight("db", 7500 + i, M, K, R, C, "bf16", 0,
                            mask=synth.uniform_block_mask(7500 + i, M // R, K // C, (M // R) * (K // C) // 3))
          for i, (R, C, M) in enumerate([(16, 16, 512), (32, 1, 256), (1, 32, 80), (64, 64, 1024)])]
    hs = [bsr.bsr_create(*build_on_gpu(w.W, w.R, w.C), w.R, w.C, w.M, w.K) for w in ws]
    X = synth.activations(7600, N, K, "bf16")
    Xd, bs = to_dev(X), [to_dev(w.bias) for w in ws]
    Ys = [torch.empty((N, w.M), dtype=torch.bfloat16, device="cuda") for w in ws]
    bsr.bsr_spmm_batch(hs, Xd, bs, Ys, N)
    for h, w, b, Y in zip(hs, ws, bs, Ys):
        single = to_host(h.spmm(Xd, b))
        assert np.array_equal(to_host(Y), single)
        check_product(single, oracle.bsr_from_dense(w.W, w.R, w.C), X, w.bias, w.M)
        assert h.check_device_status() == 0


@pytest.mark.parametrize("R,C,N", [(32, 1, 3000), (1, 1, 700), (4, 4, 129)])
def test_dense_takes_sparse_narrow_weights_of_the_simt_variant(R, C, N):
    """bf16 blocks too sparse for the block-by-block kernel (1/12 fill): the
    schedule's variant stays the SIMT kernel, calls may run on dense tiles;
    either way the product is the oracle's, and a batch is the single calls."""
    import paper_2106_08846_gb300 as bsr
    M, K = 768, 1024
    ws = [synth.make_weight("dx", 7800 + i, M, K, R, C, "bf16", 0,
                            mask=synth.uniform_block_mask(7800 + i, M // R, K // C, (M // R) * (K // C) * (3 + i) // 100))
          for i in range(2)]
    hs = [bsr.bsr_create(*build_on_gpu(w.W, R, C), R, C, M, K) for w in ws]
    assert all(h.schedule()["variant"] == "xstage" and "dense" in h.schedule()["kernels"] for h in hs)
    X = synth.activations(7801, N, K, "bf16")
    Xd, b = to_dev(X), to_dev(ws[0].bias)
    Ys = [torch.empty((N, M), dtype=torch.bfloat16, device="cuda") for _ in ws]
    bsr.bsr_spmm_batch(hs, Xd, [b, None], Ys, N)
    rows = np.unique(np.concatenate([np.arange(0, N, 13), np.arange(N - 130 if N > 130 else 0, N)]))
    for i, (h, w, Y) in enumerate(zip(hs, ws, Ys)):
        single = to_host(h.spmm(Xd, b if i == 0 else None))
        assert np.array_equal(to_host(Y), single)
        check_product(single, oracle.bsr_from_dense(w.W, R, C), X, ws[0].bias if i == 0 else None, M, rows=rows)


@pytest.mark.parametrize("g", [2, 34, 48])
def test_dense_back_to_back_launches_of_few_chunks(g):
    """One chunk or two per unit, so that a CTA's last arrivals (ring stages,
    accumulators, the second CTA's of a pair) come just before it ends and the
    next launch takes its shared memory: 400 launches, bit for bit the first."""
    code = """
import torch, oracle, synth
import paper_2106_08846_gb300 as bsr
from tests.gpu_util import as_f64, build_on_gpu, check_product, to_dev, to_host
for K, N in ((64, 300), (128, 5000)):
    w = synth.make_weight("de", 7900 + K, 512, K, 16, 16, "bf16", 50)
    h = bsr.bsr_create(*build_on_gpu(w.W, 16, 16), 16, 16, 512, K)
    X = synth.activations(7902, N, K, "bf16")
    Xd, b = to_dev(X), to_dev(w.bias)
    Ys = torch.empty((200, N, 512), dtype=torch.bfloat16, device="cuda")
    for Y in Ys:
        bsr.bsr_spmm(h, Xd, b, Y)
    assert h.check_device_status() == 0
    check_product(to_host(Ys[0]), oracle.bsr_from_dense(w.W, 16, 16), X, w.bias, 512)
    assert all(torch.equal(Y, Ys[0]) for Y in Ys)
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, BSR_DENSE_G=str(g)),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-3000:]


@pytest.mark.parametrize("g", [5, 16, 48])
def test_dense_each_unit_adds_its_own_bias(g):
    """Tasks of more than four row groups, with chunks and without, the biases
    of one unit unlike the next one's: a warp's lanes read one another's."""
    code = """
import numpy as np, torch, oracle, synth
import paper_2106_08846_gb300 as bsr
from tests.gpu_util import build_on_gpu, to_dev, to_host
M, K, N = 16 * 203, 128, 2000
cnt = np.zeros(M // 16, dtype=np.int64)
cnt[::3] = 2
w = synth.make_weight("dg", 8100, M, K, 16, 16, "bf16", 0, mask=synth.mask_from_row_counts(8100, cnt, K // 16))
h = bsr.bsr_create(*build_on_gpu(w.W, 16, 16), 16, 16, M, K)
bias = torch.arange(1, M + 1, device="cuda").bfloat16().float()
Y = h.spmm(torch.zeros((N, K), dtype=torch.bfloat16, device="cuda"), bias)
assert h.check_device_status() == 0
assert torch.equal(Y.float(), bias.expand(N, M))
"""
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, BSR_DENSE_G=str(g)),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-3000:]


def test_kernels_that_allocate_tensor_memory_follow_one_another():
    """Launches of the kernels that allocate tensor memory, one behind another
    without a synchronisation, small enough to share an SM: each allocates
    before the next may start, and every output is that of the call alone."""
    import paper_2106_08846_gb300 as bsr
    runs = []
    for i, (kernel, R, C, M, K, dt, sp, N) in enumerate([
            ("tcgen05", 16, 16, 4096, 4096, "bf16", 97, 2048),   # two CTAs an SM
            ("dense", 16, 16, 512, 64, "bf16", 50, 200),
            ("tcgen05", 32, 32, 256, 64, "f32", 0, 200),
            ("gk", 64, 1, 512, 768, "f32", 85, 1000),
            ("xcol", 32, 1, 1024, 768, "f32", 50, 2000),
            ("dense", 64, 64, 512, 192, "bf16", 0, 700)]):
        w = synth.make_weight("tm", 8200 + i, M, K, R, C, dt, sp)
        h = bsr.bsr_create(*build_on_gpu(w.W, R, C), R, C, M, K)
        X = to_dev(synth.activations(8300 + i, N, K, dt))
        h.reserve(N)
        assert h.call_info(N)["kernel"] == kernel
        Y = h.spmm(X, to_dev(w.bias))
        torch.cuda.synchronize()
        runs.append((h, X, to_dev(w.bias), Y, torch.empty((8, *Y.shape), dtype=Y.dtype, device="cuda")))
    pairs = [(a, b) for a in range(len(runs)) for b in range(len(runs))]
    for rep in range(60):
        for h, X, b, _, Ys in (runs[k] for k in pairs[rep % len(pairs)]):
            for k in range(4):
                bsr.bsr_spmm(h, X, b, Ys[k + 4 * (rep & 1)])
    for rep in range(8):
        for h, X, b, _, Ys in runs:
            bsr.bsr_spmm(h, X, b, Ys[rep])
    for h, X, b, Y, Ys in runs:
        assert h.check_device_status() == 0
        assert all(torch.equal(Y, Yk) for Yk in Ys)


@pytest.mark.parametrize("R,C,share", [(32, 1, 1.0), (32, 1, 0.04), (1, 1, 1.0), (4, 4, 1.0), (16, 16, 1.0), (64, 16, 0.04)])
def test_dense_non_finite_tokens_at_large_k(R, C, share, monkeypatch):
    """A NaN or an infinity in every token (or a few of each 32): its outputs
    that do not keep the column are computed again, which takes far longer than
    a wait's limit (1 ms) and leaves no call unfinished; N is several units a
    CTA. Other tokens keep the finite call's bits."""
    import paper_2106_08846_gb300 as bsr
    M, K, N = 1024, 8192, 20000
    MB, KB = M // R, K // C
    w = synth.make_weight("dnf", 8600 + R, M, K, R, C, "bf16", 0, mask=synth.uniform_block_mask(8600 + R, MB, KB, MB * KB // 5))
    gpu = build_on_gpu(w.W, R, C)
    monkeypatch.setenv("BSR_WAIT_LIMIT_NS", "1000000")
    h = bsr.bsr_create(*gpu, R, C, M, K)
    monkeypatch.delenv("BSR_WAIT_LIMIT_NS")
    gen = torch.Generator(device="cuda").manual_seed(8601)
    X = torch.randn(N, K, device="cuda", generator=gen).bfloat16()
    b = to_dev(w.bias)
    finite = h.spmm(X, b)
    tokens = torch.rand(N, device="cuda", generator=gen) < share
    at = torch.randint(K, (N,), device="cuda", generator=gen)
    special = torch.tensor([float("nan"), float("inf"), float("-inf")], device="cuda").bfloat16()[torch.arange(N, device="cuda") % 3]
    X[tokens, at[tokens]] = special[tokens]
    Y = h.spmm(X, b)
    assert h.check_device_status() == 0
    assert torch.equal(Y[~tokens], finite[~tokens])
    rows = tokens.nonzero()[:, 0][::max(1, int(tokens.sum()) // 40)]
    Xs, ref = to_host(X[rows]), oracle.bsr_from_dense(w.W, R, C)
    with np.errstate(invalid="ignore"):
        want = oracle.bsr_spmm(*ref, Xs, w.bias, M)
    got, fin = as_f64(to_host(Y[rows])), np.isfinite(want)
    assert fin.mean() > 0.5 and np.array_equal(np.isfinite(got), fin)
    assert np.array_equal(got[~fin], want[~fin], equal_nan=True)
    E = oracle.err_bound(*ref, np.where(np.isfinite(as_f64(Xs)), Xs, 0).astype(np.uint16), w.bias, M)
    assert np.all(np.abs(got[fin] - want[fin]) <= 1e-2 * E[fin])


@pytest.mark.parametrize("M,K", [(0, 64), (64, 0), (0, 0)])
@pytest.mark.parametrize("R,C", [(16, 16), (32, 1)])
def test_dense_weights_without_elements(R, C, M, K):
    """M = 0: nothing to write; K = 0: the bias; through every call form."""
    import paper_2106_08846_gb300 as bsr
    N = 200
    lib = bsr.load()
    stream = torch.cuda.current_stream().cuda_stream
    hs = [bsr.bsr_create(torch.zeros(M // R + 1, dtype=torch.int32, device="cuda"), torch.zeros(0, dtype=torch.int32, device="cuda"),
                         torch.zeros((0, R, C), dtype=torch.bfloat16, device="cuda"), R, C, M, K) for _ in range(2)]
    X = torch.zeros(N * max(K, 8), dtype=torch.bfloat16, device="cuda")
    bias = torch.arange(1, M + 2, device="cuda").float()
    Ys = [torch.full((N * max(M, 8),), 7.0, dtype=torch.bfloat16, device="cuda") for _ in hs]
    want = bias[:M].bfloat16().expand(N, M).flatten() if M else Ys[0].clone()
    for call in (lib.bsr_spmm, lib.bsr_spmm_noalloc):
        Ys[0].fill_(7.0)
        assert call(hs[0].ptr, X.data_ptr(), bias.data_ptr(), Ys[0].data_ptr(), N, stream) == 0
        assert torch.equal(Ys[0], want)
    ptrs = (ctypes.c_void_p * 2)
    assert lib.bsr_spmm_batch(ptrs(*(h.ptr for h in hs)), 2, X.data_ptr(), ptrs(bias.data_ptr(), bias.data_ptr()),
                              ptrs(*(Y.data_ptr() for Y in Ys)), N, stream) == 0
    assert all(torch.equal(Y, want) for Y in Ys)
    assert all(h.check_device_status() == 0 for h in hs)


@pytest.mark.parametrize("R,C", [(32, 1), (4, 4), (16, 16)])
@pytest.mark.parametrize("every", [1, 16])
def test_dense_infinities_in_the_weight_too(R, C, every):
    """Infinities, NaN and zeros of both signs in kept elements, against X with
    infinities, NaN and zeros in the same columns and in others: NaN and
    infinite outputs where the oracle has them (tokens: all, or two of 32)."""
    import paper_2106_08846_gb300 as bsr
    M, K, N = 256, 320, 200
    w = synth.make_weight("dw", 9600 + R, M, K, R, C, "bf16", 60)
    W, rng = w.W.copy(), np.random.RandomState(5)
    rows, cols = np.nonzero(W)
    pick = rng.permutation(rows.size)[:24]
    for k, at in enumerate(pick):
        W[rows[at], cols[at]] = (0x7f80, 0xff80, 0x7fc0, 0x8000, 0x0000)[k % 5]
    gpu, ref = build_on_gpu(W, R, C), oracle.bsr_from_dense(W, R, C)
    h = bsr.bsr_create(*gpu, R, C, M, K)
    assert h.call_info(N)["kernel"] == "dense"
    X = synth.activations(9601, N, K, "bf16")
    for t in range(0, N, every):
        for k, c in enumerate([cols[pick[t % 24]], rng.randint(K)]):
            X[t, c] = (0x7f80, 0xff80, 0x7fc1, 0x0000, 0x8000)[(t // every + k) % 5]
    got = as_f64(to_host(h.spmm(to_dev(X), to_dev(w.bias))))
    assert h.check_device_status() == 0
    with np.errstate(invalid="ignore"):
        want = oracle.bsr_spmm(*ref, X, w.bias, M)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    inf = np.isinf(want)
    assert inf.any() and np.array_equal(np.isinf(got), inf) and np.array_equal(got[inf], want[inf])
    fin = np.isfinite(want)
    assert np.allclose(got[fin], want[fin], rtol=2e-2, atol=2e-2)
