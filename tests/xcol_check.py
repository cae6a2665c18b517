"""Parity sweep of the column-list SIMT kernel, for a process started with
BSR_XC_TILE (one token tile) or BSR_XC=1 and perhaps BSR_XC_G (items per
task). Run by tests/test_gpu_xcol.py in a subprocess;
exit status 0 when every output is right."""
import os
import sys

import numpy as np

SHAPES = [(32, 1, 32, 64, 1), (32, 1, 352, 100, 63), (32, 1, 384, 1000, 64), (32, 1, 1024, 768, 113),
          (32, 1, 160, 260, 1000), (32, 1, 736, 512, 4000), (32, 4, 352, 264, 400),
          (16, 1, 16, 64, 1), (16, 1, 176, 100, 127), (16, 1, 384, 1000, 129), (16, 4, 352, 528, 1000),
          (16, 4, 736, 260, 300), (16, 2, 512, 768, 2000)]   # R, C, M, K, N


def main() -> int:
    import torch

    import oracle
    import synth
    import paper_2106_08846_gb300 as bsr
    from paper_2106_08846_gb300 import bsrlib as b
    from tests.gpu_util import build_on_gpu, check_product, to_dev, to_host
    fails = 0
    for k, (R, C, M, K, N) in enumerate(SHAPES):
        for rows in ("even", "uneven", "full"):
            MB, KB = M // R, K // C
            cnt = np.full(MB, max(1, int(0.3 * KB)), dtype=np.int64)
            seed = 9000 + 10 * k
            if rows != "even":   # short and empty rows, and a long one (split into pieces: partial tiles in the workspace)
                cnt[::2] = min(3, KB)
                cnt[1::5] = 0
            mask = synth.mask_from_row_counts(seed, cnt, KB)
            if rows != "even":   # 56 columns of every 64, the most of 32 rows that the ring's stages hold, or all
                mask[MB // 2] = (np.arange(KB) * C % 64 < 56) | (rows == "full")
            w = synth.make_weight("xc", seed, M, K, R, C, "f32", 0, mask=mask)
            h = bsr.bsr_create(*build_on_gpu(w.W, R, C), R, C, M, K)
            ref = oracle.bsr_from_dense(w.W, R, C)
            X = synth.activations(seed + 1, N, K, "f32")
            tokens = np.unique(np.concatenate([np.arange(0, N, 7), np.arange(max(0, N - 130), N)]))
            name = f"{R}x{C} {rows} M={M} K={K} N={N}"
            try:
                # (K = 100: the full row's pieces hold 50 columns of a chunk)
                kernel = "xstage" if rows == "full" and R == 32 and K != 100 else "xcol"
                assert h.call_info(N)["kernel"] == kernel, h.call_info(N)
                if rows != "even" and MB > 8:
                    assert h.schedule()["split_rows"] == 1 and h.schedule()["empty_rows"] > 0
                for bias in (w.bias, None):
                    Y = to_host(h.spmm(to_dev(X), None if bias is None else to_dev(bias)))
                    assert h.check_device_status() == 0
                    check_product(Y, ref, X, bias, M, rows=tokens)
                # infinities and NaN of X reach the rows that keep their column, and no others
                Xs = X.copy()
                Xs[0, 0], Xs[N // 2, K // 2], Xs[N - 1, K - 1] = np.inf, -np.inf, np.nan
                got = to_host(h.spmm(to_dev(Xs), to_dev(w.bias)))
                with np.errstate(invalid="ignore"):
                    want = oracle.bsr_spmm(*ref, Xs, w.bias, M)
                assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))
            except AssertionError as ex:
                fails += 1
                print(f"{name}: FAIL {str(ex)[:300]}", flush=True)
                continue
            print(f"{name}: ok", flush=True)
            h.destroy()
    # three products of one grid (not by length) are bit for bit the single calls
    X = to_dev(synth.activations(9201, 700, 512, "f32"))
    for R in (16, 32):
        ws = [synth.make_weight("xb", 9200 + i, 416, 512, R, 1, "f32", s) for i, s in enumerate((50, 90, 70))]
        hs = [bsr.bsr_create(*build_on_gpu(w.W, R, 1), R, 1, w.M, w.K) for w in ws]
        Ys = [torch.empty((700, w.M), device="cuda") for w in ws]
        bsr.bsr_spmm_batch(hs[::-1], X, None, Ys[::-1], 700)
        fails += sum(not torch.equal(h.spmm(X), Y) for h, Y in zip(hs, Ys))
    # a chunk that is never loaded: bounded waits, BSR_ERR_TIMEOUT, usable context
    os.environ.update(BSR_WAIT_LIMIT_NS="2000000", BSR_TEST_STALL_CHUNK="3")
    gpu = build_on_gpu(ws[0].W, 32, 1)
    h = bsr.bsr_create(*gpu, 32, 1, 416, 512)
    del os.environ["BSR_WAIT_LIMIT_NS"], os.environ["BSR_TEST_STALL_CHUNK"]
    h.spmm(X)
    fails += h.check_device_status() != b.BSR_ERR_TIMEOUT
    fails += not torch.equal(bsr.bsr_create(*gpu, 32, 1, 416, 512).spmm(X), Ys[0])
    print("failures:", fails)
    return 1 if fails else 0


if __name__ == "__main__":
    sys.exit(main())
