"""Parity sweep of the dense-tile tensor-core kernel, for a process started
with BSR_DENSE_G (row groups per task) or BSR_DENSE=1 (the kernel's own
choice), or without (which kernel included). Run by tests/test_gpu_dense.py in a subprocess; exit status 0 when
every output is right."""
import os
import sys

import numpy as np

SHAPES = [  # R, C, M, K, N
    (16, 16, 272, 336, 1), (16, 16, 1040, 1024, 129), (32, 32, 256, 96, 127), (64, 16, 320, 208, 300),
    (128, 32, 256, 160, 1000), (32, 1, 416, 200, 257), (1, 1, 144, 72, 130), (4, 4, 272, 264, 128),
    (16, 64, 64, 64, 5000),
]


def main() -> int:
    import torch

    import oracle
    import synth
    import paper_2106_08846_gb300 as bsr
    from tests.gpu_util import as_f64, build_on_gpu, check_product, to_dev, to_host
    fails = 0
    for k, (R, C, M, K, N) in enumerate(SHAPES):
        for rows in ("even", "uneven"):
            MB, KB = M // R, K // C
            cnt = np.full(MB, max(1, int(0.4 * KB)), dtype=np.int64)
            if rows == "uneven":   # short, dense and empty rows: another order, tasks with few chunks
                cnt[::3] = 1
                cnt[1::5] = 0
                cnt[MB // 2] = KB
            seed = 7000 + 10 * k
            w = synth.make_weight("dn", seed, M, K, R, C, "bf16", 0, mask=synth.mask_from_row_counts(seed, cnt, KB))
            h = bsr.bsr_create(*build_on_gpu(w.W, R, C), R, C, M, K)
            ref = oracle.bsr_from_dense(w.W, R, C)
            X = synth.activations(seed + 1, N, K, "bf16")
            name = f"{R}x{C} {rows} M={M} K={K} N={N}"
            try:
                if "BSR_DENSE_G" in os.environ or "BSR_DENSE" in os.environ:
                    assert h.call_info(N)["kernel"] == "dense", h.call_info(N)
                Y = to_host(h.spmm(to_dev(X), to_dev(w.bias)))
                assert h.check_device_status() == 0
                check_product(Y, ref, X, w.bias, M)
                Y0 = to_host(h.spmm(to_dev(X), None))
                check_product(Y0, ref, X, None, M)
                # an output that is only 16-byte aligned (no 32-byte stores)
                buf = torch.empty(N * M + 8, dtype=torch.bfloat16, device="cuda")
                Yu = buf[8:].view(N, M)
                bsr.bsr_spmm(h, to_dev(X), to_dev(w.bias), Yu)
                assert np.array_equal(to_host(Yu), Y)
                # infinities and NaN of X reach the outputs of the rows that keep their columns, and no others
                Xs = X.copy()
                Xs[0, 0], Xs[N // 2, K // 2], Xs[N - 1, K - 1] = 0x7f80, 0xff80, 0x7fc1
                got = as_f64(to_host(h.spmm(to_dev(Xs), to_dev(w.bias))))
                with np.errstate(invalid="ignore"):
                    want = oracle.bsr_spmm(*ref, Xs, w.bias, M)
                assert np.array_equal(np.isnan(got), np.isnan(want)), "NaN outputs"
                inf = np.isinf(want)
                assert np.array_equal(np.isinf(got), inf) and np.array_equal(got[inf], want[inf]), "infinite outputs"
                clean = np.isfinite(as_f64(Xs)).all(1)
                assert np.array_equal(got[clean], as_f64(Y)[clean])
                fin = np.isfinite(want)
                E = oracle.err_bound(*ref, np.where(np.isfinite(as_f64(Xs)), Xs, 0).astype(np.uint16), w.bias, M)
                assert np.all(np.abs(got - want)[fin] <= 1e-2 * E[fin])
            except AssertionError as ex:
                fails += 1
                print(f"{name}: FAIL {str(ex)[:300]}", flush=True)
                continue
            print(f"{name}: ok", flush=True)
            h.destroy()
    torch.cuda.synchronize()
    return 1 if fails else 0


if __name__ == "__main__":
    sys.exit(main())
