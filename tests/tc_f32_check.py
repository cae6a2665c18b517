"""Parity sweep of the tensor-core kernel on fp32 blocks, for a process
started with BSR_TC_G (one task size, which fixes how many ring stages and
tensor-memory slots there are, where that size fits) and BSR_TC_F32_R16=1.
Run by tests/test_gpu_tc_f32.py in a subprocess; exit status 0 when every
output is right."""
import sys

import numpy as np

SHAPES = [  # R, C, K (in chunks of 32 columns: one, a half, fewer than the stages, many), N
    (16, 16, 32, 1), (16, 16, 112, 127), (16, 32, 160, 400), (16, 16, 1024, 300), (32, 16, 208, 129), (32, 32, 768, 1000),
    (64, 32, 64, 128), (64, 16, 528, 260), (128, 32, 96, 33), (128, 16, 720, 200)]


def main() -> int:
    import torch

    import oracle
    import synth
    import paper_2106_08846_gb300 as bsr
    from tests.gpu_util import build_on_gpu, check_product, to_dev, to_host
    fails = 0
    for k, (R, C, K, N) in enumerate(SHAPES):
        for rows in ("sparse", "dense"):
            MB, KB = 11 if R < 64 else 5, K // C
            M = MB * R
            cnt = np.full(MB, max(1, KB // 6) if rows == "sparse" else KB, dtype=np.int64)
            if rows == "sparse":   # empty rows, chunks without blocks, one dense row
                cnt[1::5] = 0
                cnt[MB // 2] = KB
            seed = 9500 + 10 * k
            w = synth.make_weight("tcf", seed, M, K, R, C, "f32", 0, mask=synth.mask_from_row_counts(seed, cnt, KB))
            h = bsr.bsr_create(*build_on_gpu(w.W, R, C), R, C, M, K)
            ref = oracle.bsr_from_dense(w.W, R, C)
            X = synth.activations(seed + 1, N, K, "f32")
            name = f"{R}x{C} {rows} K={K} N={N}"
            try:
                assert h.schedule()["variant"] == "tcgen05"
                for bias in (w.bias, None):
                    Y = to_host(h.spmm(to_dev(X), None if bias is None else to_dev(bias)))
                    assert h.check_device_status() == 0
                    check_product(Y, ref, X, bias, M)
                print(f"{name}: ok", flush=True)
            except AssertionError as ex:
                fails += 1
                print(f"{name}: FAIL {str(ex)[:300]}", flush=True)
            h.destroy()
            torch.cuda.synchronize()
    return 1 if fails else 0


if __name__ == "__main__":
    sys.exit(main())
