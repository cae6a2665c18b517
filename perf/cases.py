"""The product's measured work: what a program that uses this library has it do.

Every case goes through the public entry points (``bsr_from_dense``,
``bsr_spmm``, ``bsr_spmm_batch``, ``bsr_plan_create`` / ``Plan.launch``), on
pruned transformer weights in Block Sparse Row form and dense activations. The
sizes are those of the repository's workloads (BERT-base and BERT-large
attention projections, the block-shape sweep, the Zipf-row weight), with small
and ragged token counts beside them; ``draw`` varies all of them.

A case is a dict of plain values:
  kind      "spmm" (one product), "batch" (products sharing X in one call),
            "plan" (a captured sequence of independent products) or "build"
            (dense weight to BSR arrays)
  dtype     "f32" or "bf16"
  R, C      block shape; M, K weight shape; N tokens
  sparsity  share of the blocks removed, in per cent ("plan": of the first
            weight; the weights step through 50, 70, 80, 90 and 95 from there)
  rows      "uniform" (kept blocks anywhere) or "zipf" (Zipf(1.2) row lengths)
  weights   products of a "batch" or "plan" (1 otherwise)
  bias      whether the products add a bias
"""
import numpy as np
import torch

import paper_2106_08846_gb300 as bsr

_TORCH = {"f32": torch.float32, "bf16": torch.bfloat16}
_LEVELS = (50, 70, 80, 90, 95)
_SHAPES = ((1, 1), (4, 4), (8, 1), (16, 1), (32, 1), (1, 32), (16, 16), (32, 32))


def _case(name, kind, dtype, R, C, M, K, N, sparsity, rows="uniform", weights=1, bias=True):
    c = dict(kind=kind, dtype=dtype, R=R, C=C, M=M, K=K, N=N, sparsity=sparsity, rows=rows, weights=weights, bias=bias)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a request of one short sentence through one BERT-base projection: latency
        _case("base_f32_32x1_n128", "spmm", "f32", 32, 1, 768, 768, 128, 90),
        # a handful of tokens through a BERT-large projection in bf16: latency
        _case("large_bf16_16x16_n16", "spmm", "bf16", 16, 16, 1024, 1024, 16, 90),
        # a layer's query, key and value projections of a ragged batch, one call
        _case("qkv_f32_32x1_n1000", "batch", "f32", 32, 1, 768, 768, 1000, 80, weights=3),
        # irregular pruning (no block structure), a small batch
        _case("base_f32_1x1_n1024", "spmm", "f32", 1, 1, 768, 768, 1024, 80),
        # one-row blocks along the input features, ragged and without bias
        _case("base_f32_1x32_n900", "spmm", "f32", 1, 32, 768, 768, 900, 80, bias=False),
        # narrow blocks in bf16 at the size of a small serving batch
        _case("base_bf16_32x1_n1024", "spmm", "bf16", 32, 1, 768, 768, 1024, 80),
        # a large batch through a BERT-large projection: the benchmark's sizes
        _case("large_f32_32x1_n16384", "spmm", "f32", 32, 1, 1024, 1024, 16384, 90),
        _case("large_f32_16x16_n16384", "spmm", "f32", 16, 16, 1024, 1024, 16384, 90),
        _case("large_bf16_16x16_n16384", "spmm", "bf16", 16, 16, 1024, 1024, 16384, 90),
        # heavily unequal rows (a few hold most of the blocks)
        _case("zipf_bf16_16x16_n8192", "spmm", "bf16", 16, 16, 4096, 4096, 8192, 95, rows="zipf"),
        # every attention projection of BERT-base as one captured plan
        _case("plan_f32_32x1_n1024", "plan", "f32", 32, 1, 768, 768, 1024, 50, weights=48),
        # converting a pruned dense weight when a model is loaded
        _case("build_f32_32x1_4096", "build", "f32", 32, 1, 4096, 4096, 0, 90),
    ]


def draw(rng):
    """Another case of the same ranges: block shapes and types of the sweep,
    weights of 256 to 1536 features a side (a build: to 4096), 50 to 95 per
    cent removed, 1 to 16384 tokens."""
    def log_int(lo, hi):
        return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))

    kind = rng.choices(("spmm", "batch", "plan", "build"), (7, 1, 1, 1))[0]
    dtype = rng.choice(("f32", "bf16"))
    R, C = rng.choice(_SHAPES)
    sparsity = rng.randint(50, 95)
    rows = "zipf" if rng.random() < 0.15 else "uniform"
    if kind == "build":
        M, K = (32 * log_int(8, 128) for _ in range(2))
        return _case(None, kind, dtype, R, C, M, K, 0, sparsity, rows)
    M, K = (32 * log_int(8, 48) for _ in range(2))
    if C <= 8 and rng.random() < 0.3:
        K += 8 * rng.randint(1, 3)
    if R <= 8 and rng.random() < 0.3:
        M += 8 * rng.randint(1, 3)
    weights = rng.randint(2, 4) if kind == "batch" else rng.randint(4, 12) if kind == "plan" else 1
    N = log_int(1, 16384)
    if N > 8 and rng.random() < 0.5:
        N -= N % 8
    # multiply-adds of one pass: below the largest listed case's
    most = 6e8 if R == 1 else 1.5e9
    per_token = weights * M * K * (0.27 if kind == "plan" else 1 - sparsity / 100)
    return _case(None, kind, dtype, R, C, M, K, max(1, min(N, int(most / per_token))), sparsity, rows, weights,
                 rng.random() < 0.8)


def _levels(case):
    if case["kind"] != "plan":
        return [case["sparsity"]] * case["weights"]
    at = min(range(len(_LEVELS)), key=lambda i: abs(_LEVELS[i] - case["sparsity"]))
    return [_LEVELS[(at + i) % len(_LEVELS)] for i in range(case["weights"])]


def _kept(case, sparsity):
    return max(1, ((case["M"] // case["R"]) * (case["K"] // case["C"]) * (100 - sparsity) + 50) // 100)


def _zipf_lengths(MB, KB, keep, seed):
    """Row lengths min(KB, floor(c z)), z ~ Zipf(1.2), that add up to keep."""
    z = np.minimum(np.random.RandomState(seed % (1 << 32)).zipf(1.2, MB), 1 << 40).astype(np.float64)
    lo, hi = 0.0, float(keep + KB)
    for _ in range(80):
        mid = (lo + hi) / 2
        lo, hi = (mid, hi) if np.minimum(KB, np.floor(mid * z)).sum() < keep else (lo, mid)
    n = np.minimum(KB, np.floor(hi * z)).astype(np.int64)
    over = int(n.sum()) - keep
    for i in np.argsort(-n, kind="stable"):
        cut = min(over, int(n[i]))
        n[i] -= cut
        over -= cut
        if over <= 0:
            break
    return n


def _weight(case, sparsity, gen, seed):
    """A dense [M, K] weight with whole blocks removed, values N(0, 0.02)."""
    R, C, M, K = case["R"], case["C"], case["M"], case["K"]
    MB, KB, keep = M // R, K // C, _kept(case, sparsity)
    if case["rows"] == "zipf":
        n = torch.from_numpy(_zipf_lengths(MB, KB, keep, seed)).cuda()
        order = torch.rand(MB, KB, device="cuda", generator=gen).argsort(1)
        rank = torch.empty_like(order)
        rank.scatter_(1, order, torch.arange(KB, device="cuda").expand(MB, KB).contiguous())
        mask = rank < n[:, None]
    else:
        mask = torch.zeros(MB * KB, dtype=torch.bool, device="cuda")
        mask[torch.randperm(MB * KB, device="cuda", generator=gen)[:keep]] = True
        mask = mask.view(MB, KB)
    W = (torch.randn(M, K, device="cuda", generator=gen) * 0.02).to(_TORCH[case["dtype"]])
    W = torch.where(W == 0, torch.full_like(W, 0.02), W)   # a kept element is never zero
    return (W.view(MB, R, KB, C) * mask[:, None, :, None]).view(M, K)


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    Ws = [_weight(case, s, gen, int(seed) + 7919 * i) for i, s in enumerate(_levels(case))]
    X = torch.randn(case["N"], case["K"], device="cuda", generator=gen).to(_TORCH[case["dtype"]])
    biases = [torch.randn(case["M"], device="cuda", generator=gen) * 0.02 if case["bias"] else None for _ in Ws]
    return Ws, X, biases


def prepare(case, seed):
    Ws, X, biases = _inputs(case, seed)
    if case["kind"] == "build":
        return {"case": case, "W": Ws[0]}
    handles, Ys = [], []
    for W in Ws:
        arrays = bsr.bsr_from_dense(W, case["R"], case["C"], 0.0)
        handles.append(bsr.bsr_create(*arrays, case["R"], case["C"], case["M"], case["K"]))
        handles[-1].reserve(case["N"])
        Ys.append(torch.empty(case["N"], case["M"], dtype=X.dtype, device="cuda"))
    s = {"case": case, "handles": handles, "X": X, "biases": biases, "Ys": Ys}
    if case["kind"] == "plan":
        s["plan"] = bsr.bsr_plan_create(handles, [X] * len(Ws), biases, Ys, independent=True)
    return s


def run(state):
    kind = state["case"]["kind"]
    if kind == "build":
        return bsr.bsr_from_dense(state["W"], state["case"]["R"], state["case"]["C"], 0.0)
    if kind == "plan":
        state["plan"].launch()
        return state["Ys"]
    if kind == "batch":
        bsr.bsr_spmm_batch(state["handles"], state["X"], state["biases"], state["Ys"])
        return state["Ys"]
    bsr.bsr_spmm(state["handles"][0], state["X"], state["biases"][0], state["Ys"][0])
    return state["Ys"][0]


def work(case):
    es = 4 if case["dtype"] == "f32" else 2
    M, K, N = case["M"], case["K"], case["N"]
    kept = [_kept(case, s) for s in _levels(case)]
    arrays = sum(k * (case["R"] * case["C"] * es + 4) + 4 * (M // case["R"] + 1) for k in kept)
    if case["kind"] == "build":
        return {"bytes": M * K * es + arrays, "flops": 0}
    dense = N * K * es + len(kept) * (N * M * es + (4 * M if case["bias"] else 0))
    return {"bytes": arrays + dense, "flops": 2 * N * sum(kept) * case["R"] * case["C"]}


def tolerance(case):
    # build: a copy. Products: the 2-norm of another summation order (f32,
    # three-term tensor-core splits among them) or of one rounding to bf16.
    if case["kind"] == "build":
        return "exact"
    return {"rel": 4e-6, "max": 4e-5} if case["dtype"] == "f32" else {"rel": 7e-3, "max": 3e-2}


def exact(case, seed):
    Ws, X, biases = _inputs(case, seed)
    R, C, M, K = case["R"], case["C"], case["M"], case["K"]
    if case["kind"] == "build":
        blocks = Ws[0].view(M // R, R, K // C, C).transpose(1, 2)
        keep = (blocks != 0).flatten(2).any(2)
        indptr = torch.zeros(M // R + 1, dtype=torch.int32, device="cuda")
        indptr[1:] = keep.sum(1).cumsum(0)
        return indptr, keep.nonzero()[:, 1].to(torch.int32), blocks[keep].double()
    Ys = []
    for W, b in zip(Ws, biases):
        Y = X.double() @ W.double().T
        Ys.append(Y if b is None else Y + b.double())
    return Ys[0] if case["kind"] == "spmm" else Ys
