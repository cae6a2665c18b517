// GPU construction of the BSR arrays of a dense weight (Section 2.2: "data
// values, indices, and indptr", SciPy convention). A CTA works on a segment of
// one block row: up to about 32 KB of W (`nb` blocks of R x C).
//
//   k_count  blocks kept per segment: keep iff some |w| > thr (fp32 compare
//            written !(|w| <= thr), so NaN keeps a block);
//   k_scan   one CTA: exclusive scan over the rows and their segments -> indptr
//            and every segment's first kept block;
//   k_fill   reads its segment once into shared memory, marks and compacts its
//            kept block columns (ascending), and writes their values in block
//            order from there (consecutive threads, consecutive addresses).
//
// A query reads W once (k_count), a fill twice (k_count, k_fill; the second
// time from L2 where W fits it), by 16-byte loads where W and its rows are
// 16-byte aligned; what bounds a conversion beside that are the two calls'
// launches and synchronisations (about 65 us for a small weight). A conversion
// (query and fill, fp32, 4096 x 4096 at 90%, us; before: one thread per block, a
// flag per block in memory, one CTA per row compacting through 64-bit
// divisions): 32x1 98 (195), 16x16 97 (159), 1x1 191 (896), 64x64 of 2048 x 4096
// 82 (1110), 8x1 of 768 x 768 66 (102).
#include <cuda_bf16.h>

#include "bsr_internal.h"

namespace bsr {

namespace {

constexpr int kThreads = 256;
constexpr int kSegMax = 2048;        // blocks per segment
constexpr int kSegElems = 8192;      // elements per segment (more for one larger block: at most 4096 a block)

struct Seg {
    int64_t MB, KB, K;
    int R, C, nb;        // nb: blocks per segment
    int pitch;           // elements per row of a segment in shared memory
    int64_t nseg;        // segments per block row
    int vec;             // 16-byte loads
};

__device__ __forceinline__ bool kept(uint32_t bits, float thr) { return !(fabsf(__uint_as_float(bits)) <= thr); }
__device__ __forceinline__ bool kept(uint16_t bits, float thr) {
    return !(fabsf(__uint_as_float((uint32_t)bits << 16)) <= thr);
}

// The elements of one segment, row by row: f(row in the block row, column in
// the segment, bits). Threads take consecutive columns.
template <typename B, typename F>
__device__ __forceinline__ void for_segment(const B *__restrict__ W, const Seg &s, int64_t i, int64_t j0, int cols, F f) {
    constexpr int V = 16 / (int)sizeof(B);
    const B *base = W + i * s.R * s.K + j0 * s.C;
    if (s.vec && cols % V == 0) {
        const int nv = cols / V;
#pragma unroll 4
        for (int e = threadIdx.x; e < nv * s.R; e += kThreads) {
            const int r = e / nv, c = (e - r * nv) * V;
            const uint4 q = __ldg(reinterpret_cast<const uint4 *>(base + (int64_t)r * s.K + c));
            const B *v = reinterpret_cast<const B *>(&q);
#pragma unroll
            for (int k = 0; k < V; k++) f(r, c + k, v[k]);
        }
    } else {
#pragma unroll 4
        for (int e = threadIdx.x; e < cols * s.R; e += kThreads) {
            const int r = e / cols, c = e - r * cols;
            f(r, c, __ldg(base + (int64_t)r * s.K + c));
        }
    }
}

// Inclusive scan inside a warp.
__device__ __forceinline__ int64_t warp_scan(int64_t x, int lane) {
    for (int o = 1; o < 32; o <<= 1) {
        int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Exclusive block-wide scan of v over blockDim.x (a multiple of 32, <= 1024)
// threads; returns the exclusive prefix and writes the block total.
__device__ int64_t block_exclusive_scan(int64_t v, int64_t *total, int64_t *warp_tot) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int64_t x = warp_scan(v, lane);
    if (lane == 31) warp_tot[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int64_t t = lane < nw ? warp_tot[lane] : 0;
        t = warp_scan(t, lane);
        if (lane < nw) warp_tot[lane] = t;
    }
    __syncthreads();
    int64_t excl = x - v + (wid ? warp_tot[wid - 1] : 0);
    *total = warp_tot[nw - 1];
    __syncthreads();
    return excl;
}

// Whether block b of a segment keeps an element, from the marks of its columns.
__device__ __forceinline__ bool block_kept(const uint8_t *col_keep, int b, int C) {
    bool k = false;
    for (int c = 0; c < C; c++) k |= col_keep[b * C + c] != 0;
    return k;
}

template <typename B>
__global__ void __launch_bounds__(kThreads)
k_count(const B *__restrict__ W, const Seg s, float thr, int32_t *__restrict__ counts) {
    __shared__ uint8_t col_keep[kSegElems];
    __shared__ int total;
    for (int64_t t = blockIdx.x; t < s.MB * s.nseg; t += gridDim.x) {
        const int64_t i = t / s.nseg, j0 = (t - i * s.nseg) * s.nb;
        const int blocks = (int)min((int64_t)s.nb, s.KB - j0), cols = blocks * s.C;
        for (int c = threadIdx.x; c < cols; c += kThreads) col_keep[c] = 0;
        if (threadIdx.x == 0) total = 0;
        __syncthreads();
        for_segment(W, s, i, j0, cols, [&](int, int c, B v) {
            if (kept(v, thr)) col_keep[c] = 1;
        });
        __syncthreads();
        int n = 0;
        for (int b = threadIdx.x; b < blocks; b += kThreads) n += block_kept(col_keep, b, s.C);
        n = __reduce_add_sync(0xffffffffu, n);
        if ((threadIdx.x & 31) == 0 && n) atomicAdd(&total, n);
        __syncthreads();
        if (threadIdx.x == 0) counts[t] = total;
        __syncthreads();
    }
}

// counts [MB][nseg] -> indptr, in place the first kept block of every segment,
// and indptr[MB] once more in *nnzb (if given).
__global__ void k_scan(int32_t *__restrict__ counts, int64_t MB, int64_t nseg, int32_t *__restrict__ indptr,
                       int32_t *__restrict__ nnzb) {
    __shared__ int64_t warp_tot[32];
    int64_t carry = 0;
    if (threadIdx.x == 0) indptr[0] = 0;
    for (int64_t base = 0; base < MB; base += blockDim.x) {
        const int64_t idx = base + threadIdx.x;
        int64_t v = 0, total;
        if (idx < MB)
            for (int64_t k = 0; k < nseg; k++) v += counts[idx * nseg + k];
        const int64_t excl = block_exclusive_scan(v, &total, warp_tot);
        int64_t at = carry + excl;
        // An nnzb beyond int32 is reported as -1 and rejected by the host.
        if (idx < MB) {
            indptr[idx + 1] = at + v > INT32_MAX ? -1 : (int32_t)(at + v);
            for (int64_t k = 0; k < nseg; k++) {
                const int32_t c = counts[idx * nseg + k];
                counts[idx * nseg + k] = (int32_t)at;
                at += c;
            }
        }
        carry += total;
    }
    if (threadIdx.x == 0 && nnzb) *nnzb = carry > INT32_MAX ? -1 : (int32_t)carry;
}

template <typename B>  // B: uint32_t (fp32 bits) or uint16_t (bf16 bits)
__global__ void __launch_bounds__(kThreads)
k_fill(const B *__restrict__ W, const Seg s, float thr, const int32_t *__restrict__ first, int32_t *__restrict__ indices,
       B *__restrict__ data) {
    extern __shared__ unsigned char smem[];
    __shared__ int64_t warp_tot[32];
    const int pitch = s.pitch;
    B *seg = reinterpret_cast<B *>(smem);
    uint16_t *list = reinterpret_cast<uint16_t *>(seg + (((size_t)pitch * s.R + 7) & ~size_t(7)));
    uint8_t *col_keep = reinterpret_cast<uint8_t *>(list + s.nb);
    const int RC = s.R * s.C;
    for (int64_t t = blockIdx.x; t < s.MB * s.nseg; t += gridDim.x) {
        const int64_t i = t / s.nseg, j0 = (t - i * s.nseg) * s.nb;
        const int blocks = (int)min((int64_t)s.nb, s.KB - j0), cols = blocks * s.C;
        for (int c = threadIdx.x; c < cols; c += kThreads) col_keep[c] = 0;
        __syncthreads();
        for_segment(W, s, i, j0, cols, [&](int r, int c, B v) {
            seg[r * pitch + c] = v;
            if (kept(v, thr)) col_keep[c] = 1;
        });
        __syncthreads();
        // each thread's consecutive blocks, then their places among the kept ones
        const int per = (blocks + kThreads - 1) / kThreads;
        const int b0 = min(blocks, (int)threadIdx.x * per), b1 = min(blocks, b0 + per);
        int n = 0;
        for (int b = b0; b < b1; b++) n += block_kept(col_keep, b, s.C);
        int64_t total64;
        int at = (int)block_exclusive_scan(n, &total64, warp_tot);
        const int total = (int)total64;
        const int64_t p = first[t];
        for (int b = b0; b < b1; b++)
            if (block_kept(col_keep, b, s.C)) {
                indices[p + at] = (int32_t)(j0 + b);
                list[at++] = (uint16_t)b;
            }
        __syncthreads();
        B *out = data + p * RC;
        for (int e = threadIdx.x; e < total * RC; e += kThreads) {
            const int q = e / RC, rc = e - q * RC, r = rc / s.C, c = rc - r * s.C;
            out[e] = seg[r * pitch + list[q] * s.C + c];
        }
        __syncthreads();
    }
}

Seg segments(const void *W, int es, int64_t M, int64_t K, int R, int C) {
    Seg s;
    s.MB = M / R;
    s.KB = K / C;
    s.K = K;
    s.R = R;
    s.C = C;
    s.nb = std::max(1, std::min({kSegMax, kSegElems / (R * C), kSegElems / C}));
    // whole 16-byte vectors per segment where the rows allow them
    const int v = 16 / es;
    if (s.nb * C % v && s.nb >= v) s.nb -= s.nb % v;
    // odd: the rows of a block column in distinct banks (not for the tallest blocks: 48 KB)
    s.pitch = s.nb * C;
    if ((s.pitch | 1) * R <= kSegElems + 1024) s.pitch |= 1;
    s.nseg = std::max<int64_t>(1, (s.KB + s.nb - 1) / s.nb);
    s.vec = reinterpret_cast<uintptr_t>(W) % 16 == 0 && K * es % 16 == 0 && (s.nb * C * es) % 16 == 0;
    return s;
}

size_t fill_smem(const Seg &s, int es) {
    return (((size_t)s.pitch * s.R + 7) & ~size_t(7)) * es + (size_t)s.nb * 2 + (size_t)s.nb * s.C;
}

int grid_for(int64_t tasks) { return (int)std::max<int64_t>(1, std::min<int64_t>(tasks, 1 << 20)); }

}  // namespace

int64_t builder_segments(int64_t M, int64_t K, int R, int C, bsr_dtype_t dt) {
    const Seg s = segments(nullptr, (int)dtype_size(dt), M, K, R, C);
    return s.MB * s.nseg;
}

cudaError_t launch_builder_count(const void *W, bsr_dtype_t dt, int64_t M, int64_t K, int R, int C,
                                 float thr, int32_t *counts, int32_t *indptr, int32_t *nnzb, cudaStream_t s) {
    const Seg sg = segments(W, (int)dtype_size(dt), M, K, R, C);
    if (sg.MB * sg.KB > 0) {
        const int g = grid_for(sg.MB * sg.nseg);
        if (dt == BSR_F32)
            k_count<uint32_t><<<g, kThreads, 0, s>>>((const uint32_t *)W, sg, thr, counts);
        else
            k_count<uint16_t><<<g, kThreads, 0, s>>>((const uint16_t *)W, sg, thr, counts);
    } else if (sg.MB > 0) {
        cudaError_t e = cudaMemsetAsync(counts, 0, (size_t)(sg.MB * sg.nseg) * 4, s);
        if (e != cudaSuccess) return e;
    }
    k_scan<<<1, 1024, 0, s>>>(counts, sg.MB, sg.nseg, indptr, nnzb);
    return cudaGetLastError();
}

cudaError_t launch_builder_compact(const void *W, bsr_dtype_t dt, int64_t M, int64_t K, int R, int C, float thr,
                                   const int32_t *first, int32_t *indices, void *data, cudaStream_t s) {
    const Seg sg = segments(W, (int)dtype_size(dt), M, K, R, C);
    if (sg.MB == 0) return cudaSuccess;
    const int g = grid_for(sg.MB * sg.nseg);
    const size_t smem = fill_smem(sg, (int)dtype_size(dt));   // at most about 44 KB
    if (dt == BSR_F32)
        k_fill<uint32_t><<<g, kThreads, smem, s>>>((const uint32_t *)W, sg, thr, first, indices, (uint32_t *)data);
    else
        k_fill<uint16_t><<<g, kThreads, smem, s>>>((const uint16_t *)W, sg, thr, first, indices, (uint16_t *)data);
    return cudaGetLastError();
}

}  // namespace bsr
