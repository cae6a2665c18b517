// SIMT kernel over column lists for fp32 blocks of 32 or 16 rows and up to four
// columns ("xcol").
//
// A warp multiplies an item (a block row) with 8 TT tokens: lane = tg + 8 rg,
// tg picks tokens tg, tg + 8, ..., rg a group of 8 output rows. Per column a
// lane loads TT activations and 8 weights from shared memory and does 8 TT
// multiply-adds, packed in pairs of tokens. For blocks of 16 rows a lane has 4
// outputs and TT = 16 tokens: the same multiply-adds, 20 words instead of 16.
//
// What bounds it: the FP32 pipe as the register file feeds it. A packed
// multiply-add reads three 64-bit operands; with the weight pair kept over
// consecutive instructions (tokens inside, outputs outside) it takes 2.5 cycles
// instead of 2, with the activations kept 3.4; plain ones run at 87% of the
// rate but leave no issue slots for the loads. Shared memory delivers 32 words
// a cycle whatever is broadcast: TT + 8 words for 8 TT multiply-adds, equal to
// the pipe's need at TT = 8 and 79% of it at TT = 14, the largest tile that
// three warps a scheduler have registers for.
//
// Persistent: one CTA per SM walks units (task of G items, token tile). The
// producer warp streams X chunks (two TMA boxes of 32 columns) and, beside
// each, the task's packed columns of that chunk (one bulk copy; one for each item
// took the producer longer than the warps: with 8 items a task, 2048 x 2048 at 70%,
// 2000 tokens 128 us, then 120) through a ring; every consumer warp waits for
// chunks, works through its columns and frees them, and goes on to the next unit
// when its own tile is stored: no barrier over all warps.
// Which items make a task and how many tokens a tile changes no output's bits, so a
// launch chooses both for all of its products together: few items a task spread a
// small call over the SMs (768 x 768 at 50%, 1024 tokens 43 -> 30 us), 48 products
// of 1024 tokens fill the GPU with larger ones (plan of 48 weights at 50 to 95%, of
// which those at 50% run here, 617 -> 499 us).
// Items of a task are neighbours in length, so warps stay within the ring of one
// another.
//
// So that an output is not one long chain of additions, a warp adds its tile to
// a running sum after every segment of chunks (at most about 40 columns, or one
// chunk; fewer, down to half a chunk, where the per-task kernel's error would be
// smaller: xcol_segment). A tile of 64 tokens has registers for a second set; for the larger ones
// registers and shared memory are full and the sums live in tensor memory, which
// nothing else uses here: a warp reaches 32 lanes of it, so up to three tiles of
// 112 columns. An addition there costs the largest tile about 1900 cycles (it
// spills a dozen registers around it): one chain per output would run 1024 x 1024
// at 90%, 16384 tokens in 86 us where this takes 99, with a relative error of
// 1.8e-7 instead of 1.15e-7 (the per-task kernel's: 1.33e-7).
//
// Measured, with the per-task kernel beside it: choose_xcol.
//
// Every wait is bounded by the global timer; a timeout sets the device status
// word, stops the CTA's roles, lets the issued copies land and returns.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>

#include "bsr_internal.h"
#include "launch.cuh"
#include "ptx.cuh"
#include "status.cuh"
#include "tcgen05.cuh"

namespace bsr {

namespace {

constexpr int NW = kXcWarps;
constexpr int kThreads = 32 * (NW + 1);
constexpr int kStagesMax = kXcStagesMax;
constexpr uint32_t kTmemCols = 512;   // three warps a lane quarter, a tile's 112 columns each (a power of two)
constexpr uint32_t kTileCols = 8 * kXcTT[kXcTileSizes - 1];   // of the largest tile
constexpr uint64_t kDrainNs = 200000000ull;

struct XcArgs {
    const int32_t *table;        // per chunk and item: the packed chunk's start / 16, in order (and the end)
    const unsigned char *packed;
    const Item *items;
    const float *bias;
    float *Y, *ws;
    int *status;
    int64_t M;
    uint64_t wait_ns;
    int n_items, n_tasks;
    int seg;                     // chunks per segment (0: two segments a chunk)
    unsigned tiles;
    int stall_chunk;
};

template <int MAXB>
struct XcBatch {
    int n, ns;
    uint32_t stage_bytes;   // a stage: two X boxes, then the items' packed chunks
    int nch;
    int64_t N;
    unsigned start[MAXB + 1];
    XcArgs args[MAXB];
};

typedef unsigned long long f2_t;   // two packed fp32
__device__ __forceinline__ f2_t pack2(float lo, float hi) {
    f2_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f2_t v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
// (volatile: in the order written)
__device__ __forceinline__ f2_t ffma2(f2_t a, f2_t b, f2_t c) {
    f2_t d;
    asm volatile("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ f2_t fadd2(f2_t a, f2_t b) {
    f2_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// The unit a CTA takes in its k-th turn (>= `units`: none). Several products come
// longest first: to and fro over the grid, so that a CTA's units add up to the
// same as another's.
__device__ __forceinline__ unsigned turn_unit(unsigned k, int products) {
    return k * gridDim.x + (products > 1 && k & 1 ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
}

struct Unit {
    int i0, n;    // first item, items
    int64_t n0;   // first token
};
template <int TT>
__device__ __forceinline__ Unit unit_at(const XcArgs &a, unsigned v) {
    Unit u;   // the tasks of a token tile side by side: their reads of X meet in L2
    const unsigned tile = v / (unsigned)a.n_tasks;
    unsigned task = v - tile * (unsigned)a.n_tasks;
    // where the grid is whole tiles, a CTA would have the same task (the longest,
    // say) in every turn: another one in each
    if (a.n_tasks > 1 && gridDim.x % (unsigned)a.n_tasks == 0)
        task = (task + tile / (gridDim.x / (unsigned)a.n_tasks)) % (unsigned)a.n_tasks;
    u.i0 = xcol_first((int)task, a.n_tasks, a.n_items);
    u.n = xcol_first((int)task + 1, a.n_tasks, a.n_items) - u.i0;
    u.n0 = (int64_t)tile * (8 * TT);
    return u;
}

// One column: TT activations at p and NR weights at w (the lane's first four
// outputs, and 16 further its last four).
template <int TT, int NR>
__device__ __forceinline__ void column(f2_t (&acc)[TT / 2][NR], const unsigned char *p, const float *w) {
    f2_t x[TT / 2];
#pragma unroll
    for (int i = 0; i < TT / 2; i++)
        x[i] = pack2(*reinterpret_cast<const float *>(p + 2 * i * 1024),
                     *reinterpret_cast<const float *>(p + (2 * i + 1) * 1024));
    float v[NR];
#pragma unroll
    for (int j = 0; j < NR; j += 4) {
        const float4 q = *reinterpret_cast<const float4 *>(w + 4 * j);
        v[j] = q.x, v[j + 1] = q.y, v[j + 2] = q.z, v[j + 3] = q.w;
    }
#pragma unroll
    for (int j = 0; j < NR; j++) {
        const f2_t wj = pack2(v[j], v[j]);
#pragma unroll
        for (int i = 0; i < TT / 2; i++) acc[i][j] = ffma2(x[i], wj, acc[i][j]);
    }
}

// HALF: segments of half a chunk occur (tiles whose running sums are in registers).
template <int MAXB, int TT, int NR, bool HALF>
__global__ void __launch_bounds__(kThreads, 1)
k_xcol(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ XcBatch<MAXB> b) {
    constexpr uint32_t kX = 2 * kXcBox;
    constexpr int R = 4 * NR;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = ptx::align_smem(smem_raw);
    __shared__ uint64_t full[kStagesMax], empty[kStagesMax];
    __shared__ int stop;
    __shared__ uint32_t tmem_s;
    __shared__ uint32_t place[kStagesMax][NW];   // where a stage's items begin
    const int ns = b.ns;
    const uint32_t stage_bytes = b.stage_bytes;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < ns; s++) {
            ptx::mbar_init(&full[s], 1);
            ptx::mbar_init(&empty[s], NW);
        }
        stop = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 0) tc5::alloc(&tmem_s, kTmemCols);
    tc5::fence_before();
    __syncthreads();
    tc5::fence_after();
    ptx::pdl_launch_dependents();   // (after the allocation: ptx.cuh)
    const unsigned units = b.start[b.n];
    const bool elected = ptx::elect_one();
    auto halt = [&](int *status) {
        if (elected) {
            if (!aborted(&stop)) set_status(status, DEV_TIMEOUT);
            atomicExch(&stop, 1);
        }
    };
    const int nch = b.nch;
    int h = 0, s = 0;

    if (warp == NW) {
        // ---------------- producer
        uint32_t phase = 1;   // the parity of `empty` that a first use of a stage passes at once
        uint32_t stalled = 0; // test hook: stages whose load was left out
        int issued = 0;
        bool ok = true, waited = false;
        if (elected) ptx::prefetch_tensormap(&xmap);
        for (unsigned k = 0, u; ok && k * gridDim.x < units; k++) {
            if ((u = turn_unit(k, b.n)) >= units) break;
            while (u >= b.start[h + 1]) h++;
            const XcArgs &a = b.args[h];
            const Unit un = unit_at<TT>(a, u - b.start[h]);
            // (the task's packed chunk is one range; lane g knows where item g's begins)
            const int32_t *tab = a.table + un.i0 + min(lane, un.n);
            int at = __ldg(tab);
            auto load_w = [&](int st, int v) {
                const int from = __shfl_sync(0xffffffffu, v, 0), to = __shfl_sync(0xffffffffu, v, un.n);
                if (lane < NW) place[st][lane] = (uint32_t)(v - from) * 16;
                __syncwarp();
                if (elected) {
                    const uint32_t bytes = (uint32_t)(to - from) * 16;
                    ptx::mbar_arrive_expect_tx(&full[st], 2 * TT * 1024 + bytes);
                    ptx::bulk_load(base + (size_t)st * stage_bytes + kX, a.packed + (int64_t)from * 16, bytes, &full[st]);
                }
                __syncwarp();
            };
            // the first columns do not depend on earlier kernels
            const int ahead = waited ? 0 : min(ns, nch);
            if (!waited) {
                for (int c = 0; c < ahead; c++)
                    if (c != a.stall_chunk) load_w(c, __ldg(tab + (int64_t)c * a.n_items));
                ptx::pdl_wait();   // X may be an earlier kernel's output
                waited = true;
            }
            for (int c = 0; c < nch; c++) {
                const int next = c + 1 < nch ? __ldg(tab + (int64_t)(c + 1) * a.n_items) : 0;
                // (the stages loaded ahead are free, and their X tiles always
                // follow: a barrier phase is never left half loaded)
                if (c >= ahead) {
                    const bool got = wait_or_abort(&empty[s], phase, a.wait_ns, &stop);
                    if (!__all_sync(0xffffffffu, got && !aborted(&stop))) {
                        halt(a.status);
                        ok = false;
                        break;
                    }
                }
                if (c == a.stall_chunk) {   // never loaded: its consumers time out
                    stalled |= 1u << s;
                } else {
                    if (c >= ahead) load_w(s, at);
                    if (elected) {
                        unsigned char *st = base + (size_t)s * stage_bytes;
                        ptx::tma_load_2d(st, &xmap, c * kXcChunk, (int32_t)un.n0, &full[s]);
                        ptx::tma_load_2d(st + kXcBox, &xmap, c * kXcChunk + 32, (int32_t)un.n0, &full[s]);
                    }
                }
                issued++;
                if (++s == ns) {
                    s = 0;
                    phase ^= 1;
                }
                at = next;
            }
        }
        // no copy may outlive the CTA (a stage that was consumed has landed long ago)
        for (int k = max(0, issued - ns); k < issued; k++)
            if (!((stalled >> (k % ns)) & 1)) ptx::mbar_wait_bounded(&full[k % ns], (uint32_t)(k / ns) & 1, kDrainNs);
        __syncwarp();
    } else {
        // ---------------- consumers
        const int tg = lane & 7, rg = lane >> 3;
        const uint32_t tgx = (uint32_t)tg << 4;
        ptx::pdl_wait();   // X, the bias, Y and the workspace may be an earlier kernel's; the waits are bounded from here on
        uint32_t phase = 0;
        bool ok = true;
        for (unsigned k = 0, u; ok && k * gridDim.x < units; k++) {
            if ((u = turn_unit(k, b.n)) >= units) break;
            while (u >= b.start[h + 1]) h++;
            const XcArgs &a = b.args[h];
            const bool has = warp < unit_at<TT>(a, u - b.start[h]).n;
            f2_t acc[TT / 2][NR];   // pairs of tokens
#pragma unroll
            for (int i = 0; i < TT / 2; i++)
#pragma unroll
                for (int j = 0; j < NR; j++) acc[i][j] = 0ull;
            constexpr bool kRegSums = TT * NR == 64;   // the running sums fit the registers
            f2_t total[kRegSums ? TT / 2 : 1][NR];
            if constexpr (kRegSums) {
#pragma unroll
                for (int i = 0; i < TT / 2; i++)
#pragma unroll
                    for (int j = 0; j < NR; j++) total[i][j] = 0x8000000080000000ull;   // -0: adds nothing, to any value
            }
            auto close = [&]() {   // total += acc, which starts anew
                if constexpr (kRegSums) {
#pragma unroll
                    for (int i = 0; i < TT / 2; i++)
#pragma unroll
                        for (int j = 0; j < NR; j++) {
                            total[i][j] = fadd2(acc[i][j], total[i][j]);
                            acc[i][j] = 0ull;
                        }
                }
            };
            auto sums = [&]() {   // this warp's running sums
                return tmem_s + ((uint32_t)(32 * (warp & 3)) << 16) +
                       (uint32_t)(warp >> 2) * kTileCols;
            };
            auto add_sums = [&]() {   // acc += the running sums
                const uint32_t at = sums();
                tc5::st_wait();
                // (as many loads at once as there are registers)
                constexpr int L = TT == 12 ? 16 : 8;
#pragma unroll
                for (int k = 0; k < NR * TT; k += L) {
                    uint32_t v[L / 8][8];
#pragma unroll
                    for (int l = 0; l < L / 8; l++) tc5::ld8(at + k + 8 * l, v[l]);
                    tc5::ld_wait();
#pragma unroll
                    for (int e = 0; e < L / 2; e++) {
                        uint32_t &v0 = v[e / 4][2 * (e % 4)], &v1 = v[e / 4][2 * (e % 4) + 1];
                        asm volatile("" : "+r"(v0), "+r"(v1));   // no use moves above the wait
                        f2_t &t = acc[(k / 2 + e) / NR][(k / 2 + e) % NR];
                        float even, odd;
                        unpack2(t, even, odd);
                        t = pack2(even + __uint_as_float(v0), odd + __uint_as_float(v1));
                    }
                }
            };
            const int seg = HALF ? max(a.seg, 1) : a.seg;
            for (int c = 0, c1 = seg; c < nch; c++) {
                if (!__all_sync(0xffffffffu, ptx::mbar_try_wait(&full[s], phase))) {
                    const bool got = wait_or_abort(&full[s], phase, 2 * a.wait_ns, &stop);
                    ok = __all_sync(0xffffffffu, got && !aborted(&stop));
                    if (!ok) {
                        halt(a.status);
                        break;
                    }
                }
                if (has) {
                    const unsigned char *st = base + (size_t)s * stage_bytes;
                    const unsigned char *xs = st + tg * 128;
                    const int4 *hdr = reinterpret_cast<const int4 *>(st + kX + place[s][warp]);
                    int n = hdr->x;   // columns; then their places, then their weights
                    const int4 *oc = hdr + 1;
                    const float *w = reinterpret_cast<const float *>(oc + ((n + 3) >> 2)) + 4 * rg;
                    const int mid = HALF && a.seg == 0 ? n - ((n >> 1) & ~3) : -1;   // columns left when a segment ends
                    for (; n >= 4; n -= 4, w += 4 * R) {
                        if (HALF && n == mid) close();
                        const int4 o = *oc++;
                        column<TT, NR>(acc, xs + ((uint32_t)o.x ^ tgx), w);
                        column<TT, NR>(acc, xs + ((uint32_t)o.y ^ tgx), w + R);
                        asm volatile("" ::: "memory");   // two columns' operands at a time: no more fit the registers
                        column<TT, NR>(acc, xs + ((uint32_t)o.z ^ tgx), w + 2 * R);
                        column<TT, NR>(acc, xs + ((uint32_t)o.w ^ tgx), w + 3 * R);
                        asm volatile("" ::: "memory");
                    }
                    if (n > 0) {
                        const int4 o = *oc;
                        column<TT, NR>(acc, xs + ((uint32_t)o.x ^ tgx), w);
                        if (n > 1) column<TT, NR>(acc, xs + ((uint32_t)o.y ^ tgx), w + R);
                        if (n > 2) column<TT, NR>(acc, xs + ((uint32_t)o.z ^ tgx), w + 2 * R);
                    }
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&empty[s]);
                if (++s == ns) {
                    s = 0;
                    phase ^= 1;
                }
                if (kRegSums && c + 1 == c1 && c1 < nch) {
                    close();
                    c1 += seg;
                } else if (!kRegSums && c + 1 == c1 && c1 < nch) {
                    if (c1 > seg) add_sums();
                    const uint32_t at = sums();
#pragma unroll
                    for (int k = 0; k < NR * TT; k += 8) {
                        uint32_t v[8];
#pragma unroll
                        for (int e = 0; e < 4; e++) {
                            f2_t &t = acc[(k / 2 + e) / NR][(k / 2 + e) % NR];
                            float even, odd;
                            unpack2(t, even, odd);
                            v[2 * e] = __float_as_uint(even);
                            v[2 * e + 1] = __float_as_uint(odd);
                            t = 0ull;
                        }
                        tc5::st8(at + k, v);
                    }
                    c1 += seg;
                }
            }
            if (!ok) break;
            if constexpr (kRegSums) {
#pragma unroll
                for (int i = 0; i < TT / 2; i++)
#pragma unroll
                    for (int j = 0; j < NR; j++) acc[i][j] = fadd2(acc[i][j], total[i][j]);
            } else if (nch > seg) {
                add_sums();
            }
            if (!has) continue;
            // (the unit once more: the registers are the columns' until here)
            const Unit un = unit_at<TT>(a, u - b.start[h]);
            // ---- the bias, and the item's rows of Y (or of its slot of the
            // workspace, for a piece of a split row)
            const Item it = a.items[un.i0 + warp];
            const bool partial = it.slot >= 0;
            const int64_t pitch = partial ? R : a.M;
            float *out = partial ? a.ws + (int64_t)it.slot * b.N * R : a.Y + (int64_t)it.row * R;
            const float *bias = a.bias && !partial ? a.bias + (int64_t)it.row * R : nullptr;
            float bv[NR];
#pragma unroll
            for (int j = 0; j < NR; j++) bv[j] = bias ? __ldg(bias + (j < 4 ? 4 * rg + j : 16 + 4 * rg + j - 4)) : 0.f;
#pragma unroll
            for (int i = 0; i < TT; i++) {
                float v[NR];
#pragma unroll
                for (int j = 0; j < NR; j++) {
                    float even, odd;
                    unpack2(acc[i >> 1][j], even, odd);
                    v[j] = i & 1 ? odd : even;
                }
                const int64_t t = un.n0 + tg + 8 * i;
                if (t < b.N) {
                    float *dst = out + t * pitch + 4 * rg;
#pragma unroll
                    for (int j = 0; j < NR; j += 4)
                        *reinterpret_cast<float4 *>(dst + 4 * j) =
                            make_float4(v[j] + bv[j], v[j + 1] + bv[j + 1], v[j + 2] + bv[j + 2], v[j + 3] + bv[j + 3]);
                }
            }
        }
        __syncwarp();
    }
    tc5::fence_before();
    __syncthreads();
    if (warp == 0) {
        tc5::fence_after();
        tc5::dealloc(tmem_s, kTmemCols);
    }
}

// Weights of every packed column: src[2 k] = float offset of its R weights,
// src[2 k + 1] = C times its stored block, plus its column in it.
__global__ void k_pack_xcol(const float *__restrict__ data, const int32_t *__restrict__ src, int64_t n, int R, int C,
                            float *__restrict__ out) {
    const int64_t total = n * R;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = e / R;
        const int r = (int)(e - k * R);
        const int32_t q = src[2 * k + 1], block = q / C;
        out[(int64_t)src[2 * k] + r] = data[((int64_t)block * R + r) * C + (q - block * C)];
    }
}
__global__ void k_pack_xcol_ints(const int32_t *__restrict__ pairs, int64_t n, int32_t *__restrict__ out) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        out[pairs[2 * k]] = pairs[2 * k + 1];
}

template <int MAXB, int TT, int NR, bool HALF>
cudaError_t launch(const LaunchArgs *las, int n, int G) {
    XcBatch<MAXB> b;
    b.n = 0;
    b.N = las[0].N;
    const int64_t K = las[0].sc->K;
    b.nch = (int)((K + kXcChunk - 1) / kXcChunk);
    uint32_t item_bytes = 0;
    int64_t units = 0;
    for (int i = 0; i < n; i++) {
        const LaunchArgs &la = las[i];
        const Schedule &sc = *la.sc;
        if (la.N == 0 || sc.items.empty()) continue;
        XcArgs &a = b.args[b.n];
        a.table = sc.xc.d_table;
        a.packed = static_cast<const unsigned char *>(la.data) + sc.xc.off;
        a.items = sc.d_items;
        a.bias = la.bias;
        a.Y = static_cast<float *>(la.Y);
        a.ws = la.ws;
        a.status = la.status;
        a.M = sc.M;
        a.wait_ns = la.wait_ns;
        a.n_items = (int)sc.items.size();
        a.n_tasks = (a.n_items + G - 1) / G;
        a.seg = xcol_segment(sc, la.N);
        if (!HALF) a.seg = std::max(a.seg, 1);   // (a larger tile that was asked for)
        a.tiles = (unsigned)((la.N + 8 * TT - 1) / (8 * TT));
        a.stall_chunk = la.stall_chunk;
        b.start[b.n] = (unsigned)units;
        units += (int64_t)a.tiles * a.n_tasks;
        item_bytes = std::max(item_bytes, sc.xc.item_bytes);
        b.n++;
        if (units > INT32_MAX) return cudaErrorInvalidConfiguration;
    }
    if (b.n == 0) return cudaSuccess;
    b.start[b.n] = (unsigned)units;
    b.stage_bytes = xcol_stage_bytes(item_bytes, G);
    b.ns = (int)std::min<uint32_t>(kXcStagesMax, kXcRoom / b.stage_bytes);
    if (b.ns < 1) return cudaErrorInvalidConfiguration;
    auto enc = tensor_map_encoder();
    if (!enc) return cudaErrorNotSupported;
    CUtensorMap map;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)b.N}, strides[1] = {(cuuint64_t)K * 4};
    const cuuint32_t box[2] = {32, 8 * TT}, estr[2] = {1, 1};
    if (enc(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void *>(las[0].X), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    static std::atomic<uint64_t> attr_set{0};
    cudaError_t e = allow_smem(k_xcol<MAXB, TT, NR, HALF>, kXcMaxSmem - 1024, attr_set);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)std::min<int64_t>(units, las[0].sc->sm_count);
    return launch_kernel(k_xcol<MAXB, TT, NR, HALF>, dim3(grid), dim3(kThreads), b.ns * b.stage_bytes + 1024, las[0].stream, map,
                         b);
}

template <int TT, int NR>
cudaError_t launch_n(const LaunchArgs *las, int n, int G) {
    if constexpr (TT * NR == 64) {
        bool half = false;
        for (int i = 0; i < n; i++) half |= xcol_segment(*las[i].sc, las[i].N) == 0;
        if (half) return n == 1 ? launch<1, TT, NR, true>(las, 1, G) : launch<kXcBatchMax, TT, NR, true>(las, n, G);
    }
    return n == 1 ? launch<1, TT, NR, false>(las, 1, G) : launch<kXcBatchMax, TT, NR, false>(las, n, G);
}

}  // namespace

cudaError_t pack_xcol_data(const Schedule &sc, const void *data, void *packed, cudaStream_t s) {
    const XcPlan &pl = sc.xc;
    unsigned char *out = static_cast<unsigned char *>(packed) + pl.off;
    const int64_t ni = (int64_t)pl.ints.size() / 2, nc = (int64_t)pl.src.size() / 2;
    if (ni)
        k_pack_xcol_ints<<<(int)std::min<int64_t>((ni + 255) / 256, 4096), 256, 0, s>>>(pl.d_ints, ni,
                                                                                       reinterpret_cast<int32_t *>(out));
    if (nc)
        k_pack_xcol<<<(int)std::min<int64_t>((nc * sc.R + 255) / 256, 1 << 16), 256, 0, s>>>(
            static_cast<const float *>(data), pl.d_src, nc, sc.R, sc.C, reinterpret_cast<float *>(out));
    return cudaGetLastError();
}

cudaError_t launch_xcol(const LaunchArgs *las, int n) {
    if (n <= 0) return cudaSuccess;
    if (n > kXcBatchMax) return cudaErrorInvalidValue;
    // the longest units first
    LaunchArgs sorted[kXcBatchMax];
    const Schedule *scs[kXcBatchMax];
    std::copy(las, las + n, sorted);
    auto length = [](const LaunchArgs &la) { return (double)la.sc->nnzb * la.sc->C / (double)std::max<size_t>(la.sc->items.size(), 1); };
    std::stable_sort(sorted, sorted + n, [&](const LaunchArgs &x, const LaunchArgs &y) { return length(x) > length(y); });
    for (int i = 0; i < n; i++) scs[i] = sorted[i].sc;
    const XcShape sh = xcol_shape(scs, n, las[0].N);
    if (scs[0]->R == 16) return launch_n<kXcTT16, 4>(sorted, n, sh.G);
    switch (kXcTT[sh.tile]) {
        case 8: return launch_n<8, 8>(sorted, n, sh.G);
        case 12: return launch_n<12, 8>(sorted, n, sh.G);
        case 14: return launch_n<14, 8>(sorted, n, sh.G);
    }
    return cudaErrorInvalidConfiguration;
}

}  // namespace bsr
