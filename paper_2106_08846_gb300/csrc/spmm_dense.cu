// Dense-tile tcgen05 kernel for bf16 weights ("dense").
//
// A block-sparse weight of transformer size costs the tensor cores less as a
// zero-filled dense product than block by block: an MMA of M = 128 tokens and
// K = 16 takes 39 SM cycles at N = 16 (its A tile's shared-memory read) and
// 128 at N = 256, so one 16-row block costs as much as five rows-of-16 of a
// full-width MMA, and a list of blocks has to be decoded between MMAs. Here
// the weight is packed once as dense rows (only the 16-row groups that hold a
// block), tasks are up to 256 of those rows, and the 64-column chunks in
// which no row of a task has a block are skipped.
//
//   warps 0, 1  producers: per chunk the X tile [128 tokens x 64] and the
//               weight tile [16 g rows x 64] by 2-D TMA (128-byte swizzle)
//               into one stage of a ring of up to 8 (as many as fit)
//   warp 2      four MMAs (K = 16 each, N = 16 g) per chunk; a commit frees
//               the stage, another hands the finished unit to the epilogue
//   warps 3..6  epilogue of 32 tokens each: accumulators from tensor memory,
//               bias, bf16, one 32-byte store per token and row group straight
//               from registers
//
// Persistent: one CTA per SM walks units (token tile, task); two accumulator
// buffers of 256 tensor-memory columns let a unit's epilogue overlap the next
// unit's MMAs, and the ring runs on across units.
//
// What bounds it: shared memory. At N = 256 a chunk is 512 cycles of MMAs; its
// tiles (X 16 KB, weight 32 KB) are written once and read once, 96 KB at 128
// bytes a cycle = 750 cycles. A pair of CTAs keeps half of the weight tile
// each: 64 KB, 512 cycles. So that nothing else passes through it, Y is stored
// from registers.
//
// Measured (us, back to back, the block-by-block kernel in brackets): 1024 x
// 1024 at 90%, 16384 tokens, 16x16 blocks 26.4 (34.5), 32x1 26.5 (55.5); 4096 x
// 4096 at 95% with Zipf rows, 8192 tokens, 16x16 33.2 (123.6); 768 x 768 at 80%,
// 1024 tokens, 32x1 6.4 (8.4); 1024 x 1024, 16 tokens 5.2 (6.4). One thread
// per role, in a branch that the compiler cannot see to be uniform, had put 424
// cycles into a producer's step and 340 into four MMAs and a commit; whole
// warps with one elected lane take 200 and 59, and the two loads of a stage
// come from two warps. Y staged through shared memory for TMA stores took 1000
// to 1900 cycles per 64 columns, waiting behind the tiles.
//
// Zeros (-0, which no kept element is packed as) stand for absent blocks, so an
// infinity or NaN of X in a column that an output's row does not keep would
// make that output NaN (0 x inf). Finite X gives exactly the kept blocks' sum,
// and a zero product can only turn an output into NaN, never into another
// finite value; so every output whose accumulator is NaN is computed again,
// without what is absent, by the epilogue warp that stored it, once the
// accumulators are handed on. That takes far longer than the product: 1024 x
// 1024 at 90%, 32x1, 16384 tokens 130 us with one such token, 330 us with every
// 97th, 8.4 ms with a NaN in every token (39 us without, each call by itself;
// one lane walking each output's blocks, with the accumulators held, had taken
// 5.1, 15 and 46 ms, and at K = 8192 350 ms where it is now 23).
//
// Launched with programmatic stream serialisation: the barriers, tensor
// memory and the first weight tiles come before the wait for the previous
// kernel; X, the bias and Y after it. Every wait is bounded by the global
// timer; a timeout sets the device status word, stops every role, lets the
// issued copies and MMAs finish, frees the tensor memory and returns.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>

#include "bsr_internal.h"
#include "elem.cuh"
#include "launch.cuh"
#include "ptx.cuh"
#include "status.cuh"
#include "tcgen05.cuh"

namespace bsr {

namespace {

constexpr int TN = kDnTokens;
constexpr int KC = kDnChunk;
constexpr uint32_t kXBytes = TN * 128;             // one X tile: 128 rows of 128 bytes
constexpr int kEpiWarps = 4;
constexpr int kMmaWarp = 2;                        // after the two producers
constexpr int kThreads = 32 * (kMmaWarp + 1 + kEpiWarps);
constexpr uint32_t kBiasBytes = kEpiWarps * 256 * 4;
constexpr uint32_t kAccCols = 256;                 // tensor-memory columns per accumulator buffer
constexpr uint16_t kAbsent = 0x8000;               // -0: what the packed weight holds where no block is
constexpr uint64_t kDrainNs = 200000000ull;        // bound for copies and MMAs already issued

struct DnArgs {
    CUtensorMap wmap;             // packed weight [16 n_full, K], boxes of 16 g (a pair's CTA: 8 g) rows x 64 columns
    const int32_t *table;         // task list offsets, then chunk lists
    const int32_t *group_row;
    const uint16_t *w;            // the packed weight
    const float *bias;
    uint16_t *Y;
    int *status;
    int64_t M;
    uint64_t wait_ns;
    int g, n_groups, n_full, n_tasks, n_work;   // n_full: groups with packed rows; n_work: tasks with chunks (they come first)
    unsigned tiles;
    int task_major;               // units task by task (unequal tasks), else tile by tile
    int stall_chunk;
    int y32;                      // Y is 32-byte aligned: its rows take 32-byte stores
};

struct Unit {
    int task;
    int64_t n0;   // the unit's first token
    const int32_t *list;
    int n;   // chunks
};

template <bool PAIR>
__device__ __forceinline__ Unit unit_at(const DnArgs &a, unsigned v) {
    Unit u;
    unsigned tile;
    if (a.task_major) {
        u.task = (int)(v / a.tiles);
        tile = v - (unsigned)u.task * a.tiles;
        u.task += a.n_work;   // tasks without chunks first
        if (u.task >= a.n_tasks) u.task -= a.n_tasks;
    } else {
        tile = v / (unsigned)a.n_tasks;
        u.task = (int)(v - tile * (unsigned)a.n_tasks);
    }
    u.n0 = (int64_t)tile * (PAIR ? 2 * TN : TN);
    const int lo = __ldg(a.table + u.task), hi = __ldg(a.table + u.task + 1);
    u.list = a.table + lo;
    u.n = hi - lo;
    return u;
}


// Two values rounded to nearest even, the first in the low half.
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// acc[r] = the sum over a unit's n chunks (eights of columns first, first +
// step, ...) of activation times packed row r, leaving out what is absent.
template <typename Beat>
__device__ __forceinline__ void kept_sums(float (&acc)[kDnGroup], const uint16_t *x, const uint16_t *w, int64_t K,
                                          const int32_t *list, int n, int first, int step, Beat beat) {
#pragma unroll
    for (int r = 0; r < kDnGroup; r++) acc[r] = 0.f;
    int64_t col_next = K;   // the next eight columns and their activations, on their way (K: none; a multiple of 8)
    uint4 x_next = {};
    auto fetch = [&](int v) {
        if (v < 8 * n) col_next = min(K, (int64_t)__ldg(list + (v >> 3)) * KC + 8 * (v & 7));
        if (col_next < K) x_next = __ldg(reinterpret_cast<const uint4 *>(x + col_next));
    };
    fetch(first);
    for (int v = first, k = 0; v < 8 * n; v += step, k++) {
        if ((k & 31) == 0) beat();
        const int64_t col = col_next;
        const uint4 xq = x_next;
        fetch(v + step);
        if (col >= K) continue;
        const uint32_t xw[4] = {xq.x, xq.y, xq.z, xq.w};
        float xf[8];
        bool finite = true;
#pragma unroll
        for (int e = 0; e < 8; e++) {
            xf[e] = __uint_as_float(e & 1 ? xw[e / 2] & 0xffff0000u : xw[e / 2] << 16);
            finite = finite && (__float_as_uint(xf[e]) & 0x7f800000u) != 0x7f800000u;
        }
        if (finite) {   // (times -0 adds nothing)
#pragma unroll
            for (int r = 0; r < kDnGroup; r++) {
                const uint4 wq = __ldg(reinterpret_cast<const uint4 *>(w + r * K + col));
                const uint32_t ww[4] = {wq.x, wq.y, wq.z, wq.w};
#pragma unroll
                for (int e = 0; e < 8; e++)
                    acc[r] = fmaf(xf[e], __uint_as_float(e & 1 ? ww[e / 2] & 0xffff0000u : ww[e / 2] << 16), acc[r]);
            }
        } else {
#pragma unroll 1
            for (int e = 0; e < 8; e++) {
                const float xv = to_f32(__ldg(x + col + e));
#pragma unroll
                for (int r = 0; r < kDnGroup; r++) {
                    const uint16_t wv = __ldg(w + r * K + col + e);
                    if (wv != kAbsent) acc[r] = fmaf(xv, to_f32(wv), acc[r]);
                }
            }
            bool nan = true;   // more terms leave NaN sums so
#pragma unroll
            for (int r = 0; r < kDnGroup; r++) nan = nan && acc[r] != acc[r];
            if (nan) break;
        }
    }
}

// Computes the NaN outputs of a unit's part again, for one warp's 32 tokens
// from n0 on: row groups g0 .. g0 + gn - 1 (lane j knows the output rows 16 gl
// of group j) over the unit's chunks. Bit j / 4 of this lane's `bad`: its token
// may have such an output in group j. A few tokens of a group share the warp, a
// lane taking every 32nd eight of columns; more take a lane each. `beat` is set
// time and again, here and in the other CTA of a pair (remote: 0 without one).
__device__ __noinline__ void compute_again(const DnArgs &a, const uint16_t *X, int64_t K, int64_t n0, int g0, int gn, int gl,
                                           const int32_t *list, int chunks, uint32_t bad, int *beat_s, uint32_t remote) {
    const int lane = threadIdx.x & 31;
    __syncwarp();   // (other lanes' outputs are stored)
    for (int j = 0; j < gn; j++) {
        const int64_t row0 = (int64_t)__shfl_sync(0xffffffffu, gl, j) * kDnGroup;
        bool any = false;   // this lane's token has a NaN output in the group
        if ((bad >> (j >> 2)) & 1)
            for (int e = 0; e < kDnGroup; e++) any |= (a.Y[(n0 + lane) * a.M + row0 + e] & 0x7fffu) > 0x7f80u;
        const uint32_t tokens = __ballot_sync(0xffffffffu, any);
        if (!tokens) continue;
        const bool lane_each = __popc(tokens) > 4;
        const int speaker = lane_each ? __ffs(tokens) - 1 : 0;
        auto beat = [&]() {
            if (lane == speaker) {
                const uint32_t t = (uint32_t)ptx::globaltimer() | 1u;
                *reinterpret_cast<volatile int *>(beat_s) = (int)t;
                if (remote) ptx::store_cluster(remote, t);
            }
        };
        const uint16_t *w = a.w + (int64_t)(g0 + j) * kDnGroup * K;
        const int n = g0 + j < a.n_full ? chunks : 0;   // (groups without blocks have no packed rows)
        float acc[kDnGroup];
        if (lane_each) {
            if (any) {
                const int64_t t = n0 + lane;
                kept_sums(acc, X + t * K, w, K, list, n, 0, 1, beat);
                uint16_t *y = a.Y + t * a.M + row0;
#pragma unroll
                for (int r = 0; r < kDnGroup; r++)
                    if ((y[r] & 0x7fffu) > 0x7f80u)
                        y[r] = from_f32<uint16_t>(acc[r] + (a.bias ? __ldg(a.bias + row0 + r) : 0.f));
            }
        } else {
            for (uint32_t left = tokens; left; left &= left - 1) {
                const int64_t t = n0 + __ffs(left) - 1;
                kept_sums(acc, X + t * K, w, K, list, n, lane, 32, beat);
                __syncwarp();
                float mine = 0.f;   // row `lane`'s sum
#pragma unroll
                for (int r = 0; r < kDnGroup; r++) {
#pragma unroll
                    for (int d = 16; d > 0; d >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], d);
                    if (r == lane) mine = acc[r];
                }
                uint16_t *y = a.Y + t * a.M + row0 + lane;
                if (lane < kDnGroup && (*y & 0x7fffu) > 0x7f80u)
                    *y = from_f32<uint16_t>(mine + (a.bias ? __ldg(a.bias + row0 + lane) : 0.f));
            }
        }
        __syncwarp();
    }
}

// Several products that share X in one grid: product h owns units start[h] ..
// start[h + 1] - 1.
template <int MAXB>
struct DnBatch {
    int n;
    int ns;                  // ring stages
    uint32_t stage_bytes;    // X tile and the largest weight tile of the batch
    const uint16_t *X;       // [N, K]
    int64_t N, K;
    unsigned start[MAXB + 1];
    DnArgs args[MAXB];
};

// PAIR: a cluster of two CTAs works on 256 tokens; each loads its own 128
// tokens of X and half of the weight tile's rows, and the first CTA issues
// MMAs of M = 256 for both.
template <int MAXB, bool PAIR>
__global__ void __launch_bounds__(kThreads, 1)
k_dense(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ DnBatch<MAXB> b) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = ptx::align_smem(smem_raw);
    const int ns = b.ns;
    const uint32_t stage_bytes = b.stage_bytes;
    float *bias_s = reinterpret_cast<float *>(base + (size_t)ns * stage_bytes);
    __shared__ uint64_t full[kDnStagesMax], empty[kDnStagesMax], acc_full[2], acc_empty[2], done;
    __shared__ int stop, loads[2][2];   // loads[producer][CTA of the pair]: loads issued
    __shared__ int freed, handed;       // commits issued to `empty` and to `acc_full`
    __shared__ int beat;                // changes while an epilogue warp computes outputs again
    __shared__ uint32_t tmem_s;

    // (a shuffle, so that the warp index and what follows from it is uniform)
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const uint32_t rank = PAIR ? ptx::cluster_rank() : 0;
    const unsigned cta = PAIR ? blockIdx.x >> 1 : blockIdx.x, ctas = PAIR ? gridDim.x >> 1 : gridDim.x;
    if (threadIdx.x == 0) {
        for (int s = 0; s < ns; s++) {
            ptx::mbar_init(&full[s], 2);   // the X producer's and the weight producer's arrivals, and their bytes
            ptx::mbar_init(&empty[s], 1);
        }
        for (int i = 0; i < 2; i++) {
            ptx::mbar_init(&acc_full[i], 1);
            ptx::mbar_init(&acc_empty[i], PAIR ? 2 * kEpiWarps : kEpiWarps);
        }
        ptx::mbar_init(&done, 1);
        stop = freed = handed = beat = 0;
        ptx::fence_barrier_init();
    }
    if (warp == kMmaWarp) {
        if constexpr (PAIR) tc5::alloc_pair(&tmem_s, 2 * kAccCols);
        else tc5::alloc(&tmem_s, 2 * kAccCols);
    }
    tc5::fence_before();
    __syncthreads();
    if constexpr (PAIR) ptx::cluster_barrier();   // the other CTA's barriers exist
    tc5::fence_after();
    ptx::pdl_launch_dependents();   // (after the allocation: ptx.cuh)
    const uint32_t tmem = tmem_s;
    const unsigned units = b.start[b.n];
    const bool elected = ptx::elect_one();
    // stops every role of this CTA (and its pair); a timeout is recorded
    auto halt = [&](int *status) {
        if (elected) {
            if (!aborted(&stop)) set_status(status, DEV_TIMEOUT);
            atomicExch(&stop, 1);
            if constexpr (PAIR) ptx::store_cluster(ptx::map_to_cta(&stop, rank ^ 1), 1);
        }
    };

    // ---- producers: warp 0 X tiles, warp 1 weight tiles, each over the CTA's
    // units and their chunks
    const int prod = warp;
    const CUtensorMap *map = &xmap;
    const int32_t *list = nullptr;
    unsigned u = cta;
    int h = 0, k = 0, n = 0, row = 0, stall = -1, s = 0, issued = 0, c_next = 0;
    uint32_t bytes = 0, phase = 1;   // phase: the parity of `empty` that a first use of a stage passes at once
    uint32_t stalled = 0;            // test hook: stages whose load was left out
    uint64_t wait_ns = 0;
    int *status = nullptr;
    const uint32_t dst0 = ptx::smem_addr(base) + (prod ? kXBytes : 0), bar0 = ptx::smem_addr(&full[0]);
    const uint32_t first0 = PAIR ? ptx::map_to_cta(&full[0], 0) : bar0;   // `full` of the pair's first CTA
    uint32_t dst = dst0;
    // moves to the first chunk at or after unit u; false: none left
    auto seek = [&]() {
        for (; u < units; u += ctas) {
            while (u >= b.start[h + 1]) h++;
            const DnArgs &a = b.args[h];
            const Unit un = unit_at<PAIR>(a, u - b.start[h]);
            if (un.n == 0) continue;
            list = un.list;
            n = un.n;
            k = 0;
            c_next = __ldg(list);
            stall = a.stall_chunk;
            wait_ns = a.wait_ns;
            status = a.status;
            if (prod) {
                map = &a.wmap;
                row = un.task * a.g * kDnGroup + (PAIR ? (int)rank * a.g * kDnGroup / 2 : 0);
                bytes = (uint32_t)a.g * kDnGroup * 128;
            } else {
                row = (int)(un.n0 + rank * TN);
                bytes = PAIR ? 2 * kXBytes : kXBytes;
            }
            return true;
        }
        return false;
    };
    // loads the chunk at the cursor into stage s and moves on; false: none left
    auto load_chunk = [&]() {
        const int c = c_next;
        if (++k < n) c_next = __ldg(list + k);   // in flight during the next wait
        if (c == stall) {                        // never loaded: its consumer times out
            stalled |= 1u << s;
        } else if (elected) {
            if (rank == 0) ptx::mbar_arrive_expect_tx_at(bar0 + 8 * s, bytes);
            if constexpr (PAIR) ptx::tma_load_2d_pair_at(dst, map, c * KC, row, first0 + 8 * s);
            else ptx::tma_load_2d_at(dst, map, c * KC, row, bar0 + 8 * s);
        }
        issued++;
        dst += stage_bytes;
        if (++s == ns) {
            s = 0;
            phase ^= 1;
            dst = dst0;
        }
        if (k < n) return true;
        u += ctas;
        return seek();
    };
    bool more = false;
    if (warp < 2) {
        if (elected) ptx::prefetch_tensormap(&xmap);
        more = seek();
        // X may be an earlier kernel's output; the packed weight is not, and the
        // first ns stages are free. The next ones are when the MMAs have read X:
        // their limit does not run while an earlier kernel does
        if (prod)
            while (more && issued < ns) more = load_chunk();
        ptx::pdl_wait();
        while (more) {
            const bool got = wait_or_abort(&empty[s], phase, wait_ns, &stop, &beat);
            if (!__all_sync(0xffffffffu, got && !aborted(&stop))) {
                halt(status);
                break;
            }
            more = load_chunk();
        }
        if (elected) {
            loads[prod][rank] = issued;
            if constexpr (PAIR) ptx::store_cluster(ptx::map_to_cta(&loads[prod][rank], rank ^ 1), (uint32_t)issued);
        }
    } else if (warp == kMmaWarp) {
        if (rank == 0) {
            int ab = 0, n_freed = 0, n_handed = 0;
            uint32_t fphase = 0, aphase = 1;
            bool ok = true;
            const uint64_t ad0 = tc5::desc_sw128(ptx::smem_addr(base)), step = stage_bytes >> 4;
            uint64_t ad = ad0;
            ptx::pdl_wait();   // the waits below are bounded from here on
            for (; ok && u < units; u += ctas) {
                while (u >= b.start[h + 1]) h++;
                const DnArgs &a = b.args[h];
                const Unit un = unit_at<PAIR>(a, u - b.start[h]);
                if (un.n == 0) continue;
                const uint32_t id = tc5::idesc(false, PAIR ? 2 * TN : TN, a.g * kDnGroup);
                const uint32_t d = tmem + (uint32_t)ab * kAccCols;
                ok = __all_sync(0xffffffffu, wait_or_abort(&acc_empty[ab], aphase, a.wait_ns, &stop, &beat));
                tc5::fence_after();
                for (int i = 0; ok && i < un.n; i++) {
                    ok = __all_sync(0xffffffffu, wait_or_abort(&full[s], fphase, a.wait_ns, &stop, &beat));
                    if (!ok) break;
                    tc5::fence_after();
                    if (elected) {
                        const uint64_t bd = ad + (kXBytes >> 4);
#pragma unroll
                        for (int j = 0; j < KC / 16; j++) {   // 16 columns = 32 bytes along the swizzled rows
                            if constexpr (PAIR) tc5::mma_ss_pair(d, ad + 2 * j, bd + 2 * j, id, (i > 0) | (j > 0));
                            else tc5::mma_ss<false>(d, ad + 2 * j, bd + 2 * j, id, (i > 0) | (j > 0));
                        }
                        if constexpr (PAIR) tc5::commit_pair(&empty[s]);
                        else tc5::commit(&empty[s]);
                    }
                    __syncwarp();
                    n_freed++;
                    ad += step;
                    if (++s == ns) {
                        s = 0;
                        fphase ^= 1;
                        ad = ad0;
                    }
                }
                if (!ok) {
                    halt(a.status);
                    break;
                }
                if (elected) {
                    if constexpr (PAIR) tc5::commit_pair(&acc_full[ab]);
                    else tc5::commit(&acc_full[ab]);
                }
                __syncwarp();
                n_handed++;
                ab ^= 1;
                if (ab == 0) aphase ^= 1;
            }
            // every MMA issued has completed before the tensor memory is freed
            if (elected) {
                if constexpr (PAIR) tc5::commit_pair(&done);
                else tc5::commit(&done);
                freed = n_freed;
                handed = n_handed;
                if constexpr (PAIR) {
                    ptx::store_cluster(ptx::map_to_cta(&freed, 1), (uint32_t)n_freed);
                    ptx::store_cluster(ptx::map_to_cta(&handed, 1), (uint32_t)n_handed);
                }
            }
            __syncwarp();
            ptx::mbar_wait_bounded(&done, 0, kDrainNs);
        }
    } else {
        const int q = warp & 3;        // this warp's tensor-memory lanes (and tokens) 32 q ..
        const int ew = warp - kMmaWarp - 1;
        float *bs = bias_s + ew * 256;
        ptx::pdl_wait();   // the bias and Y may be an earlier kernel's
        int ab = 0;
        uint32_t fphase = 0;
        bool ok = true;
        for (; ok && u < units; u += ctas) {
            while (u >= b.start[h + 1]) h++;
            const DnArgs &a = b.args[h];
            const Unit un = unit_at<PAIR>(a, u - b.start[h]);
            const int g0 = un.task * a.g;                      // the task's first row group position
            const int gn = min(a.g, a.n_groups - g0);
            const int64_t nw = un.n0 + rank * TN + 32 * q;     // this warp's first token
            // the output rows of the unit's groups and their biases, on their way
            // while the MMAs run
            const int gl = lane < gn ? __ldg(a.group_row + g0 + lane) : -1;
            float bv[8];
#pragma unroll
            for (int j = 0; j < 8; j++) {   // unit columns lane + 32 j
                const int gj = __shfl_sync(0xffffffffu, gl, 2 * j + (lane >> 4) & 15);
                bv[j] = a.bias && gj >= 0 ? __ldg(a.bias + gj * 16 + (lane & 15)) : 0.f;
            }
            if (un.n > 0) {
                const bool got = wait_or_abort(&acc_full[ab], fphase, a.wait_ns * (uint64_t)(un.n + 2), &stop, &beat);
                ok = __all_sync(0xffffffffu, got);
                if (!ok) {
                    halt(a.status);
                    break;
                }
                tc5::fence_after();
            }
            const uint32_t tm = tmem + (uint32_t)ab * kAccCols + ((uint32_t)(32 * q) << 16);
            __syncwarp();   // (the last unit's biases have been read)
#pragma unroll
            for (int j = 0; j < 8; j++) bs[lane + 32 * j] = bv[j];
            __syncwarp();   // (other lanes read them)
            const int64_t nt = nw + lane;                      // this thread's token
            uint16_t *const yrow = a.Y + nt * a.M;
            uint32_t bad = 0;                                  // fours of groups with a NaN or infinite sum of this token
            for (int gq = 0; gq < gn; gq += 4) {               // 64 columns: four row groups
                const int cnt = min(4, gn - gq);
                uint32_t r[64] = {};
                if (un.n > 0) {
                    tc5::ld32(tm + 16 * gq, *reinterpret_cast<uint32_t(*)[32]>(&r[0]));
                    if (cnt > 2) tc5::ld32(tm + 16 * gq + 32, *reinterpret_cast<uint32_t(*)[32]>(&r[32]));
                }
                int gr[4];   // the four groups (past the task's last one: unused)
#pragma unroll
                for (int i = 0; i < 4; i++) gr[i] = __shfl_sync(0xffffffffu, gl, (gq + i) & 31);
                tc5::ld_wait();
#pragma unroll
                for (int j = 0; j < 64; j++) {
                    asm volatile("" : "+r"(r[j]));   // no use of a loaded register moves above the wait
                    if (un.n == 0) r[j] = 0u;
                }
                if (gq + 4 >= gn && un.n > 0) {   // the last accumulator columns are in registers
                    tc5::fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        if constexpr (PAIR) ptx::mbar_arrive_cluster(ptx::map_to_cta(&acc_empty[ab], 0));
                        else ptx::mbar_arrive(&acc_empty[ab]);
                    }
                }
                float probe = 0.f;   // NaN (or an infinity) among this token's sums makes it NaN
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    if (i >= cnt) break;
                    uint32_t pk[8];
#pragma unroll
                    for (int e = 0; e < 4; e++) {
                        const float4 bb = *reinterpret_cast<const float4 *>(bs + 16 * (gq + i) + 4 * e);
                        float v[4];
#pragma unroll
                        for (int j = 0; j < 4; j++) {
                            v[j] = __uint_as_float(r[16 * i + 4 * e + j]);
                            probe = fmaf(0.f, v[j], probe);
                        }
                        pk[2 * e] = pack_bf16(v[0] + bb.x, v[1] + bb.y);
                        pk[2 * e + 1] = pack_bf16(v[2] + bb.z, v[3] + bb.w);
                    }
                    if (nt < b.N) {
                        uint16_t *y = yrow + gr[i] * kDnGroup;
                        if (a.y32) {
                            ptx::st_global_32(y, pk);
                        } else {
                            reinterpret_cast<uint4 *>(y)[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                            reinterpret_cast<uint4 *>(y)[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                        }
                    }
                }
                if (probe != 0.f && nt < b.N) bad |= 1u << (gq >> 2);   // true for NaN only
            }
            // (the accumulators are free: the next units' MMAs run on)
            if (__any_sync(0xffffffffu, bad != 0))
                compute_again(a, b.X, b.K, nw, g0, gn, gl, un.list, un.n, bad, &beat,
                              PAIR ? ptx::map_to_cta(&beat, rank ^ 1) : 0u);
            if (un.n > 0) {
                ab ^= 1;
                if (ab == 0) fphase ^= 1;
            }
        }
    }
    // every MMA completed (the issuer waited for `done`), and of a pair neither
    // CTA reads or signals the other's shared memory any more
    auto meet = [&]() {
        __syncwarp();
        if constexpr (PAIR) ptx::cluster_barrier();
        else __syncthreads();
    };
    tc5::fence_before();
    meet();
    if (aborted(&stop)) {
        // (the same for both CTAs.) The loads that only some of the producers
        // issued are completed by the others, so that every barrier phase can
        // finish, and the CTA whose barriers count the bytes waits for the last
        // ns of them (older ones were consumed): no copy outlives the CTAs
        if (warp < 2) {
            int most = 0;
            for (int p = 0; p < 2; p++)
                for (int r = 0; r < (PAIR ? 2 : 1); r++) most = max(most, loads[p][r]);
            while (more && issued < most) more = load_chunk();
            for (int i = max(0, issued - ns); rank == 0 && i < issued; i++)
                if (!((stalled >> (i % ns)) & 1))
                    ptx::mbar_wait_bounded(&full[i % ns], (uint32_t)(i / ns) & 1, kDrainNs);
        }
        meet();
    }
    if (warp == kMmaWarp) {
        // a commit arrives by itself, at both CTAs of a pair: each CTA waits for
        // the last arrival at every barrier of its own before it gives up its
        // tensor memory and its shared memory (a barrier a lane)
        uint64_t *bar = nullptr;
        int last = 0;   // the phase of the last arrival
        if (lane < ns && lane < freed) {
            bar = &empty[lane];
            last = (freed - 1 - lane) / ns;
        } else if (lane >= 29 && lane - 29 < min(2, handed)) {
            bar = &acc_full[lane - 29];
            last = (handed - 1 - (lane - 29)) / 2;
        } else if (lane == 31) {
            bar = &done;
        }
        if (bar) ptx::mbar_wait_bounded(bar, (uint32_t)last & 1, kDrainNs);
        __syncwarp();
        tc5::fence_after();
        if constexpr (PAIR) tc5::dealloc_pair(tmem, 2 * kAccCols);
        else tc5::dealloc(tmem, 2 * kAccCols);
    }
}

__global__ void k_fill_absent(uint4 *__restrict__ out, int64_t n) {
    constexpr uint32_t two = (uint32_t)kAbsent << 16 | kAbsent;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        out[k] = make_uint4(two, two, two, two);
}

// Kept blocks into the dense rows: element (r, c) of stored block p of block
// row i goes to packed row 16 pos(group) + row % 16 (a kept -0 as 0, which
// gives the same sums).
__global__ void k_pack_dense(const uint16_t *__restrict__ data, const int32_t *__restrict__ indptr,
                             const int32_t *__restrict__ indices, const int32_t *__restrict__ group_pos, int64_t MB,
                             int R, int C, int64_t K, uint16_t *__restrict__ out) {
    for (int64_t i = blockIdx.x; i < MB; i += gridDim.x) {
        const int64_t p0 = indptr[i], total = (int64_t)(indptr[i + 1] - p0) * R * C;
        for (int64_t e = threadIdx.x; e < total; e += blockDim.x) {
            const int64_t b = e / (R * C);
            const int rc = (int)(e - b * R * C), r = rc / C, c = rc - r * C;
            const int64_t row = i * R + r;
            const uint16_t v = data[(p0 + b) * R * C + rc];
            out[((int64_t)group_pos[row / kDnGroup] * kDnGroup + row % kDnGroup) * K +
                (int64_t)indices[p0 + b] * C + c] = v == kAbsent ? 0 : v;
        }
    }
}

// A row-major bf16 matrix in boxes of `rows` x 64 columns, 128-byte swizzle.
cudaError_t encode(const void *p, int64_t n_rows, int64_t n_cols, int rows, CUtensorMap *map) {
    auto enc = tensor_map_encoder();
    if (!enc) return cudaErrorNotSupported;
    const cuuint64_t dims[2] = {(cuuint64_t)n_cols, (cuuint64_t)n_rows};
    const cuuint64_t strides[1] = {(cuuint64_t)n_cols * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)rows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(p), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
               ? cudaSuccess
               : cudaErrorInvalidValue;
}

template <int MAXB, bool PAIR>
cudaError_t launch(const LaunchArgs *las, const int *gs, int n) {
    DnBatch<MAXB> b;
    b.n = 0;
    b.X = static_cast<const uint16_t *>(las[0].X);
    b.N = las[0].N;
    b.K = las[0].sc->K;
    constexpr int kUnitTokens = PAIR ? 2 * TN : TN, kWRows = PAIR ? kDnGroup / 2 : kDnGroup;   // per row group and CTA
    int64_t units = 0;
    int gmax = 1;
    for (int i = 0; i < n; i++) {
        const LaunchArgs &la = las[i];
        const Schedule &sc = *la.sc;
        const DensePlan &pl = sc.dense;
        if (la.N == 0) continue;
        DnArgs &a = b.args[b.n];
        const int g = gs[i];
        a.table = pl.d_table + pl.table_at[g];
        a.group_row = pl.d_group_row;
        a.w = reinterpret_cast<const uint16_t *>(static_cast<const unsigned char *>(la.data) + pl.w_off);
        a.bias = la.bias;
        a.Y = static_cast<uint16_t *>(la.Y);
        a.status = la.status;
        a.M = sc.M;
        a.wait_ns = la.wait_ns;
        a.g = g;
        a.n_groups = pl.n_groups;
        a.n_full = pl.n_full;
        a.n_tasks = pl.n_tasks[g];
        a.n_work = (pl.n_full + g - 1) / g;
        a.tiles = (unsigned)((la.N + kUnitTokens - 1) / kUnitTokens);
        // unequal tasks: the longest first over all token tiles, so that every
        // SM gets its share of them (after the tasks without chunks, whose
        // stores run beside the first MMAs); equal ones: the tasks of a token
        // tile side by side, so that their reads of X meet in L2
        a.task_major = pl.max_chunks[g] * (int64_t)pl.n_tasks[g] > pl.chunks[g] + pl.chunks[g] / 4;
        a.stall_chunk = la.stall_chunk;
        a.y32 = reinterpret_cast<uintptr_t>(la.Y) % 32 == 0;   // (M is a multiple of 16)
        cudaError_t e = encode(a.w, std::max<int64_t>(1, (int64_t)pl.n_full * kDnGroup), sc.K, g * kWRows, &a.wmap);
        if (e != cudaSuccess) return e;
        b.start[b.n] = (unsigned)units;
        units += (int64_t)a.tiles * a.n_tasks;
        gmax = std::max(gmax, g);
        b.n++;
        if (units > INT32_MAX) return cudaErrorInvalidConfiguration;
    }
    if (units == 0) return cudaSuccess;
    b.start[b.n] = (unsigned)units;
    b.stage_bytes = kXBytes + (uint32_t)gmax * kWRows * 128;
    const uint32_t fixed = kBiasBytes + 1024;
    b.ns = (int)std::min<uint32_t>(kDnStagesMax, (kDnMaxSmem - 1024 - fixed) / b.stage_bytes);
    CUtensorMap xmap;
    static std::atomic<uint64_t> attr_set{0};
    cudaError_t e = allow_smem(k_dense<MAXB, PAIR>, kDnMaxSmem - 1024, attr_set);
    if (e == cudaSuccess) e = encode(las[0].X, las[0].N, las[0].sc->K, TN, &xmap);
    if (e != cudaSuccess) return e;
    const int64_t most = PAIR ? las[0].sc->sm_count / 2 : las[0].sc->sm_count;
    const unsigned grid = (unsigned)std::min<int64_t>(units, most) * (PAIR ? 2 : 1);
    return launch_clusters(k_dense<MAXB, PAIR>, PAIR ? 2 : 1, dim3(grid), dim3(kThreads), b.ns * b.stage_bytes + fixed,
                           las[0].stream, xmap, b);
}

}  // namespace

cudaError_t pack_dense_data(const Schedule &sc, const void *data, void *packed, cudaStream_t s) {
    const DensePlan &pl = sc.dense;
    unsigned char *out = static_cast<unsigned char *>(packed) + pl.w_off;
    if (pl.w_bytes == 0) return cudaSuccess;
    const int64_t eights = pl.w_bytes / 16;   // (K is a multiple of 8)
    k_fill_absent<<<(int)std::min<int64_t>((eights + 255) / 256, 1 << 16), 256, 0, s>>>(reinterpret_cast<uint4 *>(out), eights);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || sc.nnzb == 0) return e;
    const int grid = (int)std::min<int64_t>(sc.MB, 1 << 16);
    k_pack_dense<<<grid, 256, 0, s>>>(static_cast<const uint16_t *>(data), sc.d_indptr, sc.d_indices, pl.d_group_pos,
                                      sc.MB, sc.R, sc.C, sc.K, reinterpret_cast<uint16_t *>(out));
    return cudaGetLastError();
}

cudaError_t launch_dense(const LaunchArgs *las, const int *gs, int n) {
    if (n <= 0) return cudaSuccess;
    if (n > kDnBatchMax) return cudaErrorInvalidValue;
    int g[kDnBatchMax];
    for (int i = 0; i < n; i++) g[i] = gs[i] & ~kDnPair;
    if (gs[0] & kDnPair) return n == 1 ? launch<1, true>(las, g, 1) : launch<kDnBatchMax, true>(las, g, n);
    return n == 1 ? launch<1, false>(las, g, 1) : launch<kDnBatchMax, false>(las, g, n);
}

}  // namespace bsr
