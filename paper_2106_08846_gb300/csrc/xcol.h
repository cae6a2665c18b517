// The column-list SIMT kernel (spmm_xcol.cu) for fp32 blocks of 16 or 32 rows:
// parameters shared with the schedule.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <cstdint>
#include <vector>

#include "bsr.h"

namespace bsr {

constexpr int kXcWarps = 11;           // consumer warps, an item each (+ 1 producer warp: three a scheduler, 168 registers a thread)
constexpr int kXcChunk = 64;           // K columns per ring stage (two 128-byte swizzled boxes)
constexpr uint32_t kXcBox = 16384;     // bytes of a stage's box: 32 columns of up to 128 tokens
constexpr int kXcMaxSmem = 232448;     // 227 KB
constexpr uint32_t kXcRoom = kXcMaxSmem - 2048;   // of it for the ring
constexpr int kXcStagesMax = 8;
constexpr int kXcBatchMax = 64;        // products in one fused launch
constexpr int kXcTileSizes = 3;
constexpr int kXcTT[kXcTileSizes] = {8, 12, 14};   // tokens per lane (blocks of 32 rows); 8 times as many per unit
constexpr int kXcTT16 = 16;            // of 16 rows

// A task is up to kXcWarps items (block rows, or pieces of them), one per warp; a
// launch chooses how many, and its tile: neither changes an output's bits.
// Columns are packed chunk by chunk (64 columns of K) and in a chunk item by item,
// so that a task's part of a chunk is one bulk copy:
//   int32 n, 0, 0, 0   columns in this chunk
//   int32 [n]          byte offsets of theirs in the X tile, padded to 4
//   float [n][R]       their weights
struct XcPlan {
    bool ok = false;
    int64_t off = -1, bytes = 0;       // place in the handle's packed buffer
    uint32_t item_bytes = 0;           // largest packed chunk of an item
    int seg = 1;                       // most chunks per segment (one chain of additions)
    bool even = false;                 // items of about equal length
    std::vector<int32_t> table;        // per chunk and item: its start / 16 (and the end)
    std::vector<int32_t> ints;         // (place / 4 bytes, value) of the packed buffer's integers
    std::vector<int32_t> src;          // per column: its weights' place / 4 bytes, its block
    int32_t *d_table = nullptr, *d_ints = nullptr, *d_src = nullptr;
    mutable std::atomic<uint64_t> last{0};   // choose_xcol's last answer: N << 16 | (yes: 1)
};

// The first item of task t of `tasks`: equal counts, in item order.
#ifdef __CUDACC__
__host__ __device__
#endif
inline int xcol_first(int t, int tasks, int items) { return (int)((int64_t)t * items / tasks); }

// A ring stage: the X tile's two boxes, then the items' packed chunks.
inline uint32_t xcol_stage_bytes(uint32_t item_bytes, int G) { return (2 * kXcBox + G * item_bytes + 1023) & ~1023u; }

struct Schedule;
struct LaunchArgs;

// Fills sc.xc (after the items); returns the packed buffer's new end.
int64_t plan_xcol(Schedule &sc, int64_t base);
// Whether the kernel runs a call of N tokens.
bool choose_xcol(const Schedule &sc, int64_t N);
// Chunks per segment in a call of N tokens (0: two segments a chunk).
int xcol_segment(const Schedule &sc, int64_t N);
// Tile (index into kXcTT; 32 rows) and items per task of one grid of n products.
struct XcShape {
    int tile, G;
    double cycles;   // the model's, of the busiest SM
};
XcShape xcol_shape(const Schedule *const *scs, int n, int64_t N);
cudaError_t pack_xcol_data(const Schedule &sc, const void *data, void *packed, cudaStream_t s);
// n products that share X, N, K, R and the stream: one grid.
cudaError_t launch_xcol(const LaunchArgs *las, int n);

}  // namespace bsr
