// The dense-tile tensor-core kernel (spmm_dense.cu): bf16 weights as dense
// rows with zeros for absent blocks, in tiles whose K chunks without blocks
// are skipped. Parameters shared with the schedule.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <cstdint>
#include <vector>

#include "bsr.h"

namespace bsr {

constexpr int kDnTokens = 128;       // tokens per unit = MMA M = tensor-memory lanes
constexpr int kDnChunk = 64;         // K columns per ring stage (one 128-byte swizzle row of bf16)
constexpr int kDnGroup = 16;         // output rows per row group
constexpr int kDnMaxGroups = 16;     // row groups per task (N = 256, half the accumulator columns)
constexpr int kDnStagesMax = 8;      // ring stages (fewer where a stage is large)
constexpr int kDnPair = 32;          // flag beside a task size: pairs of CTAs, 256 tokens a unit
constexpr int kDnBatchMax = 64;      // products in one fused launch
constexpr int kDnMaxSmem = 232448;   // 227 KB

// The weight's rows in groups of 16; the groups that hold a kept block come
// first and are the rows of the packed dense weight [16 n_full, K] (columns
// without a kept block are -0), groups without one follow (their outputs
// are the bias). A task of size g is g consecutive groups; its table entry
// lists the 64-column chunks in which any of its groups has a block.
struct DensePlan {
    bool ok = false;
    int64_t w_off = -1;                // byte offset of the packed weight in the handle's buffer
    int64_t w_bytes = 0;
    int n_groups = 0, n_full = 0;
    std::vector<int32_t> group_row;    // position -> row group (output rows 16 group ..)
    std::vector<int32_t> group_pos;    // row group -> position
    // per g = 1..16: n_tasks + 1 list offsets, then the chunk lists, all in `table`
    std::vector<int32_t> table;
    int32_t table_at[kDnMaxGroups + 1] = {};
    int n_tasks[kDnMaxGroups + 1] = {};
    int64_t chunks[kDnMaxGroups + 1] = {};       // chunks of all tasks
    int32_t max_chunks[kDnMaxGroups + 1] = {};   // chunks of the longest task
    mutable std::atomic<uint64_t> last{0};       // choose_dense's last answer: N << 16 | task size
    int32_t *d_group_row = nullptr, *d_group_pos = nullptr, *d_table = nullptr;
};

struct Schedule;
struct LaunchArgs;

// Fills sc.dense (after the variant's plan; `base`: the first free byte of the
// packed buffer); returns the buffer's new end.
int64_t plan_dense(Schedule &sc, int64_t base);
// Row groups per task for a call of N tokens, with kDnPair where pairs of
// CTAs run it (0: the kernel does not run it).
int choose_dense(const Schedule &sc, int64_t N);
cudaError_t pack_dense_data(const Schedule &sc, const void *data, void *packed, cudaStream_t s);
// n products that share X, N, K and the stream (all with kDnPair or none): one grid.
cudaError_t launch_dense(const LaunchArgs *las, const int *gs, int n);

}  // namespace bsr
