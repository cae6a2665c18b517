// Plan and dispatch of the dense-tile kernel (dense.h): row groups, the
// chunks each task size's tasks touch, and the task size of a call.
#include <algorithm>
#include <cstdlib>

#include "bsr_internal.h"
#include "schedule.h"

namespace bsr {

namespace {

int dense_mode() {
    static const int mode = [] {
        const char *v = getenv("BSR_DENSE");
        return v && *v ? atoi(v) : -1;   // 0: never, 1: always, unset: by the model
    }();
    return mode;
}

int forced_groups() {
    static const int forced = [] {
        const char *v = getenv("BSR_DENSE_G");
        const int f = v ? atoi(v) : 0, g = f & ~kDnPair;
        return g >= 1 && g <= kDnMaxGroups && !((f & kDnPair) && g % 2) ? f : 0;
    }();
    return forced;
}

int model_takes(const Schedule &sc, int64_t N);

}  // namespace

// Nothing is kept (or packed) of a plan that no call would use.
int64_t plan_dense(Schedule &sc, int64_t base) {
    DensePlan &pl = sc.dense;
    pl.ok = false;
    const bool shape_ok = kDnGroup % sc.R == 0 || sc.R % kDnGroup == 0;
    if ((sc.variant != V_TC && sc.variant != V_XSTAGE) || sc.dt != BSR_BF16 || sc.M == 0 || sc.M % kDnGroup || sc.K % 8 ||
        !shape_ok || dense_mode() == 0)
        return base;
    const int64_t n_groups = sc.M / kDnGroup, nch = (sc.K + kDnChunk - 1) / kDnChunk;
    if (n_groups > INT32_MAX / 32 || nch > 1 << 20) return base;
    // groups with blocks first, in row order (a task's outputs are then runs of Y)
    std::vector<int32_t> rows, empty;
    for (int64_t g = 0; g < n_groups; g++) {
        const int64_t i0 = g * kDnGroup / sc.R, i1 = (g * kDnGroup + kDnGroup - 1) / sc.R;
        (sc.indptr[(size_t)i1 + 1] > sc.indptr[(size_t)i0] ? rows : empty).push_back((int32_t)g);
    }
    const int64_t n_full = (int64_t)rows.size();
    pl.w_bytes = std::max<int64_t>(n_full, 1) * kDnGroup * sc.K * 2;
    if (pl.w_bytes > (int64_t)1 << 30 && pl.w_bytes > sc.nnzb * sc.R * sc.C * 128) return base;   // 64 times the blocks
    // per group with blocks, the chunks that hold one (a byte each)
    std::vector<uint8_t> used((size_t)(n_full * nch), 0);
    std::vector<int32_t> count((size_t)n_full, 0);
    for (int64_t k = 0; k < n_full; k++) {
        uint8_t *u = &used[(size_t)(k * nch)];
        const int64_t r0 = (int64_t)rows[(size_t)k] * kDnGroup;
        for (int64_t i = r0 / sc.R; i <= (r0 + kDnGroup - 1) / sc.R; i++)
            for (int32_t p = sc.indptr[(size_t)i]; p < sc.indptr[(size_t)i + 1]; p++) {
                const int64_t col = (int64_t)sc.indices[(size_t)p] * sc.C;
                for (int64_t c = col / kDnChunk; c <= (col + sc.C - 1) / kDnChunk; c++) u[c] = 1;
            }
        count[(size_t)k] = (int32_t)std::count(u, u + nch, 1);
    }
    // by their chunk counts where full-width tasks then visit a fifth fewer
    // chunks (long groups share tasks and short ones leave chunks out)
    std::vector<int32_t> order((size_t)n_full), sorted;
    for (int64_t k = 0; k < n_full; k++) order[(size_t)k] = (int32_t)k;
    sorted = order;
    std::stable_sort(sorted.begin(), sorted.end(),
                     [&](int32_t x, int32_t y) { return count[(size_t)x] > count[(size_t)y]; });
    std::vector<uint8_t> any((size_t)nch);
    // the chunks of the task of groups [k0, k1) in an order
    auto unite = [&](const std::vector<int32_t> &o, int64_t k0, int64_t k1) {
        std::fill(any.begin(), any.end(), 0);
        for (int64_t k = k0; k < std::min(n_full, k1); k++) {
            const uint8_t *u = &used[(size_t)(o[(size_t)k] * nch)];
            for (int64_t c = 0; c < nch; c++) any[(size_t)c] |= u[c];
        }
        return std::count(any.begin(), any.end(), 1);
    };
    int64_t in_rows = 0, in_count = 0;
    for (int64_t k = 0; k < n_full; k += kDnMaxGroups) {
        in_rows += unite(order, k, k + kDnMaxGroups);
        in_count += unite(sorted, k, k + kDnMaxGroups);
    }
    if (in_count < in_rows - in_rows / 5) order.swap(sorted);
    pl.n_groups = (int)n_groups;
    pl.n_full = (int)n_full;
    for (int g = 1; g <= kDnMaxGroups; g++) {
        const int64_t tasks = (n_groups + g - 1) / g;
        const size_t at = pl.table.size();
        pl.table_at[g] = (int32_t)at;
        pl.n_tasks[g] = (int)tasks;
        pl.chunks[g] = 0;
        pl.max_chunks[g] = 0;
        pl.table.resize(at + (size_t)tasks + 1);
        for (int64_t t = 0; t < tasks; t++) {
            pl.table[at + (size_t)t] = (int32_t)(pl.table.size() - at);
            if (t * g >= n_full) continue;
            const int32_t n = (int32_t)unite(order, t * g, t * g + g);
            for (int64_t c = 0; c < nch; c++)
                if (any[(size_t)c]) pl.table.push_back((int32_t)c);
            pl.chunks[g] += n;
            pl.max_chunks[g] = std::max(pl.max_chunks[g], n);
        }
        pl.table[at + (size_t)tasks] = (int32_t)(pl.table.size() - at);
        if (pl.table.size() > (size_t)INT32_MAX / 4) break;
    }
    bool used_by_some = dense_mode() == 1 || forced_groups() > 0;   // token count
    for (int64_t N = 16; !used_by_some && N <= (int64_t)1 << 21; N += std::max<int64_t>(64, N / 640 * 64))
        used_by_some = model_takes(sc, N) > 0;
    if (pl.table.size() > (size_t)INT32_MAX / 4 || !used_by_some) {
        std::vector<int32_t>().swap(pl.table);
        return base;
    }
    pl.group_row.reserve((size_t)n_groups);
    for (int32_t k : order) pl.group_row.push_back(rows[(size_t)k]);
    pl.group_row.insert(pl.group_row.end(), empty.begin(), empty.end());
    pl.group_pos.resize((size_t)n_groups);
    for (int64_t k = 0; k < n_groups; k++) pl.group_pos[(size_t)pl.group_row[(size_t)k]] = (int32_t)k;
    pl.w_off = (base + 1023) & ~int64_t(1023);
    pl.ok = true;
    return pl.w_off + pl.w_bytes;
}

namespace {

// The busiest SM's cycles at each task size, and the least of them against the
// block-by-block kernel's. A chunk costs about 250 + 34 g cycles (one CTA) or
// 300 + 24 g (a pair: half the weight tile per CTA), and no less than 400 to 430
// (a producer's wait and issue), the start of a pair about
// 950 more, 64 columns of epilogue about 500: fitted to 1024 x 1024 weights at
// 16384 tokens (g = 8 33.9 and 32.9 us, g = 16 29.8 and 26.6 us) and 768 x 768
// ones at 1024 and 3000 tokens (g = 3 to 8). The block-by-block kernel pays
// about 300 cycles per unit of its own model (250 to 410 where measured):
// against it the dense tiles won on every 50 to 95% sparse weight tried and on
// 16x16 blocks of 1024 x 1024 at 99% (21 against 33 us at 16384 tokens). On 16x16
// blocks of 4096 x 4096 at 97%, where every chunk has a block of some row and the
// dense tiles do 33 times the kept multiply-adds, the two are close (us, dense and
// block by block: 1000 tokens 21 and 26, 2048 46 and 62, 4096 94 and 94), and
// the model keeps calls from 2048 tokens on block by block. Narrow blocks too sparse for the block-by-
// block kernel have the per-task SIMT kernel beside this one, at about 0.85
// cycles per unit of its model: 32x1 of 1024 x 1024 at 95%, 16384 tokens, 26.2
// against 68 us.
int model_takes(const Schedule &sc, int64_t N) {
    const DensePlan &pl = sc.dense;
    int best = 1;
    double best_cost = -1.0;
    for (int pair = 0; pair <= (N > kDnTokens && sc.sm_count >= 2 ? 1 : 0); pair++) {
        const int64_t tiles = (N + kDnTokens * (1 + pair) - 1) / (kDnTokens * (1 + pair));
        const int64_t sms = pair ? sc.sm_count / 2 : sc.sm_count;
        for (int g = 1 + pair; g <= kDnMaxGroups; g += 1 + pair) {
            const double chunk = pair ? std::max(430.0, 300.0 + 24.0 * g) : std::max(400.0, 250.0 + 34.0 * g);
            const double epi = 500.0 * ((g + 3) / 4);
            const int64_t n_work = (pl.n_full + g - 1) / g, units = tiles * n_work;
            // the busiest SM takes every sms-th unit, the longest of each round;
            // task by task in the order of their chunks (about: the mean, past 64 rounds)
            const int64_t rounds = (units + sms - 1) / sms;
            double mma = 0.0;
            if (rounds <= 64) {
                const int32_t *off = &pl.table[(size_t)pl.table_at[g]];
                for (int64_t r = 0; r < rounds; r++) {
                    const int64_t t = r * sms / tiles;
                    mma += (double)(off[t + 1] - off[t]);
                }
            } else {
                mma = (double)(rounds * pl.chunks[g]) / (double)std::max<int64_t>(n_work, 1);
            }
            const double stores = (double)((tiles * pl.n_tasks[g] + sms - 1) / sms) * epi;
            const double cost = std::max(mma * chunk, stores) + epi + (pair ? 950.0 : 0.0);
            if (best_cost < 0 || cost < best_cost) {
                best_cost = cost;
                best = g | (pair ? kDnPair : 0);
            }
        }
    }
    double other = 0.0;   // the variant's own kernel
    if (sc.variant == V_TC) {
        choose_tc_tasks(sc, N, &other);
        other *= 300.0;
    } else {
        choose_tasks(sc, N, &other);
        other *= 0.85;
    }
    return dense_mode() != 1 && other > 0 && best_cost > other ? 0 : best;
}

}  // namespace

int choose_dense(const Schedule &sc, int64_t N) {
    const DensePlan &pl = sc.dense;
    if (!pl.ok || N <= 0) return 0;
    if (forced_groups()) return forced_groups();
    // (the choice for the last N asked, which is what a steady stream of calls asks again)
    const uint64_t memo = pl.last.load(std::memory_order_relaxed);
    if (N < (int64_t)1 << 48 && memo >> 16 == (uint64_t)N) return (int)(memo & 0xffff);
    const int best = model_takes(sc, N);
    if (N < (int64_t)1 << 48) pl.last.store((uint64_t)N << 16 | (uint64_t)best, std::memory_order_relaxed);
    return best;
}

}  // namespace bsr
