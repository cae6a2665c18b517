// Plan and dispatch of the column-list kernel (xcol.h): packed columns, and the
// tile size of a call.
#include <algorithm>
#include <cstdlib>

#include "bsr_internal.h"
#include "schedule.h"

namespace bsr {

int64_t plan_xcol(Schedule &sc, int64_t base) {
    XcPlan &pl = sc.xc;
    pl.ok = false;
    const int64_t n_items = (int64_t)sc.items.size();
    if (sc.dt != BSR_F32 || sc.C != 1 || sc.R != 32 || sc.K % 4 || n_items == 0 || sc.variant != V_XSTAGE ||
        sc.nnzb > INT32_MAX / 256)
        return base;
    const int64_t nch = (sc.K + kXcChunk - 1) / kXcChunk;
    pl.off = (base + 1023) & ~int64_t(1023);
    pl.table.clear();
    pl.ints.clear();
    pl.src.clear();
    pl.item_bytes = 0;
    int64_t at = 0;   // 4-byte places
    auto put = [&](int64_t place, int64_t v) {
        pl.ints.push_back((int32_t)place);
        pl.ints.push_back((int32_t)v);
    };
    for (const Item &it : sc.items) {
        int32_t p = it.p0;
        for (int64_t c = 0; c < nch; c++) {
            int32_t p1 = p;
            while (p1 < it.p1 && sc.indices[(size_t)p1] < (c + 1) * kXcChunk) p1++;
            const int64_t n = p1 - p, vals = at + 4 + ((n + 3) & ~int64_t(3));
            pl.table.push_back((int32_t)(at / 4));
            put(at, n);
            for (int64_t k = 0; k < n; k++, p++) {
                const int kk = (int)(sc.indices[(size_t)p] - c * kXcChunk), b = kk & 31;
                put(at + 4 + k, ((b >> 2) << 4 | (b & 3) << 2) + (kk >> 5) * (int64_t)kXcBox);
                pl.src.push_back((int32_t)(vals + 32 * k));
                pl.src.push_back(p);
            }
            const int64_t end = vals + 32 * n;
            pl.item_bytes = std::max(pl.item_bytes, (uint32_t)((end - at) * 4));
            at = end;
            if (at > (int64_t)INT32_MAX / 2) return base;
        }
    }
    pl.table.push_back((int32_t)(at / 4));
    pl.bytes = at * 4;
    // equal segments of about 52 columns: outputs are then no further from 64
    // bits than the per-task kernel's, which shares a row among warps (relative
    // error at 102 columns in one chain 1.8e-7, at 512 4.0e-7; the per-task
    // kernel's 1.3e-7)
    const double mean = (double)sc.nnzb / (double)n_items;
    const int64_t segs = std::min<int64_t>(nch, std::max<int64_t>(1, (int64_t)(mean / 52.0 + 0.999)));
    pl.seg = (int)((nch + segs - 1) / segs);
    if (2 * xcol_stage_bytes(pl.item_bytes) > kXcRoom) return base;   // a ring of two stages
    pl.ok = true;
    return pl.off + pl.bytes;
}

// The tile that minimises the busiest scheduler's cycles, where that beats the
// per-task kernel. A task's items sit one per warp, ceil(items / 4) to a
// scheduler; a column takes it about 11.5 TT + 25 cycles, a chunk 100, a unit's
// stores 60 TT; the per-task kernel pays about 0.85 cycles per unit of its own
// model. Fitted to (us, this kernel and the per-task one): 1024 x 1024 at 90%,
// 16384 tokens 98.1 and 123 (TT = 14), 4096 tokens 30.5 and 36.5 (TT = 12); at
// 50%, 16384 tokens 377 and 659; 768 x 768 at 70%, 3000 tokens 30.4 and 37.3
// (TT = 8); 1536 x 1536 at 95%, 4000 tokens 47 and 38.9 (few columns per unit:
// stays); 768 x 768 at 50%, 1024 tokens 43 and 30.5 (24 items leave most SMs
// idle: stays).
int choose_xcol(const Schedule &sc, int64_t N) {
    static const int mode = [] {
        const char *v = getenv("BSR_XC");
        return v && *v ? atoi(v) : -1;   // 0: never
    }();
    static const int forced = [] {
        const char *v = getenv("BSR_XC_TILE");   // index into kXcTT
        return v && *v ? atoi(v) : -1;
    }();
    const XcPlan &pl = sc.xc;
    if (!pl.ok || N <= 0 || mode == 0) return -1;
    if (forced >= 0 && forced < kXcTileSizes) return forced;
    // (the choice for the last N asked, which is what a steady stream of calls asks again)
    const uint64_t memo = pl.last.load(std::memory_order_relaxed);
    if (N < (int64_t)1 << 48 && memo >> 16 == (uint64_t)N) return (int)(memo & 0xffff) - 1;
    const int64_t items = (int64_t)sc.items.size(), tasks = (items + kXcWarps - 1) / kXcWarps;
    const double warps = (double)(((items + tasks - 1) / tasks + 3) / 4);
    const double columns = (double)sc.nnzb / (double)items, chunks = (double)((sc.K + kXcChunk - 1) / kXcChunk);
    double per_task = 0.0;
    choose_tasks(sc, N, &per_task);
    double best_cost = 0.85 * per_task;
    int best = -1;
    for (int ti = 0; ti < kXcTileSizes; ti++) {
        const int TT = kXcTT[ti];
        const int64_t units = ((N + 8 * TT - 1) / (8 * TT)) * tasks;
        const double rounds = (double)((units + sc.sm_count - 1) / sc.sm_count);
        const double cost = rounds * (warps * columns * (11.5 * TT + 25.0) + 100.0 * chunks + 60.0 * TT) + 4000.0;
        if (cost < best_cost) {
            best_cost = cost;
            best = ti;
        }
    }
    if (N < (int64_t)1 << 48) pl.last.store((uint64_t)N << 16 | (uint64_t)(best + 1), std::memory_order_relaxed);
    return best;
}

}  // namespace bsr
