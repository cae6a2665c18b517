// Plan and dispatch of the column-list kernel (xcol.h): packed columns, and the
// tile size of a call.
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "bsr_internal.h"
#include "schedule.h"

namespace bsr {

namespace {

int xcol_mode() {
    static const int mode = [] {
        const char *v = getenv("BSR_XC"), *t = getenv("BSR_XC_TILE");
        if (v && *v && atoi(v) == 0) return 0;
        return (v && *v && atoi(v) == 1) || (t && *t) ? 1 : -1;   // 0: never, 1: always
    }();
    return mode;
}

bool model_takes(const Schedule &sc, int64_t N);

// The blocks [p, p1) of an item that lie in chunk c, from its first not packed yet.
int32_t chunk_end(const Schedule &sc, const Item &it, int32_t p, int64_t c) {
    while (p < it.p1 && (int64_t)sc.indices[(size_t)p] * sc.C < (c + 1) * kXcChunk) p++;
    return p;
}

}  // namespace

// Nothing is kept (or packed) of a plan that no call would use.
int64_t plan_xcol(Schedule &sc, int64_t base) {
    XcPlan &pl = sc.xc;
    pl.ok = false;
    const int64_t n_items = (int64_t)sc.items.size();
    // (wider blocks: the per-task kernel loads four activations at a time; 16x16 of
    // 768 x 768 at 70%, 4000 tokens 53 us against 71 here, 32x8 at 80% 36 against 39)
    if (sc.dt != BSR_F32 || (sc.R != 16 && sc.R != 32) || sc.C > 4 || kXcChunk % sc.C || sc.K % 4 || n_items == 0 ||
        sc.variant != V_XSTAGE || sc.nnzb > INT32_MAX / 256 / sc.C || xcol_mode() == 0)
        return base;
    const int64_t nch = (sc.K + kXcChunk - 1) / kXcChunk;
    // sizes first
    double longest = 0.0, apart = 0.0;   // of the items' blocks; from their mean
    const double mean = (double)sc.nnzb / (double)n_items;
    for (const Item &it : sc.items) {
        longest = std::max(longest, (double)(it.p1 - it.p0));
        apart += std::abs((double)(it.p1 - it.p0) - mean);
    }
    pl.even = longest <= 1.5 * mean && apart <= 0.25 * (double)sc.nnzb;
    if (!pl.even && xcol_mode() != 1) return base;
    int64_t ints = 0, most_columns = 0;   // 4-byte places
    for (const Item &it : sc.items) {
        int32_t p = it.p0;
        for (int64_t c = 0; c < nch; c++) {
            const int32_t p1 = chunk_end(sc, it, p, c);
            const int64_t n = (int64_t)(p1 - p) * sc.C;
            ints += 4 + ((n + 3) & ~int64_t(3)) + sc.R * n;
            most_columns = std::max(most_columns, n);
            p = p1;
        }
        if (ints > INT32_MAX / 2) return base;
    }
    pl.item_bytes = (uint32_t)((4 + ((most_columns + 3) & ~int64_t(3)) + sc.R * most_columns) * 4);
    if (2 * xcol_stage_bytes(pl.item_bytes, kXcWarps) > kXcRoom) return base;   // a ring of two stages
    // equal segments of at most 40 columns, or one chunk (xcol_segment may take less)
    const double per_chunk = (double)sc.nnzb * sc.C / (double)(n_items * nch);
    const int64_t most = per_chunk * (double)nch <= 40.0 ? nch : std::max<int64_t>(1, (int64_t)(40.0 / per_chunk));
    const int64_t segs = (nch + most - 1) / most;
    pl.seg = (int)((nch + segs - 1) / segs);
    bool used = xcol_mode() == 1;   // by a call of some size
    for (int64_t N = 64; !used && N <= (int64_t)1 << 21; N += std::max<int64_t>(64, N / 640 * 64)) used = model_takes(sc, N);
    if (!used) return base;
    pl.off = (base + 1023) & ~int64_t(1023);
    int64_t at = 0;
    auto put = [&](int64_t place, int64_t v) {
        pl.ints.push_back((int32_t)place);
        pl.ints.push_back((int32_t)v);
    };
    std::vector<int32_t> next(sc.items.size());   // per item: its first block not packed yet
    for (size_t i = 0; i < sc.items.size(); i++) next[i] = sc.items[i].p0;
    for (int64_t c = 0; c < nch; c++) {
        for (size_t i = 0; i < sc.items.size(); i++) {
            int32_t &p = next[i];
            const int32_t p1 = chunk_end(sc, sc.items[i], p, c);
            const int64_t n = (int64_t)(p1 - p) * sc.C, vals = at + 4 + ((n + 3) & ~int64_t(3));
            pl.table.push_back((int32_t)(at / 4));
            put(at, n);
            for (int64_t k = 0; k < n; k++) {
                const int64_t block = p + k / sc.C, in = k % sc.C;
                const int kk = (int)(sc.indices[(size_t)block] * (int64_t)sc.C + in - c * kXcChunk), b = kk & 31;
                put(at + 4 + k, ((b >> 2) << 4 | (b & 3) << 2) + (kk >> 5) * (int64_t)kXcBox);
                pl.src.push_back((int32_t)(vals + sc.R * k));
                pl.src.push_back((int32_t)(block * sc.C + in));
            }
            p = p1;
            at = vals + sc.R * n;
        }
    }
    pl.table.push_back((int32_t)(at / 4));
    pl.bytes = at * 4;
    pl.ok = true;
    return pl.off + pl.bytes;
}

// A chain of s additions per segment and one of the m segments have a squared
// error of 0.0346e-14 (s + m) relative to the sum's (within 2% for 8 sizes): so
// few enough columns a segment that this is no more than the per-task kernel's,
// which adds the chains of the warps that share a row (and of the two lane groups
// of a 16-row block): relative errors of 40 sizes and block shapes 0.77 to 0.99
// times the per-task kernel's, where segments of 40 columns had made six of them
// up to 7% larger.
int xcol_segment(const Schedule &sc, int64_t N) {
    const int64_t nch = (sc.K + kXcChunk - 1) / kXcChunk;
    const int warps = kXsConsumerWarps / std::min(choose_tasks(sc, N), kXsConsumerWarps), lanes = sc.R == 16 ? 2 : 1;
    const double n = (double)sc.nnzb * sc.C / (double)std::max<size_t>(sc.items.size(), 1);
    const double limit = 0.97 * (n / (warps * lanes) + warps + lanes - 1);
    auto chains = [&](int seg) {
        const double m = seg ? (double)((nch + seg - 1) / seg) : 2.0 * (double)nch;
        return (seg ? n * seg / (double)nch : n / m) + m;
    };
    int best = sc.xc.seg;
    for (int seg = sc.xc.seg; seg >= 0 && chains(best) > limit; seg--)
        if (chains(seg) < chains(best)) best = seg;
    return best;
}

// The tile and the items per task that minimise the busiest SM's cycles. A task's
// items sit one per warp, ceil(items / 4) to a scheduler; a column takes it 11.9
// TT cycles (a lone warp 24 more, 75 with the largest tile, which spills), a chunk
// 470, the rest of a unit 385 TT, a running sum in tensor memory 135 TT (one is in
// the 385), a launch 6000: fitted to 80 times of six sizes,
// every tile and 3 to 11 items, to 6% of them in the mean. One product's units run in rounds; those
// of several, longest first and to and fro, fill the SMs to about half of the
// longest.
XcShape xcol_shape(const Schedule *const *scs, int n, int64_t N) {
    static const int forced_tile = [] {
        const char *v = getenv("BSR_XC_TILE");   // index into kXcTT
        return v && *v ? atoi(v) : -1;
    }();
    static const int forced_G = [] {
        const char *v = getenv("BSR_XC_G");   // items per task
        return v && *v ? atoi(v) : -1;
    }();
    constexpr int kG[] = {kXcWarps, 8, 6, 4, 3, 2, 1};
    XcShape best = {0, kXcWarps, -1.0};
    const double sms = (double)scs[0]->sm_count;
    const double chunks = (double)((scs[0]->K + kXcChunk - 1) / kXcChunk);
    uint32_t item_bytes = 0;
    double segments[kXcBatchMax];
    bool half = false;   // only the tile that keeps its running sums in registers ends segments within a chunk
    for (int i = 0; i < n; i++) {
        item_bytes = std::max(item_bytes, scs[i]->xc.item_bytes);
        const int seg = xcol_segment(*scs[i], N);
        segments[i] = seg ? std::ceil(chunks / seg) : 2.0 * chunks;
        half |= seg == 0;
    }
    for (int G : kG) {
        if (forced_G >= 1 && forced_G <= kXcWarps ? G != forced_G : 2 * xcol_stage_bytes(item_bytes, G) > kXcRoom) continue;
        for (int ti = 0; ti < kXcTileSizes; ti++) {
            const bool r16 = scs[0]->R == 16;   // one tile, whose lanes do as many multiply-adds as the first's
            if (r16 || (half && forced_tile < 0) ? ti > 0 : forced_tile >= 0 && forced_tile < kXcTileSizes && ti != forced_tile) continue;
            const int TT = kXcTT[ti];
            const int64_t tokens = 8 * (r16 ? kXcTT16 : TT), tiles = (N + tokens - 1) / tokens;
            double sum = 0.0, longest = 0.0;
            int64_t units = 0;
            for (int i = 0; i < n; i++) {
                const int64_t items = (int64_t)scs[i]->items.size(), tasks = (items + G - 1) / G;
                if (!items) continue;
                const double warps = (double)(((items + tasks - 1) / tasks + 3) / 4);
                const double mean = (double)scs[i]->nnzb * scs[i]->C / (double)items;
                const double column = 11.9 * TT * warps + (warps > 1 ? 0.0 : TT == 14 ? 75.0 : 24.0);
                const double unit = mean * column + 470.0 * chunks + 385.0 * TT +
                                    (TT > 8 ? 135.0 * TT * std::max(0.0, segments[i] - 2.0) : 0.0);
                units += tiles * tasks;
                sum += unit * (double)(tiles * tasks);
                longest = std::max(longest, unit);
            }
            const double cost = n == 1 ? longest * std::ceil((double)units / sms)
                                       : std::max(longest, sum / sms + (units > sms ? 0.5 * longest : 0.0));
            // (fewer items a task read X more often: for 3% at least)
            if (best.cycles < 0 || cost < (G == best.G ? 1.0 : 0.97) * best.cycles) best = {ti, G, cost};
        }
    }
    best.cycles += 6000.0;
    return best;
}

namespace {

// Against the per-task kernel, which takes its tasks' work and about 8500 + 4000 / G
// cycles for each (G items a task; partly filled waves overlap). Measured (us, this
// kernel and the per-task one): 1024 x 1024 at 90%, 16384 tokens 99 and 124, 4096
// tokens 29.9 and 36.6; at 50%, 16384 tokens 360 and 656; 2048 x 2048 at 70%, 2000
// tokens 125 and 203; 4096 x 4096 at 90%, 512 tokens 58 and 100; 768 x 768 at 70%,
// 3000 tokens 28.3 and 37.4; at 50%, 1024 tokens 33.8 and 31.1 alone (segments of
// half a chunk, which the model leaves out), but 499 and 617 for a plan of 48
// weights of which ten are such. At 80%, 2000 tokens
// 22.8 and 19.2; at 70%, 1024 tokens 21 and 13.3; 1024 x 768 at 50%, 500 tokens 30
// and 15.6 (an item's columns are one warp's): these stay. Blocks of 16 rows: 16x1 of
// 1024 x 1024 at 90%, 16384 tokens 115 and 134; of 768 x 768 at 70%, 3000 tokens 32
// and 41; 16x4 of 1024 x 1024 at 80%, 3000 tokens 43 and 60; 32x2 at 90%, 8000 tokens
// 59 and 72.
bool model_takes(const Schedule &sc, int64_t N) {
    // rows of unequal length stay, because an item is one warp's here (pruned at
    // random, the longest row is below 1.5 means from about 40 columns on, and rows
    // are 0.15 means apart or less; 16x1 Zipf rows of 1024 x 1024 at 80%, 3000 tokens
    // 141 us, per-task 73)
    if (!sc.xc.even) return false;
    const Schedule *one = &sc;
    double cost = 0.0;
    const int G = choose_tasks(sc, N, &cost);
    const int64_t items = (int64_t)sc.items.size(), tasks = (items + G - 1) / G;
    const double waves = (double)((N + kXsTokens - 1) / kXsTokens * tasks) / (double)sc.sm_count;
    const double work = (double)sc.nnzb * sc.R * sc.C / (double)tasks;
    return xcol_shape(&one, 1, N).cycles < std::max(1.0, waves) * (8500.0 + 4000.0 / G + work);
}

}  // namespace

bool choose_xcol(const Schedule &sc, int64_t N) {
    const XcPlan &pl = sc.xc;
    if (!pl.ok || N <= 0) return false;
    if (xcol_mode() == 1) return true;
    // (the choice for the last N asked, which is what a steady stream of calls asks again)
    const uint64_t memo = pl.last.load(std::memory_order_relaxed);
    if (N < (int64_t)1 << 48 && memo >> 16 == (uint64_t)N) return memo & 1;
    const bool yes = model_takes(sc, N);
    if (N < (int64_t)1 << 48) pl.last.store((uint64_t)N << 16 | (uint64_t)yes, std::memory_order_relaxed);
    return yes;
}

}  // namespace bsr
