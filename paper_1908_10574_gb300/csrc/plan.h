// Host planner of the int16x2 Smith-Waterman launches: a pair block's queries, taken one or
// two at a time, get a register tile and launch mode (tile choice), their subjects are cut into
// CTA tasks of bounded work (add_tasks), and the tasks are grouped into one persistent launch
// per (tile, mode) bin, longest first (order_tasks).  Host code only; the host tests compile it
// on its own.
#pragma once

#include <algorithm>
#include <cstdint>
#include <utility>
#include <vector>

#include "cm_internal.h"

namespace cm {

struct Plan {
    std::vector<SwBlock> blocks;
    std::vector<int64_t> first_slot;     // per block, ascending
    std::vector<int32_t> ids;            // A ids then B ids
    std::vector<int64_t> srow;           // global row table over all B subjects (+1)
    std::vector<SwTask> tasks;           // grouped by R, cost descending inside a group
    std::vector<int> task_R;             // launch bin R * 4 + mode per task (parallel to tasks)
    std::vector<std::pair<int64_t, int>> keys;   // (cost, bin) per task (parallel to tasks)
    int64_t nslots = 0;
    int64_t cells = 0, cells_padded = 0, pairs = 0;
    int64_t max_warp_rows = 0;
    // Device-built subject lists: `ids` holds the A ids only; the B ids (n_sub of them) and the
    // row table (n_sub + 1 entries, total_rows rows) already sit in the B_IDS (after the A ids)
    // and B_SROW buffers; `srow` stays empty.
    bool dev_lists = false;
    int64_t n_sub = 0, total_rows = 0;
};

// Register tile and launch mode of a query (pair) whose longer query has m_hi residues.
struct TileChoice {
    int mode;      // SwMode
    int R;         // columns per lane per pass
    int npass;     // column passes
    int seg;       // lanes per query segment (32, or 16 in the segment modes)
    int spw;       // subject streams per warp
};

// A query without a partner runs in a single-query mode (two subject streams per 32-lane warp,
// or four over two 16-lane segments); a pair runs over 32 lanes or, when its longer query fits
// 16 lanes x 32 columns, in the 16-lane segment mode (R per lane twice that of a 32-lane tile,
// 16-column granularity).  32-lane pair tiles take passes of at most 1,024 columns (R 17..32
// above 512 residues); 32-lane single-query tiles passes of at most 512 (R 9..16), where the
// two-stream step still fits two rows into the register budget.
inline TileChoice choose_tile(int64_t m_hi, bool hi_valid)
{
    TileChoice t{};
    if (m_hi <= (hi_valid ? kSeg16MaxCols : kTwo16MaxCols)) {
        t.mode = hi_valid ? kModeSeg16 : kModeTwo16;
        t.seg = 16;
        t.R = (int)std::max<int64_t>(1, (m_hi + 15) / 16);
        t.npass = 1;
    } else if (hi_valid) {
        t.mode = kModePair;
        t.seg = 32;
        t.npass = (int)((m_hi + 1023) / 1024);
        const int64_t per = (m_hi + t.npass - 1) / t.npass;
        t.R = std::max(1, std::min(32, (int)((per + 31) / 32)));
    } else {
        t.mode = kModeTwo;
        t.seg = 32;
        t.npass = (int)((m_hi + kTwoPassCols - 1) / kTwoPassCols);
        const int64_t per = (m_hi + t.npass - 1) / t.npass;
        t.R = (int)((per + 31) / 32);
    }
    t.spw = t.mode == kModePair ? 1 : t.mode == kModeTwo16 ? 4 : 2;
    return t;
}

// Tasks of one query pair (k, k+1) or single query k against the block's subjects [0, ns), each
// holding about `target` rows per stream of its warps, divided by the query's column passes (a
// task streams its rows once per pass: sizing by rows x passes keeps the tasks of long queries
// as long as everyone else's).  With `srow` (the block's subject row table) the tasks split at
// subject boundaries by rows; without it (device-built lists) into equal subject counts,
// `rows_total` being the rows of all ns subjects.
inline void add_tasks(Plan& P, int32_t block, int32_t k, int32_t ns, bool hi_valid,
                      int64_t m_hi, const int64_t* srow, int64_t target, int64_t rows_total = 0)
{
    const TileChoice tc = choose_tile(m_hi, hi_valid);
    const int R = tc.R, np = tc.npass, mode = tc.mode, seg = tc.seg, spw = tc.spw;
    const bool single = mode == kModeTwo || mode == kModeTwo16;
    target = std::max<int64_t>(target * spw / np, 2048);
    const int64_t ntask = srow ? 0 : std::max<int64_t>(1, (rows_total + target - 1) / target);
    const int64_t per = srow ? 0 : (ns + ntask - 1) / ntask;
    int32_t s = 0;
    while (s < ns) {
        int32_t e;
        if (srow) {
            const int64_t want = srow[s] + target;
            e = (int32_t)(std::lower_bound(srow + s + 1, srow + ns + 1, want) - srow);
        } else {
            e = (int32_t)std::min<int64_t>(ns, s + per);
        }
        if (e > ns) e = ns;
        SwTask t{};
        t.block = block;
        t.k = k;
        t.s0 = s;
        t.s1 = e;
        t.npass = np;
        t.hi_valid = hi_valid ? 1 : 0;
        t.mode = mode;
        t.R = R;
        const int64_t rows = srow ? srow[e] - srow[s] : rows_total * (e - s) / std::max(ns, 1);
        P.cells_padded += rows * seg * R * np * (single ? 1 : 2);
        P.tasks.push_back(t);
        P.task_R.push_back(R * 4 + mode);         // launch bin: register tile and mode
        P.keys.push_back({rows * R * np / spw, R * 4 + mode});
        s = e;
    }
}

// 0 .. n - 1 by bucket_of(i) in [0, buckets), ties in order: a counting sort, for lists whose
// comparison sort would cost half as much as their kernel (50,000 pairs by their first sequence:
// 2.5 ms of a call of 9.0; 20,000 alignment jobs by cost: 0.35 ms of 7.7)
template <class Bucket>
inline std::vector<int64_t> counting_order(int64_t n, int64_t buckets, Bucket&& bucket_of)
{
    std::vector<int64_t> at((size_t)buckets + 1, 0), ord((size_t)n);
    for (int64_t i = 0; i < n; ++i) ++at[bucket_of(i) + 1];
    for (int64_t b = 0; b < buckets; ++b) at[b + 1] += at[b];
    for (int64_t i = 0; i < n; ++i) ord[at[bucket_of(i)]++] = i;
    return ord;
}

// bucket of a cost >= 0, larger costs first: 64 buckets a power of two, so a bucket's costs are
// within 1.6 % of each other
constexpr int64_t kCostBuckets = 64 * 64;
inline int64_t cost_bucket(int64_t cost)
{
    if (cost < 64) return kCostBuckets - 1 - cost;
    int top = 6;
    while (top < 62 && (cost >> (top + 1)) != 0) ++top;
    return kCostBuckets - 1 - ((int64_t)(top - 5) * 64 + ((cost >> (top - 6)) & 63));
}

// Groups the tasks by launch bin (descending), most work first inside a bin, ties in the
// order the tasks were made.  (The keys are sorted with their task index, not through it, so
// the sort stays cache-friendly for the millions of tasks of a large merge.)
inline void order_tasks(Plan& P)
{
    struct Key {
        int64_t cost;
        int bin;
        size_t i;
    };
    std::vector<Key> k(P.tasks.size());
    for (size_t i = 0; i < k.size(); ++i) k[i] = {P.keys[i].first, P.keys[i].second, i};
    std::sort(k.begin(), k.end(), [](const Key& x, const Key& y) {
        if (x.bin != y.bin) return x.bin > y.bin;
        if (x.cost != y.cost) return x.cost > y.cost;
        return x.i < y.i;
    });
    std::vector<SwTask> t2(k.size());
    std::vector<int> r2(k.size());
    for (size_t i = 0; i < k.size(); ++i) {
        t2[i] = P.tasks[k[i].i];
        r2[i] = P.task_R[k[i].i];
        P.keys[i] = {k[i].cost, k[i].bin};
    }
    P.tasks.swap(t2);
    P.task_R.swap(r2);
}

// Cuts the unit list of the single-query launch into ranges for `grid` CTAs, at equal shares of the
// cost (one per unit) and only between tasks: the passes of a pipelined task wait for the ones
// before them, which one ticket hands out before them.  ranges: the first unit of each, and the
// end; homes: the range that each CTA starts with.  With fewer tasks than CTAs every task is a
// range and the other CTAs join the ranges with the most cost per CTA.  24 pairs of 10,000
// residues (20 passes each): 5.9 ms per call, 6.0 with cuts inside tasks.
inline void cut_ranges(const std::vector<SwUnit>& units, const std::vector<double>& cost, int grid,
                       std::vector<int32_t>& ranges, std::vector<int32_t>& homes)
{
    const int64_t nu = (int64_t)units.size();
    auto starts_task = [&](int64_t t) { return units[t].bnd_row < 0 || units[t].pass == 0; };
    int64_t left = 0;                             // tasks that start after unit t
    double total = 0, sum = 0;
    for (int64_t t = 0; t < nu; ++t) {
        left += starts_task(t);
        total += cost[t];
    }
    const int64_t n = std::min<int64_t>(grid, left);
    std::vector<double> range_cost(1, 0.0);
    ranges.assign(1, 0);
    for (int64_t t = 0; t < nu; ++t) {
        sum += cost[t];
        range_cost.back() += cost[t];
        left -= starts_task(t);
        if (t + 1 == nu || !starts_task(t + 1)) continue;
        // range b ends at the first task that reaches its share, leaving one for the others
        const int64_t b = (int64_t)ranges.size();
        if (b < n && (sum * n >= total * b || left == n - b)) {
            ranges.push_back((int32_t)t + 1);
            range_cost.push_back(0.0);
        }
    }
    ranges.push_back((int32_t)nu);
    homes.resize((size_t)grid);
    std::vector<int> ctas((size_t)n, 1);
    for (int b = 0; b < grid; ++b) {
        homes[b] = b;
        if (b < n) continue;
        int64_t r = 0;
        for (int64_t q = 1; q < n; ++q)
            if (range_cost[q] * ctas[r] > range_cost[r] * ctas[q]) r = q;
        homes[b] = (int32_t)r;
        ++ctas[r];
    }
}

// Sizes the tasks of a plan.  First pass: count() every query pair (or lone query) with its
// subjects; second pass, after all are counted: add() makes their tasks.
//   * A pair of queries shares a CTA of W warps only if it has two subjects for each of the
//     CTA's streams (W, or 2 W over 16-lane segments); below that the streams, cut at subject
//     boundaries, are uneven or empty and the CTA waits for its longest one, so the two
//     queries run as lone queries, one warp each.
//   * Streams hold rows_per_warp rows in a large plan; in a small one as many as leave two
//     tasks for every CTA slot of the chip, but no fewer than kMinRows, since a stream also
//     pays for filling the wavefront (16 or 32 steps of four rows).
struct TaskSizer {
    static constexpr int64_t kMinRows = 512;
    int W;
    int64_t sms, rows_per_warp;
    double pair_cost = 0, single_cost = 0;           // rows x columns per lane x passes per stream

    TaskSizer(int W_, int64_t sms_, int64_t rows) : W(W_), sms(sms_), rows_per_warp(rows) {}

    bool paired(int32_t ns, bool hi_valid, int64_t m_hi) const
    {
        return hi_valid && ns >= 2 * W * (m_hi <= kSeg16MaxCols ? 2 : 1);
    }
    void count(int32_t ns, bool hi_valid, int64_t m_lo, int64_t m_hi, int64_t rows)
    {
        if (paired(ns, hi_valid, m_hi)) {
            pair_cost += cost(choose_tile(m_hi, true), rows);
        } else {
            if (hi_valid) single_cost += cost(choose_tile(m_lo, false), rows);
            single_cost += cost(choose_tile(m_hi, false), rows);
        }
    }
    // queries k and (hi_valid) k + 1 of m_lo and m_hi residues against subjects [0, ns_lo) and
    // [0, ns); srow / rows as add_tasks
    void add(Plan& P, int32_t block, int32_t k, int32_t ns_lo, int32_t ns, bool hi_valid,
             int64_t m_lo, int64_t m_hi, const int64_t* srow, int64_t rows = 0) const
    {
        if (paired(ns, hi_valid, m_hi)) {
            add_tasks(P, block, k, ns, true, m_hi, srow,
                      W * stream_target(pair_cost / (2.0 * sms * W), choose_tile(m_hi, true)), rows);
            return;
        }
        const double share = single_cost / (2.0 * sms * kSingleWarps);
        if (hi_valid && ns_lo > 0)
            add_tasks(P, block, k, ns_lo, false, m_lo, srow,
                      stream_target(share, choose_tile(m_lo, false)), rows);
        if (ns > 0)
            add_tasks(P, block, hi_valid ? k + 1 : k, ns, false, m_hi, srow,
                      stream_target(share, choose_tile(m_hi, false)), rows);
    }

private:
    static double cost(const TileChoice& t, int64_t rows)
    {
        return (double)rows * t.R * t.npass / t.spw;
    }
    // rows of a stream whose warp then has about `share` of cost (add_tasks multiplies by the
    // streams per warp and divides by the passes)
    int64_t stream_target(double share, const TileChoice& t) const
    {
        const double rows = share / t.R;
        return rows >= (double)rows_per_warp ? rows_per_warp
                                             : std::max(std::min(kMinRows, rows_per_warp), (int64_t)rows);
    }
};

}  // namespace cm
