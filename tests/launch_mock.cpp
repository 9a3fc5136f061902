// The host harness of api_mock.cpp with the launchers that the library itself always has: the lone
// queries of a plan in one launch of units, and its query pairs in one launch where that is the
// rule.  The mocks compute the same fake scores and check what the kernels rely on: tickets and
// progress words zeroed, the units of a task complete and in order, the boundary columns of
// pipelined tasks apart and long enough, every stream of a piece of a unit within its slot, the
// profiles of a merged launch within its shared memory, a task's units in one range (the first unit
// of a range waits for nobody).  A launch of one tile gets query pairs only, as the kernel's.
#include "ctx.h"

#define launch_sw16 tile_launch
#define launch_gather_stream gather_stream
#define launch_long_cells long_cells
#define main api_mock_main
#include "api_mock.cpp"
#undef main
#undef launch_long_cells
#undef launch_gather_stream
#undef launch_sw16

namespace {

cm_ctx* g_ctx = nullptr;                           // for the size of its boundary buffer
int g_huge = 0;                                    // launches of the kernel of scores from 2^28

std::vector<std::string> g_runs;                   // per plan run (one stream each), its launches

template <class T>
void record(const char* what, const T* v, int32_t n)
{
    if (g_runs.empty()) g_runs.emplace_back();
    g_runs.back().append(what).append(reinterpret_cast<const char*>(v), (size_t)n * sizeof(T));
}

SwArgs one_task(const SwArgs& a, const SwTask* t, int32_t* ticket)
{
    SwArgs b = a;
    b.tasks = t;
    b.ntasks = 1;
    b.task_counter = ticket;
    *ticket = 0;
    return b;
}

// rows of the longest stream of subjects [s0, s1) split n ways
int64_t longest_split(const int64_t* srow, int32_t s0, int32_t s1, int n)
{
    int64_t longest = 0;
    for (int i = 0; i < n; ++i) {
        const int64_t rows = srow[s1] - srow[s0];
        const int32_t lo = nearest_boundary(srow, s0, s1, srow[s0] + rows * i / n);
        const int32_t hi = nearest_boundary(srow, s0, s1, srow[s0] + rows * (i + 1) / n);
        longest = std::max(longest, srow[hi] - srow[lo]);
    }
    return longest;
}

const char* unit_fault(const SwArgs& a, const SwUnit* units, int32_t t, int32_t first)
{
    const SwUnit& u = units[t];
    const SwBlock& B = a.blocks[u.block];
    const int64_t* srow = a.srows + B.srow;
    const TileChoice tc = choose_tile(len_of(a.ids[B.a_ids + u.k]), false);
    if (u.mode != tc.mode || u.R != tc.R || u.npass != tc.npass) return "unit of another tile";
    if (u.s1 <= u.s0) return "unit without subjects";
    const int ns = u.mode == kModeTwo16 ? 4 : 2;
    if (u.bnd_row < 0) {
        if (u.pass != 0 || u.pass_end != u.npass) return "unit of some passes without its column";
        for (int32_t s0 = u.s0, s1; u.npass > 1 && s0 < u.s1; s0 = s1) {
            s1 = piece_end(srow, s0, u.s1, a.bnd_stride);
            if (s1 <= s0 || s1 > u.s1) return "piece out of its unit";
            if (longest_split(srow, s0, s1, ns) > a.bnd_stride) return "stream longer than its slot";
        }
        return nullptr;
    }
    if (u.pass_end != u.pass + 1 || u.npass < 2) return "pipelined unit of several passes";
    if (longest_split(srow, u.s0, u.s1, ns) > u.rows) return "boundary column too short";
    if (u.pass > 0) {
        const SwUnit& v = units[t - 1];
        if (t == first || v.pass + 1 != u.pass || v.block != u.block || v.k != u.k || v.s0 != u.s0 ||
            v.s1 != u.s1 || v.bnd_row != u.bnd_row)
            return "pass that does not follow the one before it";
    }
    return nullptr;
}

}  // namespace

namespace cm {

cudaError_t launch_gather_stream(const uint8_t* db, const int64_t* off, const int32_t* ids, int32_t nb,
                                 const int64_t* srow, uint8_t* stream, cudaStream_t st)
{
    g_runs.emplace_back();
    return gather_stream(db, off, ids, nb, srow, stream, st);
}

cudaError_t launch_sw16(int R, int W, int mode, int grid, const SwArgs& a, cudaStream_t st)
{
    record("tile", a.tasks, a.ntasks);
    if (mode != kModePair && mode != kModeSeg16) return cudaErrorInvalidValue;
    return tile_launch(R, W, mode, grid, a, st);
}

// without units: the kernel of huge scores, with its slots behind the strips' boundary columns
cudaError_t launch_long_cells(int grid, const SwArgs& a, const CellJob* jobs, int32_t n, int32_t* counter,
                              int32_t* res, cudaStream_t st)
{
    if (!a.cell_units) {
        ++g_huge;
        const DevBuf& b = g_ctx->buf[B_BND];
        const int64_t end = (a.bnd - static_cast<uint2*>(b.p)) + (int64_t)grid * kLongSlots * a.bnd_stride;
        if (a.bnd < b.p || end * (int64_t)sizeof(uint2) > (int64_t)b.cap) contract_error(a, "slots outside the buffer");
        for (int32_t i = 0; i < n; ++i)
            if (jobs[i].m > a.bnd_stride) contract_error(a, "rows beyond a slot");
    }
    return long_cells(grid, a, jobs, n, counter, res, st);
}

cudaError_t launch_sw16_pairs(int W, int grid, int smem, const SwArgs& a, cudaStream_t st)
{
    record("pairs", a.tasks, a.ntasks);
    if (grid < 1 || W != 16) return cudaErrorInvalidValue;
    if (*a.task_counter != 0) { contract_error(a, "task ticket not zeroed"); return cudaSuccess; }
    for (int32_t i = 0; i < a.ntasks; ++i) {
        const SwTask& t = a.tasks[i];
        if (sw16_pair_smem(t.R, t.mode) > smem) { contract_error(a, "profile too large"); return cudaSuccess; }
        int32_t ticket;
        const cudaError_t e = tile_launch(t.R, W, t.mode, grid, one_task(a, &t, &ticket), st);
        if (e != cudaSuccess) return e;
    }
    *a.task_counter = a.ntasks;
    return cudaSuccess;
}

cudaError_t launch_sw16_single(int grid, int warps, const SwArgs& a, cudaStream_t st)
{
    if (grid < 1 || warps < 1 || warps > kSingleWarps) return cudaErrorInvalidValue;
    const int32_t n = a.ranges[a.nranges];
    record("single", a.units, n);
    if (a.nranges < 1 || a.nranges > grid || a.ranges[0] != 0) { contract_error(a, "ranges"); return cudaSuccess; }
    std::vector<int32_t> range_of((size_t)n, 0);
    std::vector<char> home((size_t)a.nranges, 0);
    for (int b = 0; b < grid; ++b) {
        if (a.homes[b] < 0 || a.homes[b] >= a.nranges) { contract_error(a, "home"); return cudaSuccess; }
        home[a.homes[b]] = 1;
    }
    for (int r = 0; r < a.nranges; ++r) {
        if (a.task_counter[r] != 0 || a.ranges[r + 1] <= a.ranges[r] || !home[r]) {
            contract_error(a, "ticket not zeroed, or a range empty or without a CTA");
            return cudaSuccess;
        }
        for (int32_t t = a.ranges[r]; t < a.ranges[r + 1]; ++t) range_of[t] = a.ranges[r];
    }
    int64_t columns = 0;                           // end of the boundary columns so far
    for (int32_t t = 0; t < n; ++t) {
        const SwUnit& u = a.units[t];
        const char* fault = a.progress[t] != 0 ? "progress not zeroed" : unit_fault(a, a.units, t, range_of[t]);
        if (!fault && u.bnd_row >= 0 && u.pass == 0) {
            if (u.bnd_row < columns) fault = "boundary columns overlap";
            columns = u.bnd_row + u.rows;
        }
        if (!fault && u.bnd_row >= 0 && u.pass + 1 < u.npass &&
            (t + 1 == n || a.units[t + 1].pass != u.pass + 1))
            fault = "task without its last pass";
        if (fault) { contract_error(a, fault); return cudaSuccess; }
        if (u.pass > 0) continue;                  // a task's scores, once
        SwTask k{u.block, u.k, u.s0, u.s1, 1, 0, u.mode, u.R};
        k.npass = u.npass;
        int32_t ticket;
        SwArgs b = one_task(a, &k, &ticket);
        b.bnd_stride = INT64_MAX;                  // (its streams are checked above)
        const cudaError_t e = tile_launch(u.R, 4, u.mode, grid, b, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace cm

// "cells": the cells of every ordered pair of a set of the given lengths, with a matrix of 127: as
// the fake similarity gives them, and how many launches went to the kernel of huge scores.
// "autotune": the autotuner on such a set; every plan it makes runs twice, and both runs have to
// launch the same work in the same order.
int main(int argc, char** argv)
{
    if (argc < 3) return api_mock_main();
    if (cm_create(&g_ctx, 0)) return 1;
    g_sym = true;
    g_off.assign(1, 0);
    for (int i = 2; i < argc; ++i) g_off.push_back(g_off.back() + std::atoll(argv[i]));
    const int32_t n = argc - 2;
    std::vector<uint8_t> seqs((size_t)g_off.back(), 3);
    std::vector<int8_t> mat(400, 127);
    if (std::strcmp(argv[1], "cells") == 0) {
        std::vector<int32_t> p, got((size_t)n * n * 5);
        for (int32_t x = 0; x < n; ++x)
            for (int32_t y = 0; y < n; ++y) p.insert(p.end(), {x, y});
        const int r = sw_cells_batch(g_ctx, seqs.data(), g_off.data(), n, p.data(), (int64_t)n * n, mat.data(),
                                     11, 1, got.data(), 0);
        int differ = 0;
        for (int32_t q = 0; q < n * n; ++q) {
            int64_t c[5];
            fake_cells(p[2 * q], p[2 * q + 1], c);
            for (int k = 0; k < 5; ++k) differ += c[k] != got[5 * (size_t)q + k];
        }
        std::printf("error %d differ %d huge %d\n", r, differ, g_huge);
    } else {
        int32_t w = 0, rows = 0;
        const int r = cm_autotune(g_ctx, seqs.data(), g_off.data(), n, mat.data(), 11, 1, 0, nullptr, &w,
                                  &rows, 0);
        cm_stats st{};
        cm_get_stats(g_ctx, &st);
        int differ = 0;
        for (size_t i = 0; i + 1 < g_runs.size(); i += 2) differ += g_runs[i] != g_runs[i + 1];
        std::printf("error %d runs %zu differ %d cells %lld of %lld\n", r, g_runs.size(), differ,
                    (long long)g_cells_done, (long long)st.cells);
    }
    cm_destroy(g_ctx);
    return 0;
}
