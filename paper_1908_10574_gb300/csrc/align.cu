// sw_align_batch: one optimal local alignment per pair as run-length operations, for the
// similar pairs a clustering reports (Sec. 6.1: the pairs are re-aligned for inspection).
//
// The alignment cells (score, start and end cell, csrc/api.cu run_cells) fix the span of the
// alignment: a[i_s..i_e] against b[j_s..j_e].  Inside that rectangle the alignment is the
// global affine (Gotoh) alignment of the two substrings, which scores the local optimum:
//   H(0,0) = 0;  H(0,j) = E(0,j) = -(g1 + (j-1)e);  H(i,0) = F(i,0) = -(g1 + (i-1)e)
//   E(i,j) = max(H(i,j-1) - g1, E(i,j-1) - e)     b_j against a gap      (op D)
//   F(i,j) = max(H(i-1,j) - g1, F(i-1,j) - e)     a_i against a gap      (op I)
//   H(i,j) = max(H(i-1,j-1) + S(a_i, b_j), F(i,j), E(i,j))              (op M)
// One warp aligns one pair.  The fill is a wavefront: lane l holds 8 consecutive columns of a
// 256-column pass and at step t works on row group t - l (4 rows; row k trails row k - 1 by one
// column, so the rows are independent chains), its left neighbour's last column arriving by
// shuffle; a pass hands its last column to the next through scratch memory.  Which term won
// goes into four bits per cell (ties: the aligned pair, then F, then E; a gap's opening before
// its extension), a lane's 8 columns of a row into one word, stored in step order, so a step's
// 32 x 4 words leave as one contiguous 512 bytes: half a byte per cell.  The traceback is
// walked by the whole warp: 32 rows of two 8-column strips are fetched at once, and the walk
// reads them by shuffle until it leaves that window, about ten cells a fetch instead of one
// dependent load per cell.  The passes of a pair are units of a queue, longest pair first: each
// is taken by another warp and trails the one before it by 32 row groups (progress.cuh), so a
// long pair is a pipeline; the warp of the last pass walks back.  Pairs run in rounds whose
// scratch (direction words, boundary column, runs) fits a budget.
// Bound: issue and the ALU pipe (54 and 65 % busy on an active SM), with 12 warps of 167 registers;
// some 15 instructions update a cell, 45 are issued for it with the wavefront's fill, the padding of
// short spans, the profiles and the walks.  Measured on one GB300, 2,000 pairs of up to 1,500
// residues (4.6e8 cells): 295 ms with one thread per pair and a byte per cell, 4.9 ms with one
// warp per pair (the longest pairs crowd a few SMs), 1.5 ms with a warp per pass.
#include <algorithm>
#include <cstring>
#include <numeric>
#include <type_traits>
#include <vector>

#include "ctx.h"
#include "progress.cuh"

namespace cm {
namespace {

struct AlnMatrix {
    int16_t v[kAlpha * kAlpha];
};

struct AlnJob {
    int32_t a, b;        // sequence ids (a: first sequence of the pair)
    int32_t i0, j0;      // 0-based first residue of the span in a and b
    int32_t p, q;        // span lengths
    int32_t score;       // expected global score of the span (the local optimum)
    int32_t pad;
    int64_t dir;         // byte offset of the direction words in the scratch
    int64_t bnd;         // byte offset of the boundary column (H, E per row; several passes)
    int64_t ops;         // byte offset of the (p + q) int32 runs
};

constexpr int32_t kAlnNeg = -(1 << 29);
constexpr uint32_t kSrcF = 1, kSrcE = 2, kFOpen = 4, kEOpen = 8;
constexpr int kAlnCols = 8, kAlnRows = 4;             // per lane and step
constexpr int kAlnPass = 32 * kAlnCols;
constexpr int kAlnWarps = 12;                         // resident warps per SM

__host__ __device__ inline int32_t aln_steps(int32_t p) { return (p + kAlnRows - 1) / kAlnRows + 31; }
__host__ __device__ inline int32_t aln_passes(int32_t q) { return (q + kAlnPass - 1) / kAlnPass; }

// the four scores of a profile word, sign-extended
__device__ __forceinline__ int32_t byte_score(uint32_t w, int k)
{
    return (int32_t)(int8_t)(w >> (8 * k));
}

// directions of span columns [pass * 256, ...) into D; `progress` is this pass's word, the word
// before it the previous pass's.  False (on every lane) when a wait gave up or the score at
// (p, q) is wrong; err says which.
__device__ __forceinline__ bool align_fill(const AlnJob& J, const uint8_t* __restrict__ A, int pass,
                                           const uint2* prof, int32_t g1, int32_t ge,
                                           uint4* __restrict__ D, int2* bnd, int32_t* progress,
                                           int32_t* err)
{
    constexpr uint32_t kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int32_t groups = (J.p + kAlnRows - 1) / kAlnRows;
    const int32_t p = J.p, q = J.q, npass = aln_passes(q), nsteps = aln_steps(p);
    const int32_t c0 = pass * kAlnPass + lane * kAlnCols;     // columns before this lane's first
    auto edge = [&](int32_t n) { return n == 0 ? 0 : -(g1 + (n - 1) * ge); };
    int32_t hg[kAlnCols], f[kAlnCols];                        // H - g1 and F of the row above
#pragma unroll
    for (int c = 0; c < kAlnCols; ++c) { hg[c] = edge(c0 + c + 1) - g1; f[c] = kAlnNeg; }
    int32_t oh[kAlnRows], oe[kAlnRows];                       // last column of this lane's rows
#pragma unroll
    for (int k = 0; k < kAlnRows; ++k) { oh[k] = 0; oe[k] = kAlnNeg; }
    int32_t diag0 = edge(c0), good = 1;
    uint32_t cur = 0, prev = 0;
    int2 bv[kAlnRows] = {};
    for (int32_t t = 0; t < nsteps; ++t) {
        const int j = t & 31;
        if (j == 0) {                                         // the next 32 row groups
            if (pass > 0 && t < groups && !wait_groups(progress - 1, min(t + 32, groups), err)) {
                if (lane == 0) atomicExch(err, 2);
                return false;
            }
            prev = cur;
            cur = 0;
#pragma unroll
            for (int k = 0; k < kAlnRows; ++k) {
                const int32_t r = (t + lane) * kAlnRows + k;
                cur |= (uint32_t)(r < p ? A[r] : kPadCode) << (8 * k);
                if (pass > 0) bv[k] = r < p ? __ldcg(bnd + r) : make_int2(0, kAlnNeg);
            }
        }
        const uint32_t rv = __shfl_sync(kAll, (lane <= j) ? cur : prev, (j - lane) & 31);
        const int32_t row0 = (t - lane) * kAlnRows;
        int32_t h[kAlnRows], e[kAlnRows];                     // left neighbour column, then running
#pragma unroll
        for (int k = 0; k < kAlnRows; ++k) {
            h[k] = __shfl_up_sync(kAll, oh[k], 1);
            e[k] = __shfl_up_sync(kAll, oe[k], 1);
        }
        if (pass > 0) {
#pragma unroll
            for (int k = 0; k < kAlnRows; ++k) {
                const int32_t x = __shfl_sync(kAll, bv[k].x, j), y = __shfl_sync(kAll, bv[k].y, j);
                if (lane == 0) { h[k] = x; e[k] = y; }
            }
        } else if (lane == 0) {
#pragma unroll
            for (int k = 0; k < kAlnRows; ++k) { h[k] = edge(row0 + k + 1); e[k] = kAlnNeg; }
        }
        if (row0 >= 0 && row0 < p) {
            int32_t dg[kAlnRows];
            uint2 w[kAlnRows];
            uint32_t dir[kAlnRows];
            dg[0] = diag0;
#pragma unroll
            for (int k = 1; k < kAlnRows; ++k) dg[k] = h[k - 1];
            diag0 = h[kAlnRows - 1];
#pragma unroll
            for (int k = 0; k < kAlnRows; ++k) {
                w[k] = prof[((rv >> (8 * k)) & 31u) * 32 + lane];
                dir[k] = 0;
                h[k] -= g1;
            }
            auto cells = [&](auto last) {                     // last: the group with row p
#pragma unroll
                for (int s = 0; s < kAlnCols + kAlnRows - 1; ++s) {
#pragma unroll
                    for (int k = 0; k < kAlnRows; ++k) {
                        const int c = s - k;
                        if (c < 0 || c >= kAlnCols) continue;
                        bool eo, fo, fge, m;
                        e[k] = __vibmax_s32(h[k], e[k] - ge, &eo);
                        f[c] = __vibmax_s32(hg[c], f[c] - ge, &fo);
                        const int32_t d = dg[k] + byte_score(c < 4 ? w[k].x : w[k].y, c & 3);
                        dg[k] = hg[c] + g1;
                        const int32_t gap = __vibmax_s32(f[c], e[k], &fge);
                        h[k] = __vibmax_s32(d, gap, &m) - g1;
                        hg[c] = h[k];
                        const uint32_t bits = (m ? 0u : fge ? kSrcF : kSrcE) | (fo ? kFOpen : 0u) |
                                              (eo ? kEOpen : 0u);
                        dir[k] |= bits << (4 * c);
                        if (decltype(last)::value && c0 + c + 1 == q && row0 + k + 1 == p)
                            good = (h[k] + g1 == J.score);
                    }
                }
            };
            if (row0 + kAlnRows >= p) cells(std::true_type());
            else cells(std::false_type());
#pragma unroll
            for (int k = 0; k < kAlnRows; ++k) { oh[k] = h[k] + g1; oe[k] = e[k]; }
            D[((int64_t)pass * nsteps + t) * 32 + lane] = make_uint4(dir[0], dir[1], dir[2], dir[3]);
            if (lane == 31 && pass + 1 < npass) {
#pragma unroll
                for (int k = 0; k < kAlnRows; ++k)
                    if (row0 + k < p) __stcg(bnd + row0 + k, make_int2(oh[k], oe[k]));
                const int32_t done = groups_after_step(t, groups);
                if (done > 0) publish_groups(progress, done);
            }
        }
    }
    // all lanes' directions of this pass are written before its last group is published
    __threadfence();
    __syncwarp();
    if (lane == 31 && pass + 1 < npass) publish_groups(progress, groups);
    if (__all_sync(kAll, good != 0)) return true;
    if (lane == 0) atomicExch(err, 1);            // the span's global score is the optimum
    return false;
}

// The walk back from (p, q): runs in reverse order, then reversed; returns their number.
__device__ __forceinline__ int32_t align_trace(const AlnJob& J, const uint32_t* D, int32_t* out)
{
    constexpr uint32_t kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int32_t nsteps = aln_steps(J.p);
    int32_t i = J.p, j = J.q, state = 0, n = 0, cur = -1, run = 0;
    int32_t strip0 = -1, row0 = -1;                       // window: rows row0 - lane, strips s0, s0 - 1
    uint32_t w0 = 0, w1 = 0;
    auto word = [&](int32_t strip, int32_t r) -> uint32_t {
        if (strip < 0 || r < 0) return 0u;
        const int32_t l = strip & 31;
        return __ldcg(D + (((int64_t)(strip >> 5) * nsteps + r / kAlnRows + l) * 32 + l) * kAlnRows +
                      r % kAlnRows);
    };
    auto emit = [&](int32_t op, int32_t len) {
        if (op != cur) {
            if (run && lane == 0) out[n] = (run << 2) | cur;
            n += run ? 1 : 0;
            cur = op;
            run = 0;
        }
        run += len;
    };
    while (i > 0 && j > 0) {
        const int32_t strip = (j - 1) / kAlnCols, r = i - 1;
        if (strip > strip0 || strip < strip0 - 1 || r > row0 || r < row0 - 31) {
            strip0 = strip;
            row0 = r;
            w0 = word(strip, r - lane);
            w1 = word(strip - 1, r - lane);
        }
        const uint32_t w = __shfl_sync(kAll, strip == strip0 ? w0 : w1, row0 - r);
        const uint32_t d = (w >> (4 * ((j - 1) % kAlnCols))) & 15u;
        if (state == 0) {
            state = (int32_t)(d & 3u);                    // 1: F, 2: E
            if (state == 0) { emit(0, 1); --i; --j; }
        } else if (state == 1) {
            emit(1, 1);
            state = (d & kFOpen) ? 0 : 1;
            --i;
        } else {
            emit(2, 1);
            state = (d & kEOpen) ? 0 : 2;
            --j;
        }
    }
    if (j > 0) emit(2, j);
    if (i > 0) emit(1, i);
    if (run && lane == 0) out[n] = (run << 2) | cur;
    n += run ? 1 : 0;
    __syncwarp();
    for (int32_t k = lane; k < n / 2; k += 32) {
        const int32_t x = out[k];
        out[k] = out[n - 1 - k];
        out[n - 1 - k] = x;
    }
    __syncwarp();
    return n;
}

// one column pass of a job
struct AlnUnit {
    int32_t job, pass;
};

__global__ void __launch_bounds__(32 * kAlnWarps, 1)
align_kernel(const uint8_t* __restrict__ db, const int64_t* __restrict__ off,
             const AlnJob* __restrict__ jobs, const AlnUnit* __restrict__ units, int32_t nunits,
             const AlnMatrix mat_in, int32_t g1, int32_t ge, uint8_t* __restrict__ scratch,
             int32_t* __restrict__ nops, int32_t* progress, int32_t* counter, int32_t* err)
{
    __shared__ int8_t mat[kAlpha * kAlpha];
    extern __shared__ uint2 prof_all[];           // [warps][kProfRows][32]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint2* prof = prof_all + warp * kProfRows * 32;
    for (int i = threadIdx.x; i < kAlpha * kAlpha; i += blockDim.x) mat[i] = (int8_t)mat_in.v[i];
    __syncthreads();
    // the first, longest units go one to an SM: the warps of a CTA do not queue all at once
    __nanosleep(2000 * warp);
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(counter, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= nunits) break;
        const AlnUnit U = units[t];
        const AlnJob J = jobs[U.job];
        const uint8_t* A = db + off[J.a] + J.i0;
        const uint8_t* B = db + off[J.b] + J.j0;
        uint4* D = reinterpret_cast<uint4*>(scratch + J.dir);
        __syncwarp();
        int q[kAlnCols];
#pragma unroll
        for (int c = 0; c < kAlnCols; ++c) {
            const int32_t col = U.pass * kAlnPass + lane * kAlnCols + c;
            q[c] = col < J.q ? B[col] : 0;                    // columns past q feed nothing
        }
        for (int x = 0; x < kProfRows; ++x) {
            const int8_t* row = mat + (x < kAlpha ? x : 0) * kAlpha;       // pad rows likewise
            uint32_t w[2] = {0u, 0u};
#pragma unroll
            for (int c = 0; c < kAlnCols; ++c) w[c >> 2] |= (uint32_t)(uint8_t)row[q[c]] << (8 * (c & 3));
            prof[x * 32 + lane] = make_uint2(w[0], w[1]);
        }
        __syncwarp();
        const bool good = align_fill(J, A, U.pass, prof, g1, ge, D,
                                     reinterpret_cast<int2*>(scratch + J.bnd), progress + t, err);
        if (U.pass + 1 < aln_passes(J.q) || !good) continue;
        const int32_t n = align_trace(J, reinterpret_cast<const uint32_t*>(D),
                                      reinterpret_cast<int32_t*>(scratch + J.ops));
        if (lane == 0) nops[U.job] = n;
    }
}

constexpr int kAlnSmem = kProfRows * 32 * (int)sizeof(uint2);     // per warp

// the runs of every job of a round, one after another in job order (one warp per job)
__global__ void gather_runs_kernel(const uint8_t* __restrict__ scratch,
                                   const AlnJob* __restrict__ jobs, const int32_t* __restrict__ nops,
                                   const int64_t* __restrict__ first, int32_t njobs,
                                   int32_t* __restrict__ flat)
{
    const int lane = threadIdx.x & 31;
    const int32_t t = (int32_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (t >= njobs) return;
    const int32_t* src = reinterpret_cast<const int32_t*>(scratch + jobs[t].ops);
    for (int32_t k = lane; k < nops[t]; k += 32) flat[first[t] + k] = src[k];
}

inline int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

}  // namespace
}  // namespace cm

using namespace cm;

extern "C" int sw_align_batch(cm_ctx* c, const uint8_t* seqs, const int64_t* offsets,
                              int32_t n_seqs, const int32_t* pairs, int64_t n_pairs,
                              const int8_t* matrix, int32_t gap_open, int32_t gap_extend,
                              int32_t* cells_out, int64_t* ops_offsets, int32_t* ops_out,
                              int64_t ops_capacity, int64_t* n_ops, uint32_t flags)
{
    if (!c) return CM_ERR_ARG;
    CUDA_TRY(cudaSetDevice(c->device));
    if (n_pairs < 0 || !n_ops || ops_capacity < 0 ||
        (n_pairs > 0 && (!pairs || !cells_out || !ops_offsets)) || (ops_capacity > 0 && !ops_out))
        return fail(c, CM_ERR_ARG, "bad pairs, outputs or capacity");
    NvtxRange nv("sw_align_batch");
    Prepared P;
    int r = prepare(c, seqs, offsets, n_seqs, matrix, gap_open, gap_extend, flags, P);
    if (r) return r;
    const bool dev = (flags & CM_DEVICE_PTRS) != 0;
    const cudaMemcpyKind out_kind = dev ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost;
    *n_ops = 0;
    if (n_pairs == 0) {
        const int64_t zero = 0;
        CUDA_TRY(cudaMemcpyAsync(ops_offsets, &zero, 8, out_kind, c->stream));
        CUDA_TRY(cudaStreamSynchronize(c->stream));
        return CM_OK;
    }
    std::vector<int32_t> hp((size_t)n_pairs * 2);
    if (dev) CUDA_TRY(cudaMemcpy(hp.data(), pairs, hp.size() * 4, cudaMemcpyDeviceToHost));
    else std::memcpy(hp.data(), pairs, hp.size() * 4);
    for (int64_t k = 0; k < 2 * n_pairs; ++k)
        if (hp[k] < 0 || hp[k] >= n_seqs) return fail(c, CM_ERR_ARG, "pair index out of range");
    std::vector<int32_t> hc((size_t)n_pairs * 5);
    if ((r = run_cells(c, P, hp.data(), n_pairs, hc.data()))) return r;

    // jobs: pairs with a non-empty alignment, in rounds whose scratch slices fit the budget
    std::vector<AlnJob> jobs;
    std::vector<int64_t> job_pair;
    for (int64_t k = 0; k < n_pairs; ++k) {
        const int32_t* cl = &hc[5 * k];
        if (cl[0] == 0) continue;
        AlnJob J{};
        J.a = hp[2 * k];
        J.b = hp[2 * k + 1];
        J.i0 = cl[1] - 1;
        J.j0 = cl[3] - 1;
        J.p = cl[2] - cl[1] + 1;
        J.q = cl[4] - cl[3] + 1;
        J.score = cl[0];
        jobs.push_back(J);
        job_pair.push_back(k);
    }
    const int64_t budget = (int64_t)1 << 30;
    std::vector<int32_t> counts(jobs.size(), 0), flat;
    size_t j0 = 0;
    while (j0 < jobs.size()) {
        size_t j1 = j0;
        int64_t bytes = 0;
        while (j1 < jobs.size()) {
            AlnJob& J = jobs[j1];
            const int64_t np = aln_passes(J.q);
            const int64_t dir = np * aln_steps(J.p) * 32 * (int64_t)sizeof(uint4);
            const int64_t bnd = np > 1 ? round_up(8 * (int64_t)J.p, 16) : 0;
            const int64_t need = dir + bnd + round_up(4 * ((int64_t)J.p + J.q), 16);
            if (j1 > j0 && bytes + need > budget) break;
            J.dir = bytes;
            J.bnd = J.dir + dir;
            J.ops = J.bnd + bnd;
            bytes += need;
            ++j1;
        }
        const int32_t nj = (int32_t)(j1 - j0);
        std::vector<int32_t> order((size_t)nj);
        std::iota(order.begin(), order.end(), 0);
        std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) {
            const AlnJob &X = jobs[j0 + x], &Y = jobs[j0 + y];
            return (int64_t)X.p * X.q > (int64_t)Y.p * Y.q;
        });
        std::vector<AlnUnit> units;
        for (int32_t t : order)
            for (int32_t pass = 0; pass < aln_passes(jobs[j0 + t].q); ++pass) units.push_back({t, pass});
        if (units.size() >= (size_t)INT32_MAX) return fail(c, CM_ERR_ARG, "too many column passes");
        const int32_t nu = (int32_t)units.size();
        uint8_t* d_scr;
        AlnJob* d_jobs;
        int32_t* d_cnt;
        AlnUnit* d_units;
        int64_t* d_first;
        ENSURE(B_SCRATCH, (size_t)bytes, d_scr);
        ENSURE(B_JOBS, (size_t)nj, d_jobs);
        ENSURE(B_UNITS, (size_t)nu, d_units);
        ENSURE(B_FIRST, (size_t)nj, d_first);
        ENSURE(B_FLAGS, kFlagWords + (size_t)nj + (size_t)nu, d_cnt);
        int32_t* d_progress = d_cnt + 8 + nj;
        if ((r = copy_in(c, d_jobs, jobs.data() + j0, (size_t)nj * sizeof(AlnJob), false))) return r;
        if ((r = copy_in(c, d_units, units.data(), units.size() * sizeof(AlnUnit), false))) return r;
        CUDA_TRY(cudaMemsetAsync(d_cnt, 0, sizeof(int32_t) * (8 + (size_t)nj + (size_t)nu), c->stream));
        AlnMatrix M;
        std::memcpy(M.v, P.mat, sizeof(M.v));
        // a CTA per SM while there are units for all, then more warps in each
        const int grid = std::min(nu, c->num_sms);
        const int warps = std::min(kAlnWarps, (nu + grid - 1) / grid);
        CUDA_TRY(cudaFuncSetAttribute(align_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      kAlnWarps * kAlnSmem));
        align_kernel<<<(unsigned)grid, 32 * warps, warps * kAlnSmem, c->stream>>>(
            P.db, P.off, d_jobs, d_units, nu, M, P.g1, P.ge, d_scr, d_cnt + 8, d_progress, d_cnt + 2,
            d_cnt + 1);
        CUDA_TRY(cudaGetLastError());
        int32_t kerr = 0;
        CUDA_TRY(cudaMemcpyAsync(&kerr, d_cnt + 1, 4, cudaMemcpyDeviceToHost, c->stream));
        CUDA_TRY(cudaMemcpyAsync(counts.data() + j0, d_cnt + 8, (size_t)nj * 4,
                                 cudaMemcpyDeviceToHost, c->stream));
        CUDA_TRY(cudaStreamSynchronize(c->stream));
        if (kerr == 2) return fail(c, CM_ERR_TIMEOUT, "a column pass's wait gave up");
        if (kerr) return fail(c, CM_ERR_INTERNAL, "alignment span does not reach the local optimum");
        std::vector<int64_t> first((size_t)nj);
        int64_t total = 0;
        for (int32_t t = 0; t < nj; ++t) {
            first[t] = total;
            total += counts[j0 + t];
        }
        int32_t* d_flat;
        ENSURE(B_OUT, (size_t)total, d_flat);
        if ((r = copy_in(c, d_first, first.data(), first.size() * sizeof(int64_t), false))) return r;
        gather_runs_kernel<<<(unsigned)((nj + 7) / 8), 256, 0, c->stream>>>(d_scr, d_jobs, d_cnt + 8,
                                                                           d_first, nj, d_flat);
        CUDA_TRY(cudaGetLastError());
        c->stats.launches += 2;
        const size_t old = flat.size();
        flat.resize(old + (size_t)total);
        CUDA_TRY(cudaMemcpyAsync(flat.data() + old, d_flat, (size_t)total * 4, cudaMemcpyDeviceToHost,
                                 c->stream));
        CUDA_TRY(cudaStreamSynchronize(c->stream));
        j0 = j1;
    }
    // offsets per pair (pairs without an alignment have no runs)
    std::vector<int64_t> hoff((size_t)n_pairs + 1, 0);
    std::vector<int32_t> per_pair((size_t)n_pairs, 0);
    for (size_t t = 0; t < jobs.size(); ++t) per_pair[job_pair[t]] = counts[t];
    for (int64_t k = 0; k < n_pairs; ++k) hoff[k + 1] = hoff[k] + per_pair[k];
    *n_ops = hoff[n_pairs];
    if (hoff[n_pairs] > ops_capacity)
        return fail(c, CM_ERR_CAPACITY, "ops_capacity too small; *n_ops holds the needed size");
    CUDA_TRY(cudaMemcpyAsync(cells_out, hc.data(), hc.size() * 4, out_kind, c->stream));
    CUDA_TRY(cudaMemcpyAsync(ops_offsets, hoff.data(), hoff.size() * 8, out_kind, c->stream));
    if (!flat.empty())
        CUDA_TRY(cudaMemcpyAsync(ops_out, flat.data(), flat.size() * 4, out_kind, c->stream));
    CUDA_TRY(cudaStreamSynchronize(c->stream));
    return CM_OK;
}
