// int16x2 Smith-Waterman of lone queries: one warp per task, one query per task, the query's
// two or four subject streams in the 16-bit halves (and 16-lane segments) of the warp.
//
// Serves pair lists (a block per distinct first sequence) and every block too small to feed the
// 16 warps of sw16_kernel.  The recurrences, the bias and the saturation mark are those of
// sw16_kernel.cuh; what differs is the shape of the work:
//   * A warp has its own query profile, so a query with a handful of subjects occupies one
//     warp instead of a CTA whose other warps idle, and one launch takes the tasks of every
//     register tile (the tile is a field of the task, the tile's code a function call): no
//     launch per tile, no tail per launch.
//   * The tasks come tile by tile, and a CTA (one per SM) starts on a contiguous range of them of
//     an equal share of the cost, so its warps run the same code: a tile's loop is 5-10 KB of
//     instructions, and twelve warps on as many tiles miss the instruction cache (50,000
//     pairs: 24 ms, 25 of 28 stall cycles per issue waiting for instructions).  Warps that
//     find their CTA's range empty take from the others'.
//   * The column passes of a long query (above 512 residues) are units of their own, taken by
//     different warps: pass p trails pass p - 1 by 32 row groups over the boundary column in
//     global memory, so a long query against long subjects is a pipeline, not one warp's
//     serial chain (24 pairs of 10,000 residues: 53 ms as chains).  A task's units lie in one
//     range, whose ticket hands them out in order: a unit's predecessor was taken before it, so
//     its warp is running and waits only on passes before its own.  So the waits end, after the
//     steps by which the passes trail one another.  Each is bounded all the same.
//   * The profile holds plain matrix scores as bytes (any int8 matrix fits; pads are -128),
//     four columns per word: 16 KB for 512 columns, so 12 warps fit an SM.  The packed score
//     of a column for the two streams' residues is one byte permute with sign extension of
//     their two words.  The diagonal input is H = (H - o) + o, one plain add off the ALU pipe.
//   * Four rows per step at every tile width.
// Bound: the ALU pipe, 5.5 of its half-rate operations per packed column (E, F, D, H, half a
// running maximum and the permute).  Measured on one GB300 against CTAs of 16 warps per query
// and a launch per tile: 50,000 pairs of 5,000 proteins (ten subjects per query) 26.6 -> 9.4 ms
// per call (6.4 with the pairs ordered by a counting sort), the kernel 20+ -> 4.2 ms (ALU pipe 63 %
// busy on an active SM, SMs active 77 % of the launch); one query against 200 proteins 0.84 -> 0.4 ms;
// 24 pairs of 8,000-12,000 residues 84.5 -> 5.9 ms (3.5 ms here, 2.2 the int32 rescoring).  The cell
// update of sw16_kernel.cuh with the floor in F (profile bytes of S + o, D a plain add) was 2 %
// slower here: twelve warps wait for latency before the ALU pipe is full.
#include "progress.cuh"
#include "sw16_kernel.cuh"

namespace cm {
namespace {

constexpr int kRows = kRowGroup;                  // rows per step
constexpr int8_t kBytePad = -128;                 // score of pad rows and pad columns

// words per lane in a profile row: four columns per word, odd so that the lanes' loads of one
// word index fall into distinct banks
__host__ __device__ constexpr int single_stride(int R) { return ((R + 3) / 4) | 1; }

constexpr int kSingleProfBytes = kProfRows * 32 * single_stride(16) * 4;
constexpr int kSingleSmem = kSingleProfBytes + kTwoPassCols;

// one warp's streams against the query columns of one pass (see sw16_single_kernel)
struct SingleArgs {
    const SwBlock* B;
    const uint32_t* st_lo;        // row groups of this lane's two streams
    const uint32_t* st_hi;
    int32_t g_lo, g_hi, g_max;    // their lengths, and the longest of the warp's streams
    int32_t s_lo, s_hi;           // subject index at the start of each
    int32_t k, ns;
    int32_t pass, npass;
    uint4* bnd;                   // boundary column: two records per row group
    const int32_t* done_in;       // row groups of it written by the pass before (null: all)
    int32_t* done_out;            // ... and by this one (null: nobody waits)
    int32_t* err;
};

// packed score of two streams: byte j of each word, sign-extended to 16 bits
template <int J>
__device__ __forceinline__ uint32_t score_pair(uint32_t lo, uint32_t hi)
{
    constexpr uint32_t sel = J | ((8 | J) << 4) | ((4 + J) << 8) | ((12 + J) << 12);
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(lo), "r"(hi), "n"(sel));
    return d;
}

__device__ __forceinline__ uint32_t score_pair(uint32_t lo, uint32_t hi, int j)
{
    return j == 0 ? score_pair<0>(lo, hi) : j == 1 ? score_pair<1>(lo, hi)
         : j == 2 ? score_pair<2>(lo, hi) : score_pair<3>(lo, hi);
}

template <int R, int SEG>
__device__ __noinline__ void single_dp(const SwArgs& a, const SingleArgs& t)
{
    constexpr int NR = kRows;
    constexpr int LS = single_stride(R), ROWW = SEG * LS;
    extern __shared__ __align__(16) uint8_t smem[];
    const int lane = threadIdx.x & (SEG - 1);
    const uint32_t* plane =
        reinterpret_cast<const uint32_t*>(smem + (threadIdx.x >> 5) * kSingleSmem) + lane * LS;
    const int o = a.gap_open, ge = a.gap_extend, beta = a.beta;
    const uint32_t BETA2 = (uint32_t)beta * 0x10001u;
    const uint32_t O2 = (uint32_t)o * 0x10001u;
    const uint32_t BMO2 = BETA2 - O2;
    const uint32_t NEGE = pack2(-ge, -ge);
    constexpr uint32_t PADW = kPadCode * 0x01010101u;
    constexpr uint32_t LASTBITS = kLast * 0x01010101u;
    const int32_t pass = t.pass, npass = t.npass, g_lo = t.g_lo, g_hi = t.g_hi, g_max = t.g_max;
    const uint32_t* st_lo = t.st_lo;
    const uint32_t* st_hi = t.st_hi;
    uint4* bnd = t.bnd;
    int32_t s_lo = t.s_lo, s_hi = t.s_hi;

    uint32_t hp[R], fp[R];
#pragma unroll
    for (int k = 0; k < R; ++k) { hp[k] = BMO2; fp[k] = BMO2; }
    uint32_t best = BETA2, out_acc = BETA2;
    uint32_t oh[NR], oe[NR];
#pragma unroll
    for (int q = 0; q < NR; ++q) { oh[q] = BMO2; oe[q] = BMO2; }
    uint32_t diag0 = BMO2;
    uint32_t cur = PADW, prev = PADW, cur2 = PADW, prev2 = PADW;
    uint4 bv0 = make_uint4(BMO2, BMO2, BMO2, BMO2), bv1 = bv0;

    for (int32_t step = 0; step < g_max + SEG - 1; ++step) {
        const int j = step & (SEG - 1);
        if (j == 0) {
            const int32_t u = step + lane;
            prev = cur;
            cur = (u < g_lo) ? st_lo[u] : PADW;
            prev2 = cur2;
            cur2 = (u < g_hi) ? st_hi[u] : PADW;
            if (SEG == 32 && pass > 0) {
                bv0 = bv1 = make_uint4(BMO2, BMO2, BMO2, BMO2);
                if (t.done_in != nullptr && step < g_max &&
                    !wait_groups(t.done_in, min(step + 32, g_max), t.err)) {
                    if (lane == 0) atomicExch(t.err, 2);
                    break;
                }
                if (u < g_max) { bv0 = __ldcg(bnd + 2 * u); bv1 = __ldcg(bnd + 2 * u + 1); }
            }
        }
        const int src = (j - lane) & (SEG - 1);
        const uint32_t rv = __shfl_sync(kFull, (lane <= j) ? cur : prev, src, SEG);
        const uint32_t rw = __shfl_sync(kFull, (lane <= j) ? cur2 : prev2, src, SEG);
        uint32_t h[NR], e[NR];                    // of the left neighbour column, then running
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            h[q] = __shfl_up_sync(kFull, oh[q], 1, SEG);
            e[q] = __shfl_up_sync(kFull, oe[q], 1, SEG);
        }
        uint32_t ai = __shfl_up_sync(kFull, out_acc, 1, SEG);
        if (SEG == 32 && pass > 0) {
            const uint32_t x0 = __shfl_sync(kFull, bv0.x, j), y0 = __shfl_sync(kFull, bv0.y, j);
            const uint32_t x1 = __shfl_sync(kFull, bv0.z, j), y1 = __shfl_sync(kFull, bv0.w, j);
            const uint32_t x2 = __shfl_sync(kFull, bv1.x, j), y2 = __shfl_sync(kFull, bv1.y, j);
            const uint32_t x3 = __shfl_sync(kFull, bv1.z, j), y3 = __shfl_sync(kFull, bv1.w, j);
            if (lane == 0) {
                h[0] = x0; e[0] = y0; h[1] = x1; e[1] = y1;
                h[2] = x2; e[2] = y2; h[3] = x3; e[3] = y3;
            }
        } else if (lane == 0) {
#pragma unroll
            for (int q = 0; q < NR; ++q) { h[q] = BMO2; e[q] = BMO2; }
        }
        if (lane == 0) ai = BETA2;
        uint32_t dg[NR];                          // H of the diagonal neighbour
        dg[0] = diag0 + O2;
#pragma unroll
        for (int q = 1; q < NR; ++q) dg[q] = h[q - 1] + O2;
        diag0 = h[NR - 1];
        if ((rv | rw) & kFirst) {                 // per half: whose stream starts a subject
            const uint32_t keep = ((rv & kFirst) ? 0u : 0x0000ffffu) | ((rw & kFirst) ? 0u : 0xffff0000u);
            const uint32_t fill = BMO2 & ~keep;
#pragma unroll
            for (int k = 0; k < R; ++k) {
                hp[k] = (hp[k] & keep) | fill;
                fp[k] = (fp[k] & keep) | fill;
            }
            best = (best & keep) | (BETA2 & ~keep);
            dg[0] = (dg[0] & keep) | (BETA2 & ~keep);
        }
        const uint32_t rc = rv & 0x1f1f1f1fu, rc2 = rw & 0x1f1f1f1fu;
        const uint32_t* prow[NR];
        const uint32_t* prow2[NR];
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            prow[q] = plane + __byte_perm(rc, 0u, 0x4440u | q) * ROWW;
            prow2[q] = plane + __byte_perm(rc2, 0u, 0x4440u | q) * ROWW;
        }
        uint32_t wl[NR], wh[NR];
        uint32_t pend = 0;
        bool has_pend = false;
        // row q trails row q - 1 by one column: NR independent dependency chains
#pragma unroll
        for (int k = 0; k < R + NR - 1; ++k) {
#pragma unroll
            for (int q = 0; q < NR; ++q) {
                const int c = k - q;
                if (c < 0 || c >= R) continue;
                if ((c & 3) == 0) { wl[q] = prow[q][c >> 2]; wh[q] = prow2[q][c >> 2]; }
                e[q] = __viaddmax_s16x2(e[q], NEGE, h[q]);
                const uint32_t f = __viaddmax_s16x2(fp[c], NEGE, hp[c]);
                const uint32_t d = __viaddmax_s16x2(dg[q], score_pair(wl[q], wh[q], c & 3), BETA2);
                dg[q] = hp[c] + O2;
                const uint32_t hh = __vimax3_s16x2(d, e[q], f);
                if (has_pend) { best = __vimax3_s16x2(best, pend, hh); has_pend = false; }
                else { pend = hh; has_pend = true; }
                h[q] = hh - O2;
                hp[c] = h[q];
                fp[c] = f;
            }
        }
        if (has_pend) best = __vmaxs2(best, pend);
#pragma unroll
        for (int q = 0; q < NR; ++q) { oh[q] = h[q]; oe[q] = e[q]; }
        out_acc = __vmaxs2(ai, best);
        if (lane == SEG - 1) {
            if (rv & LASTBITS) {
                const int32_t s = s_lo++;
                if (s < t.ns)
                    store_score(a, *t.B, t.k, s, (int32_t)(int16_t)(out_acc & 0xffffu), pass);
            }
            if (rw & LASTBITS) {
                const int32_t s = s_hi++;
                if (s < t.ns) store_score(a, *t.B, t.k, s, (int32_t)(int16_t)(out_acc >> 16), pass);
            }
            if (SEG == 32 && pass + 1 < npass && step >= 31) {
                __stcg(bnd + 2 * (step - 31), make_uint4(oh[0], oe[0], oh[1], oe[1]));
                __stcg(bnd + 2 * (step - 31) + 1, make_uint4(oh[2], oe[2], oh[3], oe[3]));
                // (scores of finished subjects are stored above, before the rows are published)
                if (t.done_out != nullptr && (j == 31 || step == g_max + 30))
                    publish_groups(t.done_out, step - 30);
            }
        }
    }
}

// the query columns [c0, c0 + seg * R) as a byte profile: 25 residues x seg lanes x LS words
__device__ __forceinline__ void build_profile(const uint8_t* q, int64_t m, int64_t c0, int R, int seg,
                                              const int8_t* mat, int qs, int xs, uint8_t* smem)
{
    const int lane = threadIdx.x & 31;
    uint8_t* qres = smem + kSingleProfBytes;
    for (int c = lane; c < seg * R; c += 32) qres[c] = (c0 + c < m) ? q[c0 + c] : kPadCode;
    __syncwarp();
    const int LS = single_stride(R), ln = lane & (seg - 1);
    for (int w = 0; w * 4 < R; ++w) {
        int off[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            off[j] = (w * 4 + j < R ? qres[ln * R + w * 4 + j] : kPadCode) * qs;
        // with 16-lane segments the two half warps take alternate rows
        for (int x = lane / seg; x < kProfRows; x += 32 / seg) {
            uint32_t v = 0;
#pragma unroll
            for (int j = 0; j < 4; ++j) v |= (uint32_t)(uint8_t)mat[off[j] + x * xs] << (8 * j);
            reinterpret_cast<uint32_t*>(smem)[(x * seg + ln) * LS + w] = v;
        }
    }
    __syncwarp();
}

// A warp runs units of its CTA's first range until it is empty, then of the ranges after it.
// kModeTwo: the task's rows split into two streams at subject boundaries, over 32 lanes, in
// passes of 32 R columns whose boundary column goes through the warp's slot of `bnd`;
// kModeTwo16: four streams, two per 16-lane segment.
__global__ void __launch_bounds__(32 * kSingleWarps, 1)
sw16_single_kernel(const __grid_constant__ SwArgs a)
{
    constexpr int MS = kAlpha + 1;                // matrix with a pad row and a pad column
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ int8_t s_mat[MS * MS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < MS * MS; i += blockDim.x) {
        const int x = i / MS, y = i - x * MS;
        s_mat[i] = (x < kAlpha && y < kAlpha) ? (int8_t)a.mat[x * kAlpha + y] : kBytePad;
    }
    __syncthreads();
    uint4* bnd = reinterpret_cast<uint4*>(
        a.bnd + ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * a.bnd_stride);
    const int home = a.homes[blockIdx.x];
    for (int visited = 0; visited < a.nranges;) {
        const int range = (home + visited) % a.nranges;
        int ti = 0;
        if (lane == 0) ti = a.ranges[range] + atomicAdd(a.task_counter + range, 1);
        ti = __shfl_sync(kFull, ti, 0);
        if (ti >= a.ranges[range + 1]) {
            ++visited;
            continue;
        }
        const SwUnit T = a.units[ti];
        const SwBlock* B = a.blocks + T.block;
        const int32_t q = a.ids[B->a_ids + T.k];
        const int64_t qoff = a.off[q], m = a.off[q + 1] - qoff;
        const int64_t* srow = a.srows + B->srow;
        const bool two16 = T.mode == kModeTwo16;
        const int ns = two16 ? 4 : 2;
        const int seg = two16 ? 16 : 32;
        const int i_lo = two16 ? 2 * (lane >> 4) : 0;
        const bool piped = T.bnd_row >= 0;
        SingleArgs t;
        t.B = B;
        t.k = T.k;
        t.ns = (B->kind == kTri) ? T.k : B->nb;
        t.npass = T.npass;
        t.bnd = piped ? reinterpret_cast<uint4*>(a.piped + T.bnd_row) : bnd;
        t.err = a.err;
        for (int32_t s0 = T.s0, s1; s0 < T.s1; s0 = s1) {
            s1 = piped || T.npass == 1 ? T.s1 : piece_end(srow, s0, T.s1, a.bnd_stride);
            // the streams' boundaries, and this lane's two streams
            const int64_t R0 = srow[s0], R1 = srow[s1];
            int32_t at[3];
#pragma unroll
            for (int i = 0; i < 3; ++i)
                at[i] = nearest_boundary(srow, s0, s1, R0 + (R1 - R0) * (i_lo + i) / ns);
            t.st_lo = reinterpret_cast<const uint32_t*>(a.streams + B->stream + srow[at[0]]);
            t.st_hi = reinterpret_cast<const uint32_t*>(a.streams + B->stream + srow[at[1]]);
            t.g_lo = (int32_t)((srow[at[1]] - srow[at[0]]) / kRows);
            t.g_hi = (int32_t)((srow[at[2]] - srow[at[1]]) / kRows);
            t.g_max = __reduce_max_sync(kFull, max(t.g_lo, t.g_hi));
            t.s_lo = at[0];
            t.s_hi = at[1];
            if (T.npass > 1 && (int64_t)t.g_max * kRows > (piped ? T.rows : a.bnd_stride)) {
                if (lane == 0) atomicExch(a.err, 1);  // boundary buffer too small: refuse
                break;
            }
            for (int pass = T.pass; pass < T.pass_end; ++pass) {
                t.pass = pass;
                t.done_in = piped && pass > 0 ? a.progress + ti - 1 : nullptr;
                t.done_out = piped && pass + 1 < T.npass ? a.progress + ti : nullptr;
                __syncwarp();
                build_profile(a.db + qoff, m, (int64_t)pass * seg * T.R, T.R, seg, s_mat,
                              B->swap ? 1 : MS, B->swap ? MS : 1, smem + warp * kSingleSmem);
                if (two16) {
                    switch (T.R) {
#define CM_MODE 3
#include "sw16_inst.cuh"
#define CM_CASE(r) case r: single_dp<r, 16>(a, t); break;
                        CM_R_CASES(CM_CASE)
#undef CM_CASE
#undef CM_MODE
                    }
                } else {
                    switch (T.R) {
#define CM_MODE 1
#include "sw16_inst.cuh"
#define CM_CASE(r) case r: single_dp<r, 32>(a, t); break;
                        CM_R_CASES(CM_CASE)
#undef CM_CASE
#undef CM_MODE
                    }
                }
            }
        }
    }
}

}  // namespace

cudaError_t launch_sw16_single(int grid, int warps, const SwArgs& a, cudaStream_t st)
{
    if (warps < 1 || warps > kSingleWarps) return cudaErrorInvalidValue;
    const cudaError_t e = cudaFuncSetAttribute(
        sw16_single_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSingleWarps * kSingleSmem);
    if (e != cudaSuccess) return e;
    sw16_single_kernel<<<grid, 32 * warps, warps * kSingleSmem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace cm
