// Batched Smith-Waterman (Gotoh affine gaps) on sm_103a: the similarity f of the paper's
// protein clustering (Sec. 4), scored for many pairs at once.
//
// Recurrences (a gap of k residues costs o + (k-1)e; H >= 0 makes the alignment local):
//   E(r,c) = max(E(r,c-1) - e, H(r,c-1) - o)
//   F(r,c) = max(F(r-1,c) - e, H(r-1,c) - o)
//   H(r,c) = max(0, H(r-1,c-1) + S(q_c, x_r), E(r,c), F(r,c)),   score = max H
//
// Mapping.  A warp owns 32*R query columns (lane l holds columns l*R .. l*R+R-1 in
// registers) and streams subject rows through an anti-diagonal wavefront: at step t lane l
// computes row t-l of its columns, receiving H and E of its left neighbour's last column for
// the same row by one warp shuffle.  Many subjects are concatenated in one row stream (first
// and last rows flagged), so the fill/drain of the wavefront is paid once per stream, not once
// per pair.  The two 16-bit halves of every register carry two different queries that share
// the subject stream, so each packed DPX instruction advances two cells.
//
// Packed-int16 formulation.  Every stored value carries a bias beta >= max(o + e, -min S) + 1
// (stored = true + beta), which keeps each half within [beta - o, 32767].  The DP keeps H - o,
// the value both gap types open from, and the profile carries S + o, so the diagonal term reads
// H - o as well.  Per packed column (two cells):
//   E = viaddmax(E, -e, (H - o)_left)           F = vimax3(F - e, (H - o)_up, beta)
//   D = (H - o)_diag + (S + o)                  H = vimax3(D, E, F), then H - o
//   and half a vimax3 for the running maximum (every two columns).
// The floor beta sits in F, whose add is a plain one, instead of in D: an F below it is worth no
// more than a local alignment's start, which H takes from F then.  So three of the adds (F - e, D,
// H - o) are plain 32-bit adds of both halves, which issue beside the ALU pipe, and 3.5 operations
// are left on it (4.5 with the floor in D = viaddmax(..., beta)).  None of the three carries or
// borrows between the halves: F >= beta > e and H >= beta > o, so the differences stay positive;
// H + S >= beta + min S >= 1 and <= 32767 + 127 < 65536, so D's low half neither borrows (a
// negative S + o is spread over the word, addend2) nor carries, also past the point where a half
// has left int16 and reads as negative: H takes F there.
// If a stored best reaches 32767 - max(S), some cell may have overflowed int16; that pair is
// marked and rescored on the int32 path, so every score returned is exact.
//
// Bound: the ALU pipe (75 % busy) and the pipe of the plain adds (69 %) together, with 79 % of the
// issue slots used: 1,200 sequences of 350 residues, 11.7 ms.  With D on the ALU pipe that pipe
// was 85 % busy, 63 % of the slots were used, and the set took 12.8 ms.  The constants are kernel
// parameters, which take no register and no read port: with them in registers this update was 4 %
// slower than D on the ALU pipe.  One sixteenth of the 20,000-protein triangle: 319 -> 307 ms per
// call.
#pragma once
#include <algorithm>

#include "cm_internal.h"

namespace cm {

namespace {

constexpr uint32_t kFull = 0xffffffffu;

// Tile geometry: SEG lanes (32, or 16 for a half-warp segment) of R columns each.
template <int R, int SEG = 32>
struct Geo {
    static constexpr int LS = lane_stride(R);       // 32-bit words per lane in a profile row
    static constexpr int ROWW = SEG * LS;           // words per profile row (multiple of 64 B)
    static constexpr int PROF_WORDS = kProfRows * ROWW;
    static constexpr int COLS = SEG * R;            // query columns per pass
};

__device__ __forceinline__ uint32_t pack2(int lo, int hi)
{
    return (uint32_t)(uint16_t)(int16_t)lo | ((uint32_t)(uint16_t)(int16_t)hi << 16);
}

// profile word of two halves for a plain 32-bit add: lo + 65536 hi, so that a negative low half
// borrows what its sum with a larger value carries
__device__ __forceinline__ uint32_t addend2(int lo, int hi)
{
    return (uint32_t)lo + ((uint32_t)hi << 16);
}

__device__ __forceinline__ int64_t tri(int64_t k) { return k * (k - 1) / 2; }

__device__ __forceinline__ int32_t lower_bound64(const int64_t* v, int32_t lo, int32_t hi,
                                                 int64_t key)
{
    // first index s in [lo, hi] with v[s] >= key (v strictly increasing)
    while (lo < hi) {
        const int32_t mid = (lo + hi) >> 1;
        if (v[mid] < key) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// subject boundary in [lo, hi] nearest to row `key` (ties to the later one): stream splits
// land within half a subject of their target, so the warps of a task finish closer together
__device__ __forceinline__ int32_t nearest_boundary(const int64_t* v, int32_t lo, int32_t hi,
                                                    int64_t key)
{
    const int32_t s = lower_bound64(v, lo, hi, key);
    return (s > lo && key - v[s - 1] < v[s] - key) ? s - 1 : s;
}

__device__ __forceinline__ int64_t slot_of(const SwBlock& B, int32_t k, int32_t s)
{
    const int64_t base = (B.kind == kTri) ? (tri(k) - tri(B.k0)) : (int64_t)(k - B.k0) * B.nb;
    return B.out_base + base + s;
}

__device__ __forceinline__ void store_score(const SwArgs& a, const SwBlock& B, int32_t k,
                                            int32_t s, int32_t stored, int pass)
{
    int64_t slot = slot_of(B, k, s);
    if (B.has_map) slot = a.out_map[slot];
    const int32_t val = (stored >= a.sat_thr) ? kSat : stored - a.beta;
    if (pass == 0) {
        a.out[slot] = val;
    } else {
        const int32_t old = __ldcg(a.out + slot);    // maybe written by another SM's pass
        if (old != kSat) a.out[slot] = (val == kSat) ? kSat : max(old, val);
    }
}

// load the profile words of columns [c, c + 4) of one row (fewer at the tile's right edge;
// the lane's row segment always holds whole 16-byte units)
template <int R>
__device__ __forceinline__ void load_cols(const uint32_t* p, int c, uint32_t (&v)[4])
{
    if (c + 3 <= R) {
        const uint4 x = *reinterpret_cast<const uint4*>(p + c);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
    } else if (c + 2 == R) {
        const uint2 x = *reinterpret_cast<const uint2*>(p + c);
        v[0] = x.x; v[1] = x.y;
    } else {
        v[0] = p[c];
    }
}

// One wavefront segment of SEG lanes (a whole warp, or a half-warp when SEG = 16) against the
// profile tile of this pass: the two 16-bit halves are two queries, and the subject stream of
// n_rows rows (every subject starts on a multiple of kRowGroup) feeds both.  A step covers a
// row group; row q of the step trails row q-1 by one column inside the lane, so the rows form
// independent dependency chains and the step's fixed costs (shuffles, residue and flag
// handling) are shared by them.  The segment's last lane writes one score per finished subject
// per half.  All lanes of the warp run `nrows_max` rows (the warp's longest stream); shorter
// streams step through pad rows meanwhile.  Multi-pass tiles (boundary columns in `bnd`) use
// SEG = 32 only.
template <int R, int SEG>
__device__ __forceinline__ void warp_dp16(const SwArgs& a, const SwBlock& B,
                                          const uint32_t* __restrict__ prof,
                                          const uint8_t* __restrict__ stream, int64_t n_rows,
                                          int64_t nrows_max, int pass, int npass,
                                          uint2* __restrict__ bnd, int32_t s0, int32_t k_lo,
                                          int32_t ns_lo, int32_t ns_hi, bool hi_valid)
{
    using G = Geo<R, SEG>;
    constexpr int NR = kRowGroup;
    const int lane = threadIdx.x & (SEG - 1);    // lane within the segment
    const uint32_t BETA2 = a.beta2, O2 = a.open2, E2 = a.ext2, NEGE = a.nege2;
    const uint32_t BMO2 = a.bmo2;                 // H - o of an empty prefix; E, F floor
    constexpr uint32_t PADW = kPadCode * 0x01010101u;
    // boundary records of one step: (H - o, E) of the last column of each of its rows, as
    // uint4 pairs of rows
    constexpr int NB = NR / 2;
    uint4* bnd4 = reinterpret_cast<uint4*>(bnd);
    constexpr uint32_t CODEMASK = 0x1f1f1f1fu;                        // residue code bits
    constexpr uint32_t LASTBITS = kLast * 0x01010101u;

    // hp[c] holds H - o of the row above (the value both E and F start a gap from, and the
    // diagonal of column c+1 against a profile that carries +o); fp[c] holds F.
    uint32_t hp[R], fp[R];
#pragma unroll
    for (int k = 0; k < R; ++k) { hp[k] = BMO2; fp[k] = BMO2; }
    uint32_t best = BETA2, out_acc = BETA2;
    uint32_t oh[NR], oe[NR];                      // last column of each row: H - o and E
#pragma unroll
    for (int q = 0; q < NR; ++q) { oh[q] = BMO2; oe[q] = BMO2; }
    uint32_t diag0 = BMO2;                        // left H - o of the previous step's last row
    uint32_t cur = PADW, prev = PADW;
    uint4 bv[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) bv[q] = make_uint4(BMO2, BMO2, BMO2, BMO2);
    int32_t s_next = s0;
    const uint32_t* plane = prof + lane * G::LS;
    const int nsup = (int)(n_rows / NR);          // a warp stream holds < 2^31 rows
    const int nsup_max = (int)(nrows_max / NR);
    const int nsteps = nsup_max + SEG - 1;
    const uint32_t* stw = reinterpret_cast<const uint32_t*>(stream);

    for (int t = 0; t < nsteps; ++t) {
        const int j = t & (SEG - 1);
        if (j == 0) {
            const int u = t + lane;
            prev = cur;
            cur = (u < nsup) ? stw[u] : PADW;
            if (SEG == 32 && pass > 0) {
#pragma unroll
                for (int q = 0; q < NB; ++q)
                    bv[q] = (u < nsup_max) ? bnd4[u * NB + q] : make_uint4(BMO2, BMO2, BMO2, BMO2);
            }
        }
        const int src = (j - lane) & (SEG - 1);
        const uint32_t rv = __shfl_sync(kFull, (lane <= j) ? cur : prev, src, SEG);
        uint32_t hL[NR], eL[NR];
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            hL[q] = __shfl_up_sync(kFull, oh[q], 1, SEG);
            eL[q] = __shfl_up_sync(kFull, oe[q], 1, SEG);
        }
        uint32_t ai = __shfl_up_sync(kFull, out_acc, 1, SEG);
        if (SEG == 32 && pass > 0) {
#pragma unroll
            for (int q = 0; q < NB; ++q) {
                const uint32_t x0 = __shfl_sync(kFull, bv[q].x, j), x1 = __shfl_sync(kFull, bv[q].y, j);
                if (lane == 0) { hL[2 * q] = x0; eL[2 * q] = x1; }
                const uint32_t x2 = __shfl_sync(kFull, bv[q].z, j), x3 = __shfl_sync(kFull, bv[q].w, j);
                if (lane == 0) { hL[2 * q + 1] = x2; eL[2 * q + 1] = x3; }
            }
        } else if (lane == 0) {
#pragma unroll
            for (int q = 0; q < NR; ++q) { hL[q] = BMO2; eL[q] = BMO2; }
        }
        if (lane == 0) ai = BETA2;
        uint32_t dg[NR], h[NR], e[NR];
        dg[0] = diag0;
#pragma unroll
        for (int q = 1; q < NR; ++q) dg[q] = hL[q - 1];
        diag0 = hL[NR - 1];
        if (rv & kFirst) {                        // a subject starts at the step's first row
#pragma unroll
            for (int k = 0; k < R; ++k) { hp[k] = BMO2; fp[k] = BMO2; }
            best = BETA2;
            dg[0] = BMO2;
        }
        // profile row of each residue: one mask takes the flags off all NR bytes, one byte
        // permute moves a code to the low byte (the stream writer keeps codes <= kPadCode)
        const uint32_t rc = rv & CODEMASK;
        const uint32_t* prow[NR];
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            prow[q] = plane + __byte_perm(rc, 0u, 0x4440u | q) * G::ROWW;
            h[q] = hL[q];
            e[q] = eL[q];
        }
        uint32_t sq[NR][4];
        uint32_t pend = 0;
        bool has_pend = false;
        // row q trails row q-1 by one column; the recurrences are at the top of the file
#pragma unroll
        for (int k = 0; k < R + NR - 1; ++k) {
#pragma unroll
            for (int q = 0; q < NR; ++q) {
                const int c = k - q;
                if (c < 0 || c >= R) continue;
                if ((c & 3) == 0) load_cols<R>(prow[q], c, sq[q]);   // next profile columns
                e[q] = __viaddmax_s16x2(e[q], NEGE, h[q]);
                const uint32_t f = __vimax3_s16x2(fp[c] - E2, hp[c], BETA2);
                const uint32_t d = dg[q] + sq[q][c & 3];
                dg[q] = hp[c];
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
            const int32_t lo = (int32_t)(int16_t)(out_acc & 0xffffu);
            const int32_t hi = (int32_t)(int16_t)(out_acc >> 16);
            if (rv & LASTBITS) {
                const int32_t s = s_next++;
                if (s < ns_lo) store_score(a, B, k_lo, s, lo, pass);
                if (hi_valid && s < ns_hi) store_score(a, B, k_lo + 1, s, hi, pass);
            }
        }
        if (SEG == 32 && lane == 31 && pass + 1 < npass && t >= 31) {
#pragma unroll
            for (int q = 0; q < NB; ++q)
                bnd4[(t - 31) * NB + q] = make_uint4(oh[2 * q], oe[2 * q], oh[2 * q + 1], oe[2 * q + 1]);
        }
    }
}

// Persistent int16x2 kernel of the query pairs (two 16-bit halves).  MODE kModePair: one
// subject stream per warp over 32 lanes.  kModeSeg16: two subject streams per warp, one per
// half-warp segment of 16 lanes, for short queries (16 lanes x R).  Lone queries: sw16_single.cu.
template <int R, int W, int MODE>
__global__ void __launch_bounds__(W * 32, 16 / W)
sw16_kernel(const __grid_constant__ SwArgs a)
{
    constexpr int SEG = MODE == kModeSeg16 ? 16 : 32;
    constexpr int SPW = MODE == kModeSeg16 ? 2 : 1;            // streams per warp
    using G = Geo<R, SEG>;
    extern __shared__ __align__(16) uint8_t smem[];
    uint32_t* prof = reinterpret_cast<uint32_t*>(smem);
    uint8_t* qres = smem + (size_t)G::PROF_WORDS * 4;          // [2][COLS]
    __shared__ int16_t s_mat[kAlpha * kAlpha];
    __shared__ int s_task[2];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int i = tid; i < kAlpha * kAlpha; i += W * 32) s_mat[i] = a.mat[i];
    if (tid == 0) s_task[0] = atomicAdd(a.task_counter, 1);
    __syncthreads();

    uint2* bnd = a.bnd + ((int64_t)blockIdx.x * W + warp) * a.bnd_stride;
    for (int it = 0;; ++it) {
        const int ti = s_task[it & 1];
        if (ti >= a.ntasks) break;
        if (tid == 0) s_task[(it + 1) & 1] = atomicAdd(a.task_counter, 1);

        const SwTask T = a.tasks[ti];
        const SwBlock B = a.blocks[T.block];
        const int32_t* A_ids = a.ids + B.a_ids;
        const int32_t q_lo = A_ids[T.k];
        const int32_t q_hi = T.hi_valid ? A_ids[T.k + 1] : q_lo;
        const int64_t qoff_lo = a.off[q_lo], m_lo = a.off[q_lo + 1] - qoff_lo;
        const int64_t qoff_hi = a.off[q_hi];
        const int64_t m_hi = T.hi_valid ? a.off[q_hi + 1] - qoff_hi : 0;
        const int32_t ns_lo = (B.kind == kTri) ? T.k : B.nb;
        const int32_t ns_hi = (B.kind == kTri) ? T.k + 1 : B.nb;
        const int64_t* srow = a.srows + B.srow;

        // rows of this task split over the CTA's streams at subject boundaries
        constexpr int NS = W * SPW;
        const int64_t R0 = srow[T.s0], R1 = srow[T.s1];
        int32_t sb[SPW + 1];
        int64_t nmax = 0;
#pragma unroll
        for (int i = 0; i <= SPW; ++i) {
            sb[i] = nearest_boundary(srow, T.s0, T.s1, R0 + (R1 - R0) * (warp * SPW + i) / NS);
            if (i > 0) nmax = max(nmax, srow[sb[i]] - srow[sb[i - 1]]);
        }
        const int seg = (SEG == 16) ? (lane >> 4) : 0;          // this lane's stream
        const int32_t st0 = sb[seg], st1 = sb[seg + 1];
        int64_t n_rows = srow[st1] - srow[st0];
        if (T.npass > 1 && (SEG == 16 || nmax > a.bnd_stride)) {
            if (lane == 0) atomicExch(a.err, 1);      // boundary buffer too small: refuse
            n_rows = nmax = 0;
        }
        const uint8_t* stream = a.streams + B.stream + srow[st0];

        for (int pass = 0; pass < T.npass; ++pass) {
            const int64_t c0 = (int64_t)pass * G::COLS;
            for (int c = tid; c < G::COLS; c += W * 32) {
                qres[c] = (c0 + c < m_lo) ? a.db[qoff_lo + c0 + c] : kPadCode;
                qres[G::COLS + c] = (c0 + c < m_hi) ? a.db[qoff_hi + c0 + c] : kPadCode;
            }
            __syncthreads();
            for (int i = tid; i < kProfRows * G::COLS; i += W * 32) {
                const int x = i / G::COLS, c = i - x * G::COLS;
                const int ln = c / R, k = c - ln * R;
                const int ql = qres[c], qh = qres[G::COLS + c];
                int sl = 0, sh = 0;           // pads score -o
                if (x != kPadCode) {          // +o: the DP keeps H - o as its diagonal input
                    if (ql != kPadCode) sl = (B.swap ? s_mat[x * kAlpha + ql] : s_mat[ql * kAlpha + x]) + a.gap_open;
                    if (qh != kPadCode) sh = (B.swap ? s_mat[x * kAlpha + qh] : s_mat[qh * kAlpha + x]) + a.gap_open;
                }
                prof[x * G::ROWW + ln * G::LS + k] = addend2(sl, sh);
            }
            __syncthreads();
            if (nmax > 0)
                warp_dp16<R, SEG>(a, B, prof, stream, n_rows, nmax, pass, T.npass, bnd, st0, T.k,
                                  ns_lo, ns_hi, T.hi_valid != 0);
            __syncthreads();
        }
    }
}

}  // namespace
}  // namespace cm
