// The ranker's width-9 convolutions as implicit GEMMs on the 5th-generation tensor cores
// (tcgen05.mma, BF16 operands, FP32 accumulator in tensor memory).  Rows are the residues of
// a batch's concatenated sequences (with zero gap rows between them), channels are contiguous.
//
// conv_tc_kernel<CIN, NOUT, EPI>: out[r, n] = sum_t sum_c X[r + t - 4, c] * Wk[n, t*CIN + c]
//   (forward: Wk[n, t*CIN + c] = W[t][c][n]; backward-data: X = dY, Wk[c, t*128 + n] =
//   W[8-t][c][n]).  A tile is 128 rows x NOUT channels: K runs over the 9 taps x CIN channels, a
//   stage to a tap.  The tile's rows r0 - 4 .. r0 + 131 are loaded once by TMA straight from the
//   activation matrix (rows before 0 or past the end come back as zeros) and tap t reads them
//   from row t on; a stage holds the tap's CIN columns of Wk.  Persistent: one CTA per SM walks
//   the tiles; one thread streams rows and stages through mbarrier rings, one warp issues the
//   MMAs of a tile into one of two TMEM accumulators, and eight or sixteen warps read the other
//   accumulator back and apply the epilogue meanwhile (details below).
// wgrad_tc_kernel<CIN>: part[chunk][m = t*CIN + c][n] = sum over the chunk's rows r of
//   X[r + t - 4, c] * dY[r, n] -- a GEMM whose K runs over rows.  Both operands are read
//   MN-major (channels contiguous, one row per K index), so the tap shift stays on the row
//   coordinate of the TMA load.  One CTA = 128 values of m (one tap of 128 channels, or four
//   taps of 32) x 128 n, over `rows_per_chunk` rows in stages of 64 (about one CTA per SM,
//   each a long K loop through a 6-stage ring).
#pragma once

#include <cuda_bf16.h>

#include "tc_gemm.cuh"

namespace cm {

// Epilogues of conv_tc_kernel (rows whose rowseq is negative are gap rows and give zeros):
//   kEpiRelu   out = bf16(relu(acc + bias))
//   kEpiPool   v[seq] += (acc + bias) / len(seq) for every real row (mean pooling; the
//              pre-pooling activations are never stored).  The sums are kept in 64-bit fixed
//              point (units of 2^-32) so that the atomic adds commute: v does not depend on
//              the order in which CTAs finish, and neither do the ranker's logits.
//   kEpiSum    colsum[seq] += bf16(relu(acc + bias)) over every real row, in 64-bit fixed point
//              like Pool but in units of the weights' scale and the sequence's length (sum_unit),
//              so that no sum of these activations can leave 64 bits or fall below the unit
//              whatever the scale of the weights; the rows within 4 of a sequence's ends also go
//              to `edge`, the others nowhere (the linear third layer needs no more of the second
//              one, see pool_linear_kernel)
//   kEpiGate   out = bf16(gate > 0 ? acc : 0), and colsum[n] += the column sums of those
//              values (the bias gradient of the layer below)
//   kEpiEmbed  dE[code][c] += acc for every real row (the embedding table's gradient; dX0 is
//              never stored)
enum Epi : int { kEpiRelu = 0, kEpiPool = 1, kEpiGate = 2, kEpiEmbed = 3, kEpiSum = 4 };

struct ConvEpi {
    const float* bias;          // Relu, Pool, Sum
    const int32_t* rowseq;      // every mode: sequence index of a row, < 0 for gap rows
    const __nv_bfloat16* gate;  // Gate
    __nv_bfloat16* out;         // Relu, Gate
    const int32_t* slen;        // Pool, Sum: rows of every sequence
    const int64_t* srow;        // Sum: first row of every sequence
    __nv_bfloat16* edge;        // Sum: ns x 8 x NOUT, rows 0..3 from the start, 0..3 from the end
    const uint8_t* codes;       // Embed: residue code of every row
    float* acc;                 // Gate: column sums; Embed: dE (20 x NOUT)
    unsigned long long* acc64;  // Pool: v in units of 2^-32, Sum: column sums (ns x NOUT)
    const float* scale;         // Sum: units of an activation of 1 in a sequence of one row
};

constexpr double kPoolScale = 4294967296.0;   // 2^32: fixed-point unit of the pooled sums

// v in fixed point: the scaling by a power of two is exact in float, so only the conversion
// rounds (to nearest); no double-precision operation
__device__ __forceinline__ long long to_fixed(float v, float unit = (float)kPoolScale)
{
    return __float2ll_rn(v * unit);
}

// 2^-k for the least k with 2^k >= len: with it a sum over a sequence's rows is no larger than the
// largest of them
__device__ __forceinline__ float inv_pow2_len(int len)
{
    return __int_as_float((127 - (len <= 1 ? 0 : 32 - __clz(len - 1))) << 23);
}
// fixed-point units of an activation of 1 in the column sums of a sequence of `len` rows
__device__ __forceinline__ float sum_unit(float scale, int len) { return scale * inv_pow2_len(len); }

namespace tc {

constexpr int kTcRows = 128;        // rows (M) per CTA

// Column sums of a warp's 32 x 32 tile (lane = row, v[0..31] = columns): a transposing
// reduction (halve the columns a lane keeps at every step, adding the partner lane's copy of
// them), 31 shuffles in all; afterwards lane c holds the sum of column c.  Overwrites v.
__device__ __forceinline__ float warp_colsum32(float* v, int lane)
{
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
        const bool up = (lane & s) != 0;
#pragma unroll
        for (int k = 0; k < s; ++k) {
            const float keep = up ? v[k + s] : v[k];
            const float give = up ? v[k] : v[k + s];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, give, s);
        }
    }
    return v[0];
}

// The same for 64-bit integers.
__device__ __forceinline__ long long warp_colsum32(long long* v, int lane)
{
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
        const bool up = (lane & s) != 0;
#pragma unroll
        for (int k = 0; k < s; ++k) {
            const long long keep = up ? v[k + s] : v[k];
            const long long give = up ? v[k] : v[k + s];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, give, s);
        }
    }
    return v[0];
}

// ---- persistent convolution kernel ------------------------------------------------------
// One CTA per SM walks the 128-row tiles blockIdx.x, blockIdx.x + gridDim.x, ...  Warp 0
// (one thread) streams the A / B stages of every tile through a ring of STAGES shared-memory
// stages, across tile boundaries; warp 1 (one thread) issues the MMAs of a tile into one of
// two TMEM accumulators (tile i uses buffer i & 1) and commits it; warps 2-9 (and 10-17, taking
// every other tile, in some layers) read a finished accumulator back (warp w owns TMEM lanes 32 (w % 4) .., warps w and w + 4 one half of the
// columns each) and apply the epilogue while the MMAs of the next tile run, then release the
// buffer.  What the epilogue needs of its rows (sequence, gate) is loaded before the wait for
// the MMAs, the bias sits in shared memory, and the results leave through 4 KB of shared memory
// per warp by TMA (with each thread loading the bias and storing its own row, the pooling layer
// over 1.7M rows took 624 us against 556, the 32-channel one 337 against 224).  Barriers: full / empty per stage
// (TMA bytes landed / MMAs done reading), tfull / tempty per accumulator (MMAs done /
// epilogue done reading).  Every wait is bounded; a role that gives up sets the error word
// and stops, the others then give up at their next wait, and the teardown waits (bounded) for
// the copies and MMAs still in flight before the tensor memory is freed.
constexpr int kConvEpiWarps = 8;    // two per TMEM lane quadrant, each half of the columns
// Groups of epilogue warps: two, taking the tiles in turn, for the 32-channel layer, whose MMAs
// take a quarter of a 128-channel layer's time and whose epilogue's latency bounds it (1.7M rows:
// 174 us with one group, 114 with two); one for the others, where more warps slow the issue of
// the MMAs (the second layer with column sums 382 us with one, 405 with two).
constexpr int conv_epi_groups(int CIN) { return CIN == 32 ? 2 : 1; }
constexpr int conv_threads(int CIN) { return 64 + 32 * kConvEpiWarps * conv_epi_groups(CIN); }
constexpr int kConvStageBudget = 192 * 1024;

template <int CIN, int NOUT, int EPI>
struct ConvCfg {
    static constexpr int BK = (CIN == 32) ? 32 : 64;       // channels per swizzle row
    static constexpr int KB_PER_TAP = CIN / BK;            // boxes of a tap: one stage holds a tap
    // A tile's A rows r0 - 4 .. r0 + 131 are loaded once per block of BK channels, and tap t reads
    // them from row t on (the descriptor start moves by whole rows; the swizzle follows the
    // address, so the shifted view stays valid)
    static constexpr int AROWS = kTcRows + 8;
    static constexpr int A_BOX_BYTES = AROWS * BK * 2;     // one channel block of a tile
    static constexpr int A_TILE_BYTES = KB_PER_TAP * A_BOX_BYTES;
    static constexpr int A_SLOTS = (CIN == 32) ? 4 : 2;    // tiles in flight
    static constexpr int A_SLOTS_BYTES = A_SLOTS * A_TILE_BYTES;
    static constexpr int B_BOX_BYTES = NOUT * BK * 2;
    static constexpr int STAGE_BYTES = KB_PER_TAP * B_BOX_BYTES;     // a tap's weights
    // RESIDENT: all nine taps' weights fit beside the tiles and are loaded once per CTA;
    // otherwise they stream through a ring of stages, once per tile
    static constexpr bool RESIDENT = 9 * STAGE_BYTES <= 80 * 1024;
    static constexpr int STAGES = RESIDENT ? 9 : (kConvStageBudget - A_SLOTS_BYTES) / STAGE_BYTES;
    static constexpr uint32_t SWZ = (BK == 64) ? kSwizzle128 : kSwizzle64;
    static constexpr uint32_t SBO = 8 * BK * 2;
    static constexpr uint32_t TMEM_COLS = 2 * NOUT < 32 ? 32 : 2 * NOUT;   // two accumulators
    // the embedding-gradient epilogue's scratch: per epilogue warp a 32 x 33 transpose tile
    // and private bins of 20 codes x NOUT channels
    static constexpr int EMB_FLOATS = 4 * (32 * 33 + 20 * NOUT);
    static constexpr int GROUPS = conv_epi_groups(CIN);
    static constexpr int OUT_BYTES =                       // boxes of 32 rows x 64 channels
        EPI == kEpiRelu || EPI == kEpiGate ? GROUPS * kConvEpiWarps * 32 * 128 : 0;
    static constexpr int SMEM = A_SLOTS_BYTES + STAGES * STAGE_BYTES + OUT_BYTES + 1024;
    static_assert(A_BOX_BYTES % (8 * BK * 2) == 0 && A_SLOTS_BYTES % 1024 == 0 &&
                  STAGE_BYTES % 1024 == 0, "tiles start on whole swizzle atoms");
};

// What the epilogue of a tile needs of this thread's row (TMEM lane 32 q + lane), loaded while
// the tile's MMAs run.
struct EpiRow {
    int32_t seq;             // < 0: a gap row, or past the end
    float inv_len;           // Pool
    float unit;              // Sum
    int edge_lo, edge_hi;    // Sum: distance to the sequence's first and last row
    int code;                // Embed
    bool binned;
    uint32_t gate[2];        // Gate: bit c = the gate of column 32 j0 + c is open
};

template <int NOUT, int EPI>
__device__ __forceinline__ EpiRow epi_row(int64_t r, int64_t R, int j0, const ConvEpi& ep, float scale)
{
    EpiRow e{};
    const bool in = r < R;
    e.seq = in ? ep.rowseq[r] : -1;
    if (EPI == kEpiPool && e.seq >= 0) e.inv_len = 1.f / (float)ep.slen[e.seq];
    if (EPI == kEpiSum && e.seq >= 0) {
        const int64_t pos = r - ep.srow[e.seq];
        const int len = ep.slen[e.seq];
        e.edge_lo = (int)min(pos, (int64_t)4);
        e.edge_hi = (int)min((int64_t)len - 1 - pos, (int64_t)4);
        e.unit = sum_unit(scale, len);
    }
    if (EPI == kEpiEmbed) {
        // rows of letters outside the 20 embedded ones (zero embedding) add nothing
        const int code = e.seq >= 0 ? (int)ep.codes[r] : 20;
        e.binned = code < 20;
        e.code = e.binned ? code : 0;
    }
    if (EPI == kEpiGate && in) {
        const uint4* g4 = reinterpret_cast<const uint4*>(ep.gate + r * NOUT + 32 * j0);
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const uint4 gw = g4[t];
            const uint32_t w[4] = {gw.x, gw.y, gw.z, gw.w};
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const __nv_bfloat162 gz = *reinterpret_cast<const __nv_bfloat162*>(&w[h]);
                const uint32_t open = (__bfloat162float(gz.x) > 0.f ? 1u : 0u) |
                                      (__bfloat162float(gz.y) > 0.f ? 2u : 0u);
                e.gate[t >> 2] |= open << (8 * (t & 3) + 2 * h);
            }
        }
    }
    return e;
}

// Epilogue of one accumulator: this thread's row of the tile, columns 32 j0 .. 32 j1.
// Embed: lane = channel after a transpose through shared memory, adding into the warp's own
// bins (no atomics); Gate: column sums per warp into s_red (shared atomics, one per column).
// Relu and Gate leave their rows as bf16 in `out`, the warp's 32 x 64 box in the 128-byte swizzle.
template <int CIN, int NOUT, int EPI>
__device__ __forceinline__ void conv_epilogue(uint32_t tacc, int q, int lane, int j0, int j1,
                                              const EpiRow& e, const ConvEpi& ep,
                                              const float* s_bias, float* s_red, float* emb,
                                              uint8_t* out)
{
    const bool real = e.seq >= 0;
    // Pool, Sum: a warp whose real rows all belong to one sequence reduces its 32 rows first
    int32_t lead = -1;
    bool one_seq = false;
    float unit = (float)kPoolScale;                // of that sequence
    if (EPI == kEpiPool || EPI == kEpiSum) {
        lead = __reduce_max_sync(0xffffffffu, e.seq);
        one_seq = __all_sync(0xffffffffu, e.seq < 0 || e.seq == lead);
        // (positive floats order as their bits; gap rows have 0)
        if (EPI == kEpiSum) unit = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(e.unit)));
    }
    const float row_unit = EPI == kEpiSum ? e.unit : (float)kPoolScale;
#pragma unroll 1
    for (int j = j0; j < j1; ++j) {
        float v[32];
        tmem_ld32(tacc + ((uint32_t)(q * 32) << 16) + (uint32_t)(j * 32), v);
        const int n0 = j * 32;
        if (EPI == kEpiEmbed) {
            // transpose the warp's 32 rows x 32 channels, then lane c adds channel c of every
            // row into bin[code of the row][c] of this warp
            float* tile = emb;                                   // [32][33]
            float* bins = emb + 32 * 33;                         // [20][NOUT]
#pragma unroll
            for (int c = 0; c < 32; ++c) tile[c * 33 + lane] = e.binned ? v[c] : 0.f;
            __syncwarp();
#pragma unroll 4
            for (int rr = 0; rr < 32; ++rr) {
                const int cd = __shfl_sync(0xffffffffu, e.code, rr);
                bins[cd * NOUT + n0 + lane] += tile[lane * 33 + rr];
            }
            __syncwarp();
            continue;
        }
        if (EPI == kEpiPool || EPI == kEpiRelu || EPI == kEpiSum) {
            const float4* b4 = reinterpret_cast<const float4*>(s_bias + n0);
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const float4 b = b4[t];
                v[4 * t] += b.x;
                v[4 * t + 1] += b.y;
                v[4 * t + 2] += b.z;
                v[4 * t + 3] += b.w;
            }
        }
        if (EPI == kEpiSum) {
            uint32_t w[16];
#pragma unroll
            for (int t = 0; t < 16; ++t) {
                const __nv_bfloat162 pr = __floats2bfloat162_rn(real ? fmaxf(v[2 * t], 0.f) : 0.f,
                                                                real ? fmaxf(v[2 * t + 1], 0.f) : 0.f);
                w[t] = *reinterpret_cast<const uint32_t*>(&pr);
                v[2 * t] = __bfloat162float(pr.x);
                v[2 * t + 1] = __bfloat162float(pr.y);
            }
            if (real && min(e.edge_lo, e.edge_hi) < 4) {
                __nv_bfloat16* dst = ep.edge + (int64_t)e.seq * 8 * NOUT + n0;
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const uint4 x = make_uint4(w[4 * t], w[4 * t + 1], w[4 * t + 2], w[4 * t + 3]);
                    if (e.edge_lo < 4) reinterpret_cast<uint4*>(dst + e.edge_lo * NOUT)[t] = x;
                    if (e.edge_hi < 4) reinterpret_cast<uint4*>(dst + (4 + e.edge_hi) * NOUT)[t] = x;
                }
            }
        }
        if (EPI == kEpiPool || EPI == kEpiSum) {
            if (EPI == kEpiPool) {
#pragma unroll
                for (int t = 0; t < 32; ++t) v[t] = real ? v[t] * e.inv_len : 0.f;
            }
            if (one_seq) {
                const float t = warp_colsum32(v, lane);
                if (lead >= 0)
                    atomicAdd(ep.acc64 + (int64_t)lead * NOUT + n0 + lane, (unsigned long long)to_fixed(t, unit));
            } else {
                // the rows of each sequence, summed in fixed point (one atomic per column)
                uint32_t left = __ballot_sync(0xffffffffu, real);
                while (left) {
                    const int32_t seq = __shfl_sync(0xffffffffu, e.seq, __ffs(left) - 1);
                    long long w[32];
#pragma unroll
                    for (int t = 0; t < 32; ++t) w[t] = e.seq == seq ? to_fixed(v[t], row_unit) : 0;
                    const long long t = warp_colsum32(w, lane);
                    atomicAdd(ep.acc64 + (int64_t)seq * NOUT + n0 + lane, (unsigned long long)t);
                    left &= ~__ballot_sync(0xffffffffu, e.seq == seq);
                }
            }
            continue;
        }
        const uint32_t gate = j == j0 ? e.gate[0] : e.gate[1];
#pragma unroll
        for (int t = 0; t < 32; ++t) {
            if (EPI == kEpiRelu) v[t] = real ? fmaxf(v[t], 0.f) : 0.f;
            else v[t] = real && ((gate >> t) & 1u) ? v[t] : 0.f;
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            uint32_t w[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const __nv_bfloat162 pr = __floats2bfloat162_rn(v[8 * t + 2 * h], v[8 * t + 2 * h + 1]);
                w[h] = *reinterpret_cast<const uint32_t*>(&pr);
            }
            *reinterpret_cast<uint4*>(out + lane * 128 + (((4 * (j - j0) + t) ^ (lane & 7)) << 4)) =
                make_uint4(w[0], w[1], w[2], w[3]);
        }
        if (EPI == kEpiGate && ep.acc) {
            const float t = warp_colsum32(v, lane);
            atomicAdd(s_red + n0 + lane, t);
        }
    }
}

template <int CIN, int NOUT, int EPI>
__global__ void __launch_bounds__(conv_threads(CIN), 1)
conv_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmOut, int64_t R, const ConvEpi ep, int32_t* err)
{
    using C = ConvCfg<CIN, NOUT, EPI>;
    constexpr int S = C::STAGES;
    constexpr uint32_t IDESC = idesc_bf16_f32(kTcRows, NOUT, false, false);
    // column chunks of 32 per epilogue warp pair; with one chunk only the first four warps
    constexpr int NCH = NOUT / 32;
    constexpr int kEpiActive = NCH >= 2 ? kConvEpiWarps : 4;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    constexpr int NA = C::A_SLOTS;
    __shared__ __align__(8) uint64_t full[S], empty[S], afull[NA], aempty[NA], tfull[2], tempty[2], done;
    __shared__ uint32_t tmem_slot;
    __shared__ int32_t s_issued, s_consumed, s_aissued, s_aconsumed, s_abort;
    __shared__ float s_red[EPI == kEpiGate ? NOUT : 1];
    constexpr bool BIAS = EPI == kEpiRelu || EPI == kEpiPool || EPI == kEpiSum;
    __shared__ __align__(16) float s_bias[BIAS ? NOUT : 4];
    constexpr bool STORES = EPI == kEpiRelu || EPI == kEpiGate;
    __shared__ float s_emb[EPI == kEpiEmbed ? C::EMB_FLOATS : 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t ntiles = (R + kTcRows - 1) / kTcRows;
    if (EPI == kEpiGate)
        for (int i = threadIdx.x; i < NOUT; i += conv_threads(CIN)) s_red[i] = 0.f;
    if (BIAS)
        for (int i = threadIdx.x; i < NOUT; i += conv_threads(CIN)) s_bias[i] = ep.bias[i];
    if (EPI == kEpiEmbed)
        for (int i = threadIdx.x; i < C::EMB_FLOATS; i += conv_threads(CIN)) s_emb[i] = 0.f;

    if (threadIdx.x == 0) {
        prefetch_tmap(&tmA);
        prefetch_tmap(&tmB);
        if (STORES) prefetch_tmap(&tmOut);
        for (int s = 0; s < S; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], kEpiActive);
        }
        for (int a = 0; a < NA; ++a) { mbar_init(&afull[a], 1); mbar_init(&aempty[a], 1); }
        mbar_init(&done, 1);
        fence_mbar_init();
        s_issued = 0;
        s_consumed = 0;
        s_aissued = 0;
        s_aconsumed = 0;
        s_abort = *reinterpret_cast<volatile int32_t*>(err);   // an earlier launch gave up
    }
    __syncthreads();
    if (s_abort) return;
    if (warp == 1) tmem_alloc(&tmem_slot, C::TMEM_COLS);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = tmem_slot;

    uint8_t* bring = smem + C::A_SLOTS_BYTES;                // weight stages
    if (warp == 0) {
        if (lane == 0) {
            // ring position: stage s, phase ph of its barriers; it stages issued so far
            int it = 0, i = 0, s = 0;
            uint32_t ph = 0;
            bool ok = true;
            auto load_tap = [&](int tap) {
                mbar_expect_tx(&full[s], C::STAGE_BYTES);
                for (int cb = 0; cb < C::KB_PER_TAP; ++cb)
                    tma_load_2d(bring + s * C::STAGE_BYTES + cb * C::B_BOX_BYTES, &tmB,
                                tap * CIN + cb * C::BK, 0, &full[s]);
                ++it;
                if (++s == S) { s = 0; ph ^= 1; }
            };
            for (int64_t tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++i) {
                const int a = i % NA;
                if (i >= NA && !mbar_wait(&aempty[a], ((i / NA) - 1) & 1, err)) break;
                mbar_expect_tx(&afull[a], C::A_TILE_BYTES);
                for (int cb = 0; cb < C::KB_PER_TAP; ++cb)
                    tma_load_2d(smem + a * C::A_TILE_BYTES + cb * C::A_BOX_BYTES, &tmA, cb * C::BK,
                                (int32_t)(tile * kTcRows) - 4, &afull[a]);
                if (C::RESIDENT && i > 0) continue;
                for (int tap = 0; tap < 9; ++tap) {
                    if (it >= S && !mbar_wait(&empty[s], ph ^ 1, err)) { ok = false; break; }
                    load_tap(tap);
                }
            }
            s_issued = it;
            s_aissued = i;
        }
    } else if (warp == 1) {
        // The whole warp walks the stages (a tap each) and one elected thread issues, so that the
        // operands stay in uniform registers; descriptors are built once and a stage, tap or K step
        // moves their low word.  The issue is what bounds the kernel: a 128-channel layer over
        // 1.7M rows (an MMA takes 64 tensor cycles) took 532 us with one lane building every
        // descriptor (170 cycles an MMA), 423 with the descriptors moved, 378 with the whole
        // warp, 342 (109 cycles) with a barrier per tap instead of per half tap; leaving out the
        // weights' loads or the epilogue changes it by 3 %.
        const uint64_t adesc = smem_desc(smem, 16, C::SBO, C::SWZ);
        const uint64_t sdesc = smem_desc(bring, 16, C::SBO, C::SWZ);
        const uint32_t alo = (uint32_t)adesc, slo = (uint32_t)sdesc, hi = (uint32_t)(adesc >> 32);
        int it = 0, i = 0, s = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int64_t tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++i) {
            const int b = i & 1, a_slot = i % NA;
            if (i >= 2) ok = mbar_wait(&tempty[b], ((i / 2) - 1) & 1, err);
            ok = ok && mbar_wait(&afull[a_slot], (i / NA) & 1, err);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;
            fence_after_sync();
            const uint32_t acc = tmem + (uint32_t)(b * NOUT);
            const uint32_t atile = alo + (uint32_t)(a_slot * C::A_TILE_BYTES >> 4);
            auto issue_tap = [&](int tap, int st) {
                const uint32_t a = atile + (uint32_t)(tap * C::BK * 2 >> 4);
                const uint32_t w = slo + (uint32_t)(st * C::STAGE_BYTES >> 4);
#pragma unroll
                for (int cb = 0; cb < C::KB_PER_TAP; ++cb)
#pragma unroll
                    for (int k = 0; k < C::BK / 16; ++k)
                        mma_bf16(acc, a + (cb * C::A_BOX_BYTES >> 4) + 2 * k, hi,
                                 w + (cb * C::B_BOX_BYTES >> 4) + 2 * k, hi, IDESC,
                                 k > 0 || cb > 0 || tap > 0);
            };
            if (C::RESIDENT && i > 0) {           // every tap's weights are there
                if (elect_one()) {
#pragma unroll
                    for (int tap = 0; tap < 9; ++tap) issue_tap(tap, tap);
                }
                __syncwarp();
            } else {
                for (int tap = 0; tap < 9; ++tap, ++it) {
                    if (!(ok = __all_sync(0xffffffffu, mbar_wait(&full[s], ph, err)))) break;
                    fence_after_sync();
                    if (elect_one()) {
                        issue_tap(tap, s);
                        mma_commit(&empty[s]);
                    }
                    __syncwarp();
                    if (++s == S) { s = 0; ph ^= 1; }
                }
            }
            if (!ok) break;
            if (elect_one()) {
                mma_commit(&aempty[a_slot]);
                mma_commit(&tfull[b]);
            }
            __syncwarp();
        }
        if (elect_one()) {
            s_consumed = it;
            s_aconsumed = i;
            mma_commit(&done);            // arrives once every MMA issued above has completed
        }
        __syncwarp();
    } else if ((warp - 2) % kConvEpiWarps < kEpiActive) {
        const int group = (warp - 2) / kConvEpiWarps, ew = (warp - 2) % kConvEpiWarps;
        const int q = warp & 3;           // TMEM lane quadrant of this warp
        const int half = kEpiActive == 8 ? ew / 4 : 0;
        const int j0 = kEpiActive == 8 ? half * (NCH / 2) : 0;
        const int j1 = kEpiActive == 8 ? (half + 1) * (NCH / 2) : NCH;
        float* emb = s_emb + (EPI == kEpiEmbed ? ew * (32 * 33 + 20 * NOUT) : 0);
        uint8_t* out = bring + S * C::STAGE_BYTES + (warp - 2) * (32 * 128);
        const float scale = EPI == kEpiSum ? *ep.scale : 0.f;
        int i = group;
        for (int64_t tile = blockIdx.x + (int64_t)group * gridDim.x; tile < ntiles;
             tile += (int64_t)C::GROUPS * gridDim.x, i += C::GROUPS) {
            const int b = i & 1;
            const int64_t row0 = tile * kTcRows + q * 32;
            const EpiRow er = epi_row<NOUT, EPI>(row0 + lane, R, j0, ep, scale);
            const bool ok = mbar_wait(&tfull[b], (i / 2) & 1, err);
            if (!__all_sync(0xffffffffu, ok)) break;      // warp-uniform: tcgen05.ld is warp-wide
            fence_after_sync();
            if (STORES) {                                 // the box of the tile before has been read
                if (lane == 0) bulk_wait_read();
                __syncwarp();
            }
            conv_epilogue<CIN, NOUT, EPI>(tmem + (uint32_t)(b * NOUT), q, lane, j0, j1, er, ep, s_bias,
                                          s_red, emb, out);
            fence_before_sync();
            if (STORES) fence_async_proxy();
            __syncwarp();
            if (lane == 0) {
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n"
                             ::"r"(smem_addr(&tempty[b])) : "memory");
                if (STORES && row0 < R) tma_store_2d(&tmOut, out, 32 * j0, (int32_t)row0);
            }
        }
        if (STORES && lane == 0) bulk_wait_all();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        // MMAs issued but not awaited by an epilogue, and loads issued but never consumed
        // (only after a wait gave up): let them finish before the memory goes away
        mbar_wait(&done, 0, err);
        for (int it = s_consumed; it < s_issued; ++it)
            mbar_wait(&full[it % S], (it / S) & 1, err);
        for (int i = s_aconsumed; i < s_aissued; ++i) mbar_wait(&afull[i % NA], (i / NA) & 1, err);
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    if (EPI == kEpiGate && ep.acc)
        for (int i = threadIdx.x; i < NOUT; i += conv_threads(CIN))
            if (s_red[i] != 0.f) atomicAdd(ep.acc + i, s_red[i]);
    if (EPI == kEpiEmbed) {
        const int per = 32 * 33 + 20 * NOUT;
        for (int i = threadIdx.x; i < 20 * NOUT; i += conv_threads(CIN)) {
            float t = 0.f;
#pragma unroll
            for (int w = 0; w < 4; ++w) t += s_emb[w * per + 32 * 33 + i];
            if (t != 0.f) atomicAdd(ep.acc + i, t);
        }
    }
    if (warp == 1) tmem_free(tmem, C::TMEM_COLS);
}

template <int CIN>
struct WgradCfg {
    static constexpr int CW = (CIN == 32) ? 32 : 64;        // channels per swizzle row of A
    static constexpr int A_BOXES = 128 / CW;                // boxes making up M = 128
    static constexpr int BKR = 64;                          // rows (K) per stage
    static constexpr int A_BYTES = 128 * BKR * 2;
    static constexpr int B_BYTES = 128 * BKR * 2;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr uint32_t A_SWZ = (CW == 64) ? kSwizzle128 : kSwizzle64;
    static constexpr uint32_t A_ROW = CW * 2;               // bytes per K row of one A box
    static constexpr int STAGES = 6;                       // one CTA per SM, a deep ring
    static constexpr int SMEM = STAGES * STAGE_BYTES + 1024;
    static constexpr int MTILES = (9 * CIN + 127) / 128;
};

template <int CIN>
__global__ void __launch_bounds__(128, 1)
wgrad_tc_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmD,
                int64_t rows_per_chunk, float* __restrict__ part, int MPAD, int32_t* err)
{
    using C = WgradCfg<CIN>;
    constexpr uint32_t IDESC = idesc_bf16_f32(128, 128, true, true);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full[C::STAGES], empty[C::STAGES], done;
    __shared__ uint32_t tmem_slot;
    __shared__ int32_t s_issued, s_consumed, s_abort;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mtile = blockIdx.x;
    const int64_t chunk = blockIdx.y;
    const int64_t rbeg = chunk * rows_per_chunk;
    const int nkb = (int)(rows_per_chunk / C::BKR);
    // taps held by this m-tile's A boxes (a box past the last tap is not loaded)
    const int nbox = (CIN == 32) ? min(C::A_BOXES, 9 - 4 * mtile) : C::A_BOXES;
    const uint32_t stage_tx = (uint32_t)(nbox * (C::A_BYTES / C::A_BOXES) + C::B_BYTES);

    if (threadIdx.x == 0) {
        prefetch_tmap(&tmX);
        prefetch_tmap(&tmD);
        for (int s = 0; s < C::STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        mbar_init(&done, 1);
        fence_mbar_init();
        s_issued = 0;
        s_consumed = 0;
        s_abort = *reinterpret_cast<volatile int32_t*>(err);
    }
    __syncthreads();
    if (s_abort) return;
    if (warp == 2) tmem_alloc(&tmem_slot, 128);
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = tmem_slot;

    if (warp == 0 && lane == 0) {
        int kb = 0;
        for (; kb < nkb; ++kb) {
            const int s = kb % C::STAGES;
            if (kb >= C::STAGES && !mbar_wait(&empty[s], ((kb / C::STAGES) - 1) & 1, err)) break;
            const int64_t rr = rbeg + (int64_t)kb * C::BKR;
            uint8_t* st = smem + s * C::STAGE_BYTES;
            mbar_expect_tx(&full[s], stage_tx);
            for (int q = 0; q < nbox; ++q) {
                // CIN = 128: tap = mtile, channel half q; CIN = 32: tap 4 mtile + q
                const int tap = (CIN == 32) ? 4 * mtile + q : mtile;
                const int c0 = (CIN == 32) ? 0 : q * 64;
                tma_load_2d(st + q * (C::A_BYTES / C::A_BOXES), &tmX, c0,
                            (int32_t)(rr + tap - 4), &full[s]);
            }
            tma_load_2d(st + C::A_BYTES, &tmD, 0, (int32_t)rr, &full[s]);
            tma_load_2d(st + C::A_BYTES + C::B_BYTES / 2, &tmD, 64, (int32_t)rr, &full[s]);
        }
        s_issued = kb;
    } else if (warp == 1 && lane == 0) {
        int kb = 0;
        for (; kb < nkb; ++kb) {
            const int s = kb % C::STAGES;
            if (!mbar_wait(&full[s], (kb / C::STAGES) & 1, err)) break;
            fence_after_sync();
            const uint8_t* a = smem + s * C::STAGE_BYTES;
            const uint8_t* b = a + C::A_BYTES;
#pragma unroll
            for (int k = 0; k < C::BKR / 16; ++k)
                mma_bf16(tmem,
                         smem_desc(a + 16 * k * C::A_ROW, C::A_BYTES / C::A_BOXES, 8 * C::A_ROW,
                                   C::A_SWZ),
                         smem_desc(b + 16 * k * 128, C::B_BYTES / 2, 1024, kSwizzle128), IDESC,
                         (kb | k) != 0);
            mma_commit(&empty[s]);
        }
        s_consumed = kb;
        mma_commit(&done);
    }
    __syncwarp();
    const bool ok = mbar_wait(&done, 0, err);
    fence_after_sync();
    // warp-uniform: the TMEM loads below are warp-wide instructions
    if (__all_sync(0xffffffffu, ok && *reinterpret_cast<volatile int32_t*>(err) == 0)) {
        const int m = mtile * 128 + warp * 32 + lane;
        float* dst = part + (chunk * (int64_t)MPAD + m) * 128;
#pragma unroll 1
        for (int j = 0; j < 4; ++j) {
            float v[32];
            tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(j * 32), v);
            float4* o = reinterpret_cast<float4*>(dst + j * 32);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                o[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        }
    }
    fence_before_sync();
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int kb = s_consumed; kb < s_issued; ++kb)
            mbar_wait(&full[kb % C::STAGES], (kb / C::STAGES) & 1, err);
    }
    __syncthreads();
    if (warp == 2) tmem_free(tmem, 128);
}

}  // namespace tc
}  // namespace cm
