// int32 Smith-Waterman wavefront of one warp over one strip: the rescoring of pairs beyond the
// int16 range, and with the first cell that reaches the optimum the alignment-cells pass.  Same
// recurrences as the int16 kernel.
//
// Mapping.  The matrix is x (streamed) against y (held): lane l holds R consecutive y positions
// of a strip of 32 R, and at step t works on the 4 x positions of group t - l (x position k of a
// group trails position k - 1 by one y position inside the lane: four independent chains); H - o
// and E of the lane's last y position pass to its right neighbour by shuffle.  A strip hands
// (H - o, E) of its last y position to the next strip through memory, one pair per x position.
// Per cell, with the profile holding plain scores as bytes (four per word, pads -128):
//   E = max(E - e, (H - o)_left),  F = max(F - e, (H - o)_up),
//   D = H_diag + S (one dp4a: byte select, sign extension and add),  H = max(D, E, F, 0)
// that is 3 DPX operations and a dot product, and half a 3-input maximum of H (kTrackNone) or of
// the key 8 H + 7 - (y position in the lane) over each x position.  So the position costs one
// comparison per x position and lane, not per cell: the largest key says the score and the first
// y position that has it.
//   kTrackXRows: x are the rows, y the columns of the pair.  A new best needs a larger score;
//     x positions come in order, so the first row stays.
//   kTrackYRows: y are the rows, x the columns.  A larger key is a larger score or the same one
//     in an earlier row; an equal key is the same row, whose first column stays.
// Key range: 8 H + 7 < 2^31, so tracked scores stay below 2^28 (kWaveScoreLimit).
#pragma once
#include <cstdint>

#include "dp32.cuh"

namespace cm {
namespace {

enum WaveTrack : int { kTrackNone = 0, kTrackXRows = 1, kTrackYRows = 2 };

constexpr int kWaveRows = 4;                      // x positions per step
constexpr int kWaveProf = kProfRows * 32;         // uint2 entries of a strip's profile

// profile of y positions [y0, y0 + 32 R) of y[0..n) (back to front when `reverse`) against every
// residue below `alpha`: mat[y residue * ys + x residue * xs]
__device__ __forceinline__ void wave_profile(uint2* prof, const uint8_t* y, int64_t n, bool reverse,
                                             int64_t y0, int R, const int8_t* mat, int ys, int xs,
                                             int alpha)
{
    const int lane = threadIdx.x & 31;
    int off[kWaveMaxR];
#pragma unroll
    for (int c = 0; c < kWaveMaxR; ++c) {
        const int64_t p = y0 + lane * R + c;
        const bool in = c < R && p < n;
        off[c] = in ? (int)(reverse ? y[n - 1 - p] : y[p]) * ys : -1;
    }
    for (int r = 0; r < kProfRows; ++r) {
        uint32_t w[2] = {0u, 0u};
#pragma unroll
        for (int c = 0; c < kWaveMaxR; ++c) {
            const int8_t v = (r < alpha && off[c] >= 0) ? mat[off[c] + r * xs] : (int8_t)-128;
            w[c >> 2] |= (uint32_t)(uint8_t)v << (8 * (c & 3));
        }
        prof[r * 32 + lane] = make_uint2(w[0], w[1]);
    }
}

struct WaveStrip {
    const uint2* prof;
    const uint8_t* x;          // streamed sequence, xn positions (back to front when reverse)
    int32_t xn;
    bool reverse;
    int o, ge;
    const int2* bin;           // previous strip's last position (null: the matrix's edge), 16-byte
    int2* bout;                // aligned whole groups; this strip's (null: the last); may be bin
    int32_t y0;                // first y position of the strip
};

// One strip.  wait(groups) returns once the first `groups` groups of bin are written (false gives
// up: the strip returns false on every lane); lane 31 calls publish(groups) after that many of
// bout are.  The result, on every lane: score, x and y position of its first cell (-1 if 0, or
// untracked).
template <int R, int TRACK, class Wait, class Publish>
__device__ __forceinline__ bool wave_strip(const WaveStrip& s, Wait&& wait, Publish&& publish,
                                           int32_t& score, int32_t& xpos, int32_t& ypos)
{
    constexpr int NR = kWaveRows;
    constexpr uint32_t kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint2* plane = s.prof + lane;
    const uint8_t* x = s.x;
    const int32_t xn = s.xn, groups = (xn + NR - 1) / NR;
    const int o = s.o, ge = s.ge;
    const bool reverse = s.reverse;
    const int2* bin = s.bin;
    int2* bout = s.bout;
    int32_t hp[R], fp[R];                         // H - o and F of the x position before
#pragma unroll
    for (int k = 0; k < R; ++k) { hp[k] = -o; fp[k] = -o; }
    int32_t oh[NR], oe[NR], bh[NR], be[NR];
#pragma unroll
    for (int q = 0; q < NR; ++q) { oh[q] = -o; oe[q] = -o; bh[q] = -o; be[q] = -o; }
    int32_t diag0 = -o, lkey = TRACK != kTrackNone ? 7 : 0, lx = -1;
    constexpr uint32_t kPads = (uint32_t)kPadCode * 0x01010101u;
    uint32_t cur = kPads, prev = kPads;

    for (int32_t t = 0; t < groups + 31; ++t) {
        const int j = t & 31;
        if (j == 0) {
            if (bin != nullptr && t < groups && !wait(min(t + 32, groups))) return false;
            prev = cur;
            cur = 0;
#pragma unroll
            for (int q = 0; q < NR; ++q) {
                const int32_t r = (t + lane) * NR + q;
                const uint32_t v = (r < xn) ? (uint32_t)(reverse ? x[xn - 1 - r] : x[r])
                                            : (uint32_t)kPadCode;
                cur |= min(v, (uint32_t)kPadCode) << (8 * q);
            }
            if (bin != nullptr && t + lane < groups) {
#pragma unroll
                for (int q = 0; q < NR; q += 2) {
                    const int4 u = __ldcg(reinterpret_cast<const int4*>(bin + (t + lane) * NR + q));
                    bh[q] = u.x; be[q] = u.y; bh[q + 1] = u.z; be[q + 1] = u.w;
                }
            }
        }
        const uint32_t rv = __shfl_sync(kAll, (lane <= j) ? cur : prev, (j - lane) & 31);
        int32_t h[NR], e[NR];
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            h[q] = __shfl_up_sync(kAll, oh[q], 1);
            e[q] = __shfl_up_sync(kAll, oe[q], 1);
        }
        if (bin != nullptr) {
#pragma unroll
            for (int q = 0; q < NR; ++q) {
                const int32_t u = __shfl_sync(kAll, bh[q], j), v = __shfl_sync(kAll, be[q], j);
                h[q] = lane == 0 ? u : h[q];
                e[q] = lane == 0 ? v : e[q];
            }
        } else {
#pragma unroll
            for (int q = 0; q < NR; ++q) {
                h[q] = lane == 0 ? -o : h[q];
                e[q] = lane == 0 ? -o : e[q];
            }
        }
        int32_t dg[NR], best[NR], pend[NR];
        uint2 w[NR];
        dg[0] = diag0 + o;
#pragma unroll
        for (int q = 1; q < NR; ++q) dg[q] = h[q - 1] + o;
        diag0 = h[NR - 1];
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            w[q] = plane[__byte_perm(rv, 0u, 0x4440u | q) * 32];
            best[q] = 0;
        }
#pragma unroll
        for (int k = 0; k < R + NR - 1; ++k) {
#pragma unroll
            for (int q = 0; q < NR; ++q) {
                const int c = k - q;
                if (c < 0 || c >= R) continue;
                e[q] = __viaddmax_s32(e[q], -ge, h[q]);
                const int32_t f = __viaddmax_s32(fp[c], -ge, hp[c]);
                const int32_t d = __dp4a((int)(c < 4 ? w[q].x : w[q].y), 1 << (8 * (c & 3)), dg[q]);
                dg[q] = hp[c] + o;
                const int32_t hh = __vimax3_s32_relu(d, e[q], f);
                const int32_t key = TRACK != kTrackNone ? hh * 8 + (7 - c) : hh;
                if (c & 1) best[q] = __vimax3_s32(best[q], pend[q], key);
                else if (c == R - 1) best[q] = max(best[q], key);
                else pend[q] = key;
                h[q] = hh - o;
                hp[c] = h[q];
                fp[c] = f;
            }
        }
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            oh[q] = h[q];
            oe[q] = e[q];
            if (TRACK == kTrackNone) {
                lkey = max(lkey, best[q]);
            } else {
                const bool up = best[q] > (TRACK == kTrackYRows ? lkey : (lkey | 7));
                lkey = up ? best[q] : lkey;
                lx = up ? (t - lane) * NR + q : lx;
            }
        }
        if (bout != nullptr && t >= 31) {                 // (whole groups: bout has room for them)
            if (lane == 31) {
#pragma unroll
                for (int q = 0; q < NR; q += 2)
                    __stcg(reinterpret_cast<int4*>(bout + (t - 31) * NR + q),
                           make_int4(oh[q], oe[q], oh[q + 1], oe[q + 1]));
            }
            if (j == 31 || t == groups + 30) {
                if (lane == 31) publish(t - 30);
                __syncwarp();
            }
        }
    }
    if (TRACK == kTrackNone) {
        score = __reduce_max_sync(kAll, lkey);
        xpos = ypos = -1;
        return true;
    }
    // the lanes' first cells: larger score, then smaller row, then smaller column
    int32_t b = lkey >> 3, px = lx, py = s.y0 + lane * R + 7 - (lkey & 7);
    for (int d = 16; d >= 1; d >>= 1) {
        const int32_t ob = __shfl_xor_sync(kAll, b, d);
        const int32_t ox = __shfl_xor_sync(kAll, px, d);
        const int32_t oy = __shfl_xor_sync(kAll, py, d);
        if (TRACK == kTrackYRows ? first_max(ob, oy, ox, b, py, px) : first_max(ob, ox, oy, b, px, py)) {
            b = ob;
            px = ox;
            py = oy;
        }
    }
    score = b;
    xpos = b > 0 ? px : -1;
    ypos = b > 0 ? py : -1;
    return true;
}

}  // namespace
}  // namespace cm
