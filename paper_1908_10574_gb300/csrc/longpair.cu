// Alignment cells of pairs whose score may reach 2^28 (both sequences beyond two million
// residues), where strips.cu's position key no longer fits: a whole CTA per pair.  The CTA's LW
// warps run the pair's column passes as a pipeline: warp w takes passes w, w + LW, w + 2 LW, ...;
// pass p reads the boundary column (H - o and E of its left neighbour column for every row) that
// pass p - 1 writes, trailing it by at least 32 row groups (the wavefront of dp32.cuh: four rows
// per step).  The boundary of pass p lives in global slot (p mod LW) of the CTA; a warp
// publishes how many rows of its current pass are written in shared memory (tagged with the
// pass), after a block fence.  Waits only point from pass p to pass p - 1 (never backwards), and
// the warps of a CTA are co-resident, so the pipeline always advances; every wait is still
// bounded (SwArgs::wait_limit polls of ~100 ns) and sets the error flag (2) when it gives up.
// Slot p mod LW is rewritten by pass p + LW, which trails its reader (pass p + 1) by at least
// 32 (LW - 1) row groups through the chain of waits, so a row is never overwritten before it
// has been read.
#include "dp32.cuh"
#include "sw16_kernel.cuh"

namespace cm {
namespace {

constexpr int kLW = 8;                 // warps per CTA (passes in flight)
constexpr int kLR = 8;                 // columns per lane: 256-column passes

__global__ void __launch_bounds__(kLW * 32, 1)
huge_cells_kernel(const __grid_constant__ SwArgs a, const CellJob* __restrict__ jobs, int32_t njobs,
                  int32_t* counter, int32_t* __restrict__ res)
{
    constexpr int COLS = 32 * kLR;
    constexpr int LS = kLR;                                   // dense rows: 2-way conflicts only
    constexpr int ROWW = 32 * LS;
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ int16_t s_mat[kAlpha * kAlpha];
    __shared__ volatile int32_t s_pass[kLW];                 // pass whose boundary is in slot w
    __shared__ volatile int32_t s_prog[kLW];                 // rows of it written so far
    __shared__ int s_job;
    __shared__ int32_t s_best[kLW], s_row[kLW], s_col[kLW];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int32_t* prof = reinterpret_cast<int32_t*>(smem) + (size_t)warp * kProfRows * ROWW;
    uint8_t* qres = smem + (size_t)kLW * kProfRows * ROWW * 4 + (size_t)warp * COLS;
    for (int i = tid; i < kAlpha * kAlpha; i += kLW * 32) s_mat[i] = a.mat[i];
    const int o = a.gap_open, ge = a.gap_extend;
    int2* slots = reinterpret_cast<int2*>(a.bnd + (int64_t)blockIdx.x * kLW * a.bnd_stride);

    for (;;) {
        __syncthreads();
        if (tid == 0) s_job = *reinterpret_cast<volatile int32_t*>(a.err) ? njobs : atomicAdd(counter, 1);
        if (tid < kLW) { s_pass[tid] = -1 - kLW; s_prog[tid] = 0; }
        __syncthreads();
        const int p_job = s_job;
        if (p_job >= njobs) break;
        const CellJob J = jobs[p_job];
        const uint8_t* ra = a.db + a.off[J.a];
        const uint8_t* cb = a.db + a.off[J.b];
        int64_t m = J.m;
        const int64_t n = J.n;
        const int npass = (int)((n + COLS - 1) / COLS);
        if (m > a.bnd_stride || m >= ((int64_t)1 << 30)) {     // boundary slots too short
            if (tid == 0) atomicExch(a.err, 1);
            m = 0;
        }
        int32_t gbest = 0, grow = -1, gcol = -1;                // this warp's passes
        bool gave_up = false;
        for (int pass = warp; pass < npass && m > 0 && !gave_up; pass += kLW) {
            const int64_t c0 = (int64_t)pass * COLS;
            // this warp's slot takes pass `pass`: reset its progress, then publish the pass
            if (lane == 0) {
                s_prog[warp] = 0;
                __threadfence_block();
                s_pass[warp] = pass;
            }
            for (int c = lane; c < COLS; c += 32) {
                const int64_t cc = c0 + c;
                qres[c] = (cc < n) ? (J.reverse ? cb[n - 1 - cc] : cb[cc]) : kPadCode;
            }
            __syncwarp();
            for (int i = lane; i < kProfRows * COLS; i += 32) {
                const int x = i / COLS, c = i - x * COLS;
                const int ln = c / kLR, k = c - ln * kLR;
                const int q = qres[c];
                int32_t s = -1024;                // +o: the DP keeps H - o as its diagonal input
                if (x != kPadCode && q != kPadCode)
                    s = s_mat[x * kAlpha + q] + o;
                prof[x * ROWW + ln * LS + k] = s;
            }
            __syncwarp();
            const int src = (warp + kLW - 1) % kLW;               // slot of pass - 1
            // rows [0, need) of pass - 1's boundary written: lane 0 polls, bounded
            auto wait = [&](int32_t need) {
                int ok = 1;
                if (lane == 0) {
                    int spins = 0;
                    for (;;) {
                        const int32_t ps = s_pass[src];
                        if (ps > pass - 1 || (ps == pass - 1 && s_prog[src] >= need)) break;
                        if (++spins > a.wait_limit) { ok = 0; break; }
                        __nanosleep(100);
                    }
                    __threadfence_block();
                }
                __syncwarp();                     // orders the other lanes' reads too
                return __shfl_sync(0xffffffffu, ok, 0) != 0;
            };
            auto publish = [&](int32_t rows) {
                __threadfence_block();
                s_prog[warp] = rows;
            };
            D32Best r;
            if (!dp32_pass<kLR, LS>(prof + lane * LS, ra, m, J.reverse != 0, o, ge,
                                           pass > 0 ? slots + (int64_t)src * a.bnd_stride : nullptr,
                                           pass + 1 < npass ? slots + (int64_t)warp * a.bnd_stride : nullptr,
                                           (int32_t)c0 + lane * kLR, wait, publish, r)) {
                if (lane == 0) atomicExch(a.err, 2);
                gave_up = true;
                break;
            }
            if (first_max(r.b, r.r, r.c, gbest, grow, gcol)) { gbest = r.b; grow = r.r; gcol = r.c; }
        }
        // combine the warps' passes: largest score, then smallest row, then smallest column
        if (lane == 0) { s_best[warp] = gbest; s_row[warp] = grow; s_col[warp] = gcol; }
        __syncthreads();
        if (tid == 0) {
            int32_t b = 0, rw = -1, cl = -1;
            for (int w = 0; w < kLW; ++w)
                if (first_max(s_best[w], s_row[w], s_col[w], b, rw, cl)) { b = s_best[w]; rw = s_row[w]; cl = s_col[w]; }
            res[3 * (int64_t)p_job] = b;
            res[3 * (int64_t)p_job + 1] = b > 0 ? rw : -1;
            res[3 * (int64_t)p_job + 2] = b > 0 ? cl : -1;
        }
    }
}

constexpr int long_smem_bytes() { return kLW * (kProfRows * 32 * kLR * 4 + 32 * kLR); }

}  // namespace

cudaError_t launch_huge_cells(int grid, const SwArgs& a, const CellJob* jobs, int32_t njobs,
                              int32_t* counter, int32_t* res, cudaStream_t st)
{
    if (njobs == 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(huge_cells_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         long_smem_bytes());
    if (e != cudaSuccess) return e;
    huge_cells_kernel<<<grid, kLW * 32, long_smem_bytes(), st>>>(a, jobs, njobs, counter, res);
    return cudaGetLastError();
}

}  // namespace cm
