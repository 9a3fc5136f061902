// The two int32 passes over lists of pairs, by wave32.cuh's wavefront:
//   alignment cells: per job the optimum and its first row-major cell.  Rows stream the job's
//     first sequence a[0..m) (reversed when J.reverse), the strips hold its second one b[0..n)
//     (reversed likewise);
//   rescoring of the pairs flagged by the int16 pass: rows stream the subject, the strips hold
//     the query.
//
// A unit is one strip of one job; warps take units from a queue, longest job first, and strip s
// trails strip s - 1 by 32 row groups over the job's boundary column (progress.cuh), so every
// strip of a long pair runs at once.  A strip passes the best so far on with its last group;
// the last strip writes the job's result.
// Bound: the ALU pipe, 3.5 half-rate DPX operations per cell and the dot product's share.
// Measured on one GB300, 20,000 pairs of related proteins (1.0e10 cells in both directions):
// 5.4 ms (1.9 Tcells/s, the ALU pipe 73 % busy); 14.4 ms for a warp per job with an int32
// profile (38 KB: five warps on an SM) and four more operations per cell to track the position,
// plus whole CTAs for the long jobs.  Two rows per step instead of four: the same time (less
// wavefront to fill, more overhead per row).  Rescoring of 24 pairs of 8,000-12,000 residues
// (2.4e9 cells): 2.3 ms; 9.8 ms on CTAs of eight warps that pipelined one pair's passes.
#include "progress.cuh"
#include "sw16_kernel.cuh"
#include "wave32.cuh"

namespace cm {
namespace {

constexpr int kCellWarps = 10;                   // warps per CTA, two CTAs per SM

struct CellUnitArgs {
    WaveStrip s;
    const int32_t* done_in;
    int32_t* done_out;
    int32_t* err;
    int32_t limit;
};

template <int R, int TRACK>
__device__ __noinline__ bool unit_strip(const CellUnitArgs& u, int32_t& b, int32_t& row, int32_t& col)
{
    WaveStrip s = u.s;
    extern __shared__ uint2 cell_prof[];
    s.prof = cell_prof + (threadIdx.x >> 5) * kWaveProf;
    const int32_t* in = u.done_in;
    int32_t* out = u.done_out;
    auto wait = [&](int32_t need) { return wait_groups(in, need, u.err, u.limit); };
    // the last group is published with the strip's result, by the caller
    const int32_t groups = (s.xn + kWaveRows - 1) / kWaveRows;
    auto publish = [&](int32_t g) { if (g < groups) publish_groups(out, g); };
    return wave_strip<R, TRACK>(s, wait, publish, b, row, col);
}

template <bool CELLS>
__global__ void __launch_bounds__(32 * kCellWarps, 2)
strips_kernel(const __grid_constant__ SwArgs a, const CellJob* __restrict__ jobs,
              const PairRef* __restrict__ refs, int32_t* counter, int32_t* res)
{
    extern __shared__ uint2 cell_prof[];
    __shared__ int8_t s_mat[kAlpha * kAlpha];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint2* prof = cell_prof + warp * kWaveProf;
    for (int i = threadIdx.x; i < kAlpha * kAlpha; i += blockDim.x) s_mat[i] = (int8_t)a.mat[i];
    __syncthreads();
    // the first, longest units go one to an SM: the warps of a CTA do not queue all at once
    __nanosleep(1000 * warp);
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(counter, 1);
        t = __shfl_sync(kFull, t, 0);
        if (t >= a.ncells) break;
        const CellUnit U = a.cell_units[t];
        CellJob J;
        int64_t slot = 0;
        int ys = 1, xs = kAlpha;                   // score: mat[row residue][column residue]
        if (CELLS) {
            J = jobs[U.job];
        } else {
            const PairRef P = refs[U.job];
            J = CellJob{P.x, P.q, (int32_t)(a.off[P.x + 1] - a.off[P.x]),
                        (int32_t)(a.off[P.q + 1] - a.off[P.q]), 0, 0};
            slot = P.slot;
            if (!P.swap) { ys = kAlpha; xs = 1; }  // mat[query][subject]
        }
        const uint8_t* ra = a.db + a.off[J.a];
        const uint8_t* cb = a.db + a.off[J.b];
        const int32_t strips = cell_strips(J.m, J.n), R = wave_R(J.n);
        const bool last = U.strip + 1 == strips;
        CellUnitArgs u;
        // (a reversed prefix a[0..m) read back to front)
        u.s.x = ra;
        u.s.xn = J.n > 0 ? J.m : 0;
        u.s.reverse = J.reverse != 0;
        u.s.o = a.gap_open;
        u.s.ge = a.gap_extend;
        int2* bnd = reinterpret_cast<int2*>(a.bnd) + U.bnd_row;
        u.s.bin = U.strip > 0 ? bnd : nullptr;
        u.s.bout = last ? nullptr : bnd;
        u.s.y0 = U.strip * 32 * R;
        u.done_in = a.progress + t - 1;
        u.done_out = a.progress + t;
        u.err = a.err;
        u.limit = U.limit;
        __syncwarp();
        wave_profile(prof, cb, J.n, J.reverse != 0, u.s.y0, R, s_mat, ys, xs, kAlpha);
        __syncwarp();
        int32_t b = 0, row = -1, col = -1;
        bool ok = true;
        switch (R) {
#define CM_CASE(r) case r: ok = unit_strip<r, CELLS ? kTrackXRows : kTrackNone>(u, b, row, col); break;
            CM_CASE(1) CM_CASE(2) CM_CASE(3) CM_CASE(4) CM_CASE(5) CM_CASE(6) CM_CASE(7) CM_CASE(8)
#undef CM_CASE
        }
        if (!ok) {
            if (lane == 0) atomicExch(a.err, 2);
            continue;
        }
        // lane 31 wrote the boundary column, so it also publishes the last group
        if (lane == 31) {
            if (U.strip > 0) {                     // all of it was read: its result is there too
                const int4 p = __ldcg(a.cell_best + t - 1);
                if (!CELLS) b = max(b, p.x);
                else if (first_max(p.x, p.y, p.z, b, row, col)) { b = p.x; row = p.y; col = p.z; }
            }
            if (last && !CELLS) {
                a.out[slot] = b;
            } else if (last) {
                res[3 * (int64_t)U.job] = b;
                res[3 * (int64_t)U.job + 1] = b > 0 ? row : -1;
                res[3 * (int64_t)U.job + 2] = b > 0 ? col : -1;
            } else {
                __stcg(a.cell_best + t, make_int4(b, row, col, 0));
                publish_groups(a.progress + t, (u.s.xn + kWaveRows - 1) / kWaveRows);
            }
        }
        __syncwarp();
    }
}

template <bool CELLS>
cudaError_t launch(const SwArgs& a, const CellJob* jobs, const PairRef* refs, int32_t* counter,
                   int32_t* res, cudaStream_t st)
{
    constexpr int smem = kWaveProf * (int)sizeof(uint2);              // per warp
    const cudaError_t e = cudaFuncSetAttribute(strips_kernel<CELLS>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               kCellWarps * smem);
    if (e != cudaSuccess) return e;
    const int grid = std::min(a.ncells, 2 * a.num_sms);
    const int warps = std::min(kCellWarps, (a.ncells + grid - 1) / grid);
    strips_kernel<CELLS><<<grid, 32 * warps, warps * smem, st>>>(a, jobs, refs, counter, res);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_cells_wf(int, const SwArgs& a, const CellJob* jobs, int32_t njobs,
                            int32_t* counter, int32_t* res, cudaStream_t st)
{
    return njobs == 0 ? cudaSuccess : launch<true>(a, jobs, nullptr, counter, res, st);
}

cudaError_t launch_long_cells(int grid, const SwArgs& a, const CellJob* jobs, int32_t njobs,
                              int32_t* counter, int32_t* res, cudaStream_t st)
{
    if (njobs == 0) return cudaSuccess;
    return a.cell_units ? launch<true>(a, jobs, nullptr, counter, res, st)
                        : launch_huge_cells(grid, a, jobs, njobs, counter, res, st);
}

cudaError_t launch_sw32(int, int, const SwArgs& a, const PairRef* pr, int32_t npairs,
                        int32_t* counter, cudaStream_t st)
{
    return npairs == 0 ? cudaSuccess : launch<false>(a, nullptr, pr, counter, nullptr, st);
}

cudaError_t launch_long_sw32(int, const SwArgs& a, const PairRef* pr, int32_t npairs,
                             int32_t* counter, cudaStream_t st)
{
    return npairs == 0 ? cudaSuccess : launch<false>(a, nullptr, pr, counter, nullptr, st);
}

}  // namespace cm
