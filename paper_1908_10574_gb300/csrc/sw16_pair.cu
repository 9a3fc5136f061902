// The query-pair kernel of all tiles: one launch for the tasks of every register tile and mode
// of a plan too small to fill the chip tile by tile.  The tile is a field of the task; a CTA of
// 16 warps fills an SM whatever its tile.
//
// For plans of up to kMergedTasks tasks per SM and tile.  A launch per tile (sw16_kernel), two at a
// time, leaves SMs idle at the end of each: with the 20 to 48 tiles of a small plan most of the
// chip (all-against-all of 200 proteins 4.7 ms against 1.7 in one launch, of 2,000 in two parts 59
// against 27, ClusterMerge of 3,000 proteins 440 against 91).  Where a tile has enough tasks the
// kernels of one tile are 3 to 7 % faster, as their row loops share no register budget and no
// instruction cache with other tiles'.  The line, measured at one launch / a launch per tile, in
// ms: 4,000 proteins whole (some 45 tiles) 200 / 216, in 2 parts 99.2 / 111, in 4 (fewer lengths
// each) 51.8 / 49.8; 7,000 in 4 parts 160 / 155; a 32nd of 20,000 (two or three tiles) 171 / 160.
#include "sw16_kernel.cuh"

namespace cm {
namespace {

// One task on the CTA's warps.
template <int R, int SEG>
__device__ __forceinline__ void pair_task(const SwArgs& a, const SwTask& T, const int16_t* s_mat)
{
    using G = Geo<R, SEG>;
    constexpr int SPW = SEG == 16 ? 2 : 1;                     // streams per warp
    extern __shared__ __align__(16) uint8_t smem[];
    uint32_t* prof = reinterpret_cast<uint32_t*>(smem);
    const int tid = threadIdx.x, nthreads = blockDim.x, W = nthreads >> 5;
    const int warp = tid >> 5, lane = tid & 31;
    const SwBlock& B = a.blocks[T.block];
    const int32_t* A_ids = a.ids + B.a_ids;
    const int32_t q_lo = A_ids[T.k];
    const int32_t q_hi = T.hi_valid ? A_ids[T.k + 1] : q_lo;
    const int64_t qoff_lo = a.off[q_lo], m_lo = a.off[q_lo + 1] - qoff_lo;
    const int64_t qoff_hi = a.off[q_hi];
    const int64_t m_hi = T.hi_valid ? a.off[q_hi + 1] - qoff_hi : 0;
    const int64_t* srow = a.srows + B.srow;

    // rows of this task split over the CTA's streams at subject boundaries
    const int64_t R0 = srow[T.s0], R1 = srow[T.s1];
    const int i0 = warp * SPW + (SEG == 16 ? lane >> 4 : 0);
    const int32_t st0 = nearest_boundary(srow, T.s0, T.s1, R0 + (R1 - R0) * i0 / (W * SPW));
    const int32_t st1 = nearest_boundary(srow, T.s0, T.s1, R0 + (R1 - R0) * (i0 + 1) / (W * SPW));
    int64_t rows = srow[st1] - srow[st0];
    int64_t nmax = (int64_t)__reduce_max_sync(kFull, (uint32_t)(rows / kRowGroup)) * kRowGroup;
    if (T.npass > 1 && (SEG == 16 || nmax > a.bnd_stride)) {
        if (lane == 0) atomicExch(a.err, 1);      // boundary buffer too small: refuse
        rows = nmax = 0;
    }
    uint2* bnd = a.bnd + ((int64_t)blockIdx.x * W + warp) * a.bnd_stride;
    const int qs = B.swap ? 1 : kAlpha, xs = B.swap ? kAlpha : 1;
    for (int pass = 0; pass < T.npass; ++pass) {
        const int64_t c0 = (int64_t)pass * G::COLS;
        // a thread's column: its two residues against every row residue (+o: the DP keeps
        // H - o as its diagonal input)
        for (int c = tid; c < G::COLS; c += nthreads) {
            const int ql = (c0 + c < m_lo) ? a.db[qoff_lo + c0 + c] : kPadCode;
            const int qh = (c0 + c < m_hi) ? a.db[qoff_hi + c0 + c] : kPadCode;
            const int ln = c / R;
            uint32_t* out = prof + ln * G::LS + (c - ln * R);
            for (int x = 0; x < kAlpha; ++x)
                out[x * G::ROWW] = addend2(ql != kPadCode ? s_mat[ql * qs + x * xs] + a.gap_open : 0,
                                           qh != kPadCode ? s_mat[qh * qs + x * xs] + a.gap_open : 0);
            out[kPadCode * G::ROWW] = 0;          // pads score -o
        }
        __syncthreads();
        if (nmax > 0)
            warp_dp16<R, SEG>(a, B, prof, a.streams + B.stream + srow[st0], rows, nmax, pass, T.npass,
                              bnd, st0, T.k, (B.kind == kTri) ? T.k : B.nb,
                              (B.kind == kTri) ? T.k + 1 : B.nb, T.hi_valid != 0);
        __syncthreads();
    }
}

__global__ void __launch_bounds__(512, 1) sw16_pairs_kernel(const __grid_constant__ SwArgs a)
{
    __shared__ int16_t s_mat[kAlpha * kAlpha];
    __shared__ int s_task[2];
    const int tid = threadIdx.x;
    for (int i = tid; i < kAlpha * kAlpha; i += blockDim.x) s_mat[i] = a.mat[i];
    if (tid == 0) s_task[0] = atomicAdd(a.task_counter, 1);
    __syncthreads();
    for (int it = 0;; ++it) {
        const int ti = s_task[it & 1];
        if (ti >= a.ntasks) break;
        if (tid == 0) s_task[(it + 1) & 1] = atomicAdd(a.task_counter, 1);
        const SwTask& T = a.tasks[ti];
        if (T.mode == kModeSeg16) {
            switch (T.R) {
#define CM_MODE 2
#include "sw16_inst.cuh"
#define CM_CASE(r) case r: pair_task<r, 16>(a, T, s_mat); break;
                CM_R_CASES(CM_CASE)
#undef CM_CASE
#undef CM_MODE
            }
        } else {
            switch (T.R) {
#define CM_MODE 0
#include "sw16_inst.cuh"
#define CM_CASE(r) case r: pair_task<r, 32>(a, T, s_mat); break;
                CM_R_CASES(CM_CASE)
#undef CM_CASE
#undef CM_MODE
            }
        }
        __syncthreads();
    }
}

}  // namespace

cudaError_t launch_sw16_pairs(int W, int grid, int smem, const SwArgs& a, cudaStream_t st)
{
    const cudaError_t e = cudaFuncSetAttribute(
        sw16_pairs_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, sw16_pair_smem(32, kModePair));
    if (e != cudaSuccess) return e;
    sw16_pairs_kernel<<<grid, W * 32, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace cm
