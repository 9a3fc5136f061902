// Instantiations of the int16x2 query-pair kernel for one CTA width (CM_W) and one launch mode
// (CM_MODE: kModePair or kModeSeg16), every register tile width of sw16_inst.cuh.  Each (width, mode) pair is its own
// translation unit so the build runs them in parallel; the including file defines CM_W,
// CM_MODE, CM_LAUNCH and CM_OCC.
#include "sw16_kernel.cuh"
#include "sw16_inst.cuh"

namespace cm {
namespace {

template <int R>
constexpr int inst_smem()
{
    using G = Geo<R, CM_MODE == kModeSeg16 ? 16 : 32>;
    return G::PROF_WORDS * 4 + 2 * G::COLS;
}

template <int R>
cudaError_t inst_launch(int grid, const SwArgs& a, cudaStream_t st)
{
    cudaError_t e = cudaFuncSetAttribute(sw16_kernel<R, CM_W, CM_MODE>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         inst_smem<R>());
    if (e != cudaSuccess) return e;
    sw16_kernel<R, CM_W, CM_MODE><<<grid, CM_W * 32, inst_smem<R>(), st>>>(a);
    return cudaGetLastError();
}

template <int R>
int inst_occ()
{
    if (cudaFuncSetAttribute(sw16_kernel<R, CM_W, CM_MODE>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, inst_smem<R>()) !=
        cudaSuccess)
        return 1;
    int m = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&m, sw16_kernel<R, CM_W, CM_MODE>,
                                                      CM_W * 32, inst_smem<R>()) != cudaSuccess)
        return 1;
    return m;
}

}  // namespace

cudaError_t CM_LAUNCH(int R, int grid, const SwArgs& a, cudaStream_t st)
{
    switch (R) {
#define CM_CASE(r) case r: return inst_launch<r>(grid, a, st);
    CM_R_CASES(CM_CASE)
#undef CM_CASE
    default: return cudaErrorInvalidValue;
    }
}

int CM_OCC(int R)
{
    switch (R) {
#define CM_CASE(r) case r: return inst_occ<r>();
    CM_R_CASES(CM_CASE)
#undef CM_CASE
    default: return 1;
    }
}

}  // namespace cm
