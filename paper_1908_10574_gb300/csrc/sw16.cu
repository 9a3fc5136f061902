// Launchers of the Smith-Waterman kernels (templates in sw16_kernel.cuh); the int16x2
// query-pair kernel by CTA width and the int32 rescoring kernel.
#include "sw16_kernel.cuh"

namespace cm {

#define CM_DECL(w, m)                                                                     \
    cudaError_t launch_sw16_w##w##_m##m(int R, int grid, const SwArgs& a, cudaStream_t st); \
    int sw16_occ_w##w##_m##m(int R);
CM_DECL(4, 0) CM_DECL(4, 2)
CM_DECL(8, 0) CM_DECL(8, 2)
CM_DECL(16, 0) CM_DECL(16, 2)
#undef CM_DECL

int sw16_ctas_per_sm(int R, int W, int mode)
{
#define CM_OCC_CASE(w)                                                                   \
    case w:                                                                              \
        return mode == kModePair ? sw16_occ_w##w##_m0(R) : sw16_occ_w##w##_m2(R);
    switch (W) {
    CM_OCC_CASE(4)
    CM_OCC_CASE(8)
    CM_OCC_CASE(16)
    default: return 1;
    }
#undef CM_OCC_CASE
}

int sw32_ctas_per_sm()
{
    const int smem = sw32_smem_bytes(16);
    if (cudaFuncSetAttribute(sw32_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             smem) != cudaSuccess)
        return 1;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, sw32_kernel<16>, 32, smem) !=
        cudaSuccess)
        return 1;
    return n;
}

cudaError_t launch_sw16(int R, int W, int mode, int grid, const SwArgs& a, cudaStream_t st)
{
    if (mode != kModePair && mode != kModeSeg16) return cudaErrorInvalidValue;
#define CM_LAUNCH_CASE(w)                                                                \
    case w:                                                                              \
        return mode == kModePair ? launch_sw16_w##w##_m0(R, grid, a, st)                 \
                                 : launch_sw16_w##w##_m2(R, grid, a, st);
    switch (W) {
    CM_LAUNCH_CASE(4)
    CM_LAUNCH_CASE(8)
    CM_LAUNCH_CASE(16)
    default: return cudaErrorInvalidValue;
    }
#undef CM_LAUNCH_CASE
}

int sw32_smem_bytes(int R)
{
    const int LS = lane_stride(R);
    return kProfRows * 32 * LS * 4 + 32 * R;
}

cudaError_t launch_sw32(int R, int grid, const SwArgs& a, const PairRef* pr, int32_t npairs,
                        int32_t* counter, cudaStream_t st)
{
    if (R != 16) return cudaErrorInvalidValue;
    const int smem = sw32_smem_bytes(16);
    cudaError_t e = cudaFuncSetAttribute(sw32_kernel<16>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    sw32_kernel<16><<<grid, 32, smem, st>>>(a, pr, npairs, counter);
    return cudaGetLastError();
}

}  // namespace cm
