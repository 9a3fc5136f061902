// Launchers of the query-pair kernel of one tile, by CTA width and mode.
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

}  // namespace cm
