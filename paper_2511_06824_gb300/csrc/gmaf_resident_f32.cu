// FP32 kernels of the resident PCG (gmaf_resident.cuh).
#include "gmaf_resident.cuh"

namespace gmaf {

ResKernel res_kernel_f32(int vec, int rr, bool cs)
{
#define GMAF_RES(V, R)                                              \
    if (vec == V && rr == R) {                                      \
        if (cs) GMAF_RES_KERNEL((k_resident<float, V, R, true>));  \
        GMAF_RES_KERNEL((k_resident<float, V, R, false>));         \
    }
    GMAF_RES(1, 1) GMAF_RES(1, 2) GMAF_RES(1, 4) GMAF_RES(1, 8)
    GMAF_RES(4, 1) GMAF_RES(4, 2) GMAF_RES(4, 4)
#undef GMAF_RES
    return {};
}

}  // namespace gmaf
