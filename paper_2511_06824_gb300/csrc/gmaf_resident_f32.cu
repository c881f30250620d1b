// FP32 kernels of the resident PCG (gmaf_resident.cuh).
#include "gmaf_resident.cuh"

namespace gmaf {

const void *res_kernel_f32(int vec, int rr, bool cs)
{
#define GMAF_RES(V, R)                                                             \
    if (vec == V && rr == R)                                                       \
        return cs ? (const void *)k_resident<float, V, R, true>                    \
                  : (const void *)k_resident<float, V, R, false>;
    GMAF_RES(1, 1) GMAF_RES(1, 2) GMAF_RES(1, 4) GMAF_RES(1, 8)
    GMAF_RES(4, 1) GMAF_RES(4, 2) GMAF_RES(4, 4)
#undef GMAF_RES
    return nullptr;
}

}  // namespace gmaf
