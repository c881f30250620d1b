// Tensor memory: 256 KB an SM that the matrix instructions would accumulate in; here a second
// register file.  A warp reaches a quarter of its 128 lanes, so each of 512 threads has 128 words of
// its own.  The instructions are the whole warp's.
#pragma once

#include "gmaf_internal.cuh"
#include "gmaf_pcg_kernels.cuh"

namespace gmaf {

constexpr int kTmCols = 512;                // columns (32-bit words a lane): all

__device__ __forceinline__ void tm_alloc(unsigned *slot)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(slot)),
                 "n"(kTmCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void tm_free(unsigned base)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(base), "n"(kTmCols) : "memory");
}
// 16 bytes of this thread; valid after tm_wait_ld, which names every word loaded so that no
// use moves before it.
struct TmRow {
    unsigned w[4];
};
__device__ __forceinline__ void tm_ld(unsigned at, TmRow &x)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(x.w[0]), "=r"(x.w[1]), "=r"(x.w[2]), "=r"(x.w[3])
                 : "r"(at));
}
template <int N>
__device__ __forceinline__ void tm_wait_ld(TmRow (&x)[N])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int k = 0; k < N; ++k)
        asm volatile("" : "+r"(x[k].w[0]), "+r"(x[k].w[1]), "+r"(x[k].w[2]), "+r"(x[k].w[3])::"memory");
}
__device__ __forceinline__ void tm_get(const TmRow &t, float (&x)[4])
{
#pragma unroll
    for (int e = 0; e < 4; ++e) x[e] = __uint_as_float(t.w[e]);
}
__device__ __forceinline__ void tm_get(const TmRow &t, double (&x)[2])
{
#pragma unroll
    for (int e = 0; e < 2; ++e) x[e] = __hiloint2double((int)t.w[2 * e + 1], (int)t.w[2 * e]);
}
__device__ __forceinline__ void tm_st(unsigned at, const float (&x)[4])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(at), "f"(x[0]), "f"(x[1]),
                 "f"(x[2]), "f"(x[3])
                 : "memory");
}
__device__ __forceinline__ void tm_st(unsigned at, const double (&x)[2])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(at),
                 "r"(__double2loint(x[0])), "r"(__double2hiint(x[0])), "r"(__double2loint(x[1])),
                 "r"(__double2hiint(x[1]))
                 : "memory");
}
__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }

}  // namespace gmaf
