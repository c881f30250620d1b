// The resident PCG for the largest systems it takes (FP32 inside FP64 refinement): its
// vectors in shared and tensor memory.
//
// Runs of 16 rows: r and the product live in the SM's tensor memory (64 words a thread each),
// u stays in shared memory, and the
// coefficients and x are streamed from L2, one group of rows ahead of the one worked on.
// The diagonal is rebuilt from the couplings, as in the phase A of gmaf_drec.cu, to save
// its traffic; a matrix whose diagonal is another one is left to the phase kernels.
//
// On 9 conditions of 1024 x 512 cells an iteration takes 37 to 39 us (A 16.8, B 21.2), with two
// exchanges of 1.5 us; the phase kernels take 68.3.  The coefficients and x are 175 MB of it from
// L2, where 321 MB are counted: the rest is spills (96 registers a thread) and polling.  On 9 of
// 700 x 300 it is 33.3 us against 56.7.
#include "gmaf_resident.cuh"
#include "gmaf_tmem.cuh"

namespace gmaf {

__device__ __forceinline__ void tm_ld(unsigned at, float (&x)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n"
                 : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3])
                 : "r"(at));
}
// Waits for this thread's loads; the values are tied to it so that no use moves before it.
__device__ __forceinline__ void tm_wait_ld(float (&x)[4])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" : "+f"(x[0]), "+f"(x[1]), "+f"(x[2]), "+f"(x[3])::"memory");
}
__device__ __forceinline__ void tm_wait_ld(float (&x)[4], float (&y)[4])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                 : "+f"(x[0]), "+f"(x[1]), "+f"(x[2]), "+f"(x[3]), "+f"(y[0]), "+f"(y[1]), "+f"(y[2]), "+f"(y[3])::"memory");
}
// As res_iterate (whose comments hold here), for runs of kTmRows rows.  tmem: the block's base.
__device__ __forceinline__ unsigned res_iterate_tm(const ResParams<float> &q, ResShared<float> &sh,
                                                   unsigned ep, unsigned tmem)
{
    using T = float;
    constexpr int VEC = 4, RR = kTmRows, G = 2;      // G: rows of a group
    using V = Vec<T, VEC>;
    constexpr int S = kResThreads * VEC, NS = kResSegs;
    extern __shared__ __align__(16) unsigned char g_res_smem[];
    const int nth = q.nth, nz = q.nz, TC = q.threads, all = TC + 32;
    int tid;
    asm volatile("mov.u32 %0, %%tid.x;\n" : "=r"(tid));
    const int lane = tid & 31, wid = tid >> 5;
    const int cond = blockIdx.x / q.bpc, bc = blockIdx.x - cond * q.bpc;
    const int j0 = (int)((long long)bc * nz / q.bpc), j1 = (int)((long long)(bc + 1) * nz / q.bpc);
    const int R = j1 - j0;
    const bool assor = q.precond == 1;

    // ---- this thread's columns and rows
    const int run = tid / q.P, cg = tid - run * q.P, c = cg * VEC;
    const int lr0 = run * RR;                               // first local row
    int nr = R - lr0;
    nr = cg >= q.ncg || nr < 0 ? 0 : (nr > RR ? RR : nr);
    const bool act = nr > 0;
    const bool top = act && lr0 + nr == R;
    const bool hasS = act && run == 0 && j0 > 0, hasN = top && j1 < nz;    // a block below, above
    const bool segw = (cg & 31) == 0, sege = (cg & 31) == 31 || cg == q.ncg - 1;
    const bool atw = cg == 0, ate = cg == q.ncg - 1;
    const bool last = top && j1 == nz;                      // this run ends at row nz - 1
    // (whatever fits on the SMs has less than 2^32 cells)
    const unsigned off = (unsigned)cond * (unsigned)q.n + (unsigned)((j0 + lr0) * nth + c);
    const unsigned coff = (unsigned)q.cslot[cond] * (unsigned)q.n + (unsigned)((j0 + lr0) * nth + c);

    // ---- shared memory: private fields (u, coefficients, r), then rows and edges
    T *const sm = reinterpret_cast<T *>(g_res_smem);
    T *const P = sm + tid * VEC;                            // u: P[rr * S]
    T *const HU = reinterpret_cast<T *>(g_res_smem + q.o_rows);   // [2][nth] u on the halo rows
    T *const HR = HU + 2 * nth;                             // [2][nth] r on the halo rows
    T *const HI = HR + 2 * nth;                             // [2][nth] omega/D on the halo rows
    T *const HE = HI + 2 * nth;                             // [nth] aE on the north halo row
    T *const YR = HE + nth;                                 // [nrr][nth] y south of each run
    T *const WR = YR + q.nrr * nth;                         // [nrr - 1][nth] w north of each run but the last
    // edges of a row's segments of 32 threads, [rows + 1][NS]: last y, last aE; first w
    T *const edge = reinterpret_cast<T *>(g_res_smem + q.o_edge);
    const int er = (q.rows + 1) * NS;
    T *const EY = edge + lr0 * NS + (cg >> 5);
    T *const EYl = edge + lr0 * NS + (atw ? (q.ncg - 1) >> 5 : (cg >> 5) - 1);     // west segment
    T *const EWr = edge + 2 * er + lr0 * NS + (ate ? 0 : (cg >> 5) + 1);           // east segment
    // y of column 0 and w of column nth - 1: [rows + 1][2] behind them
    T *const EC = edge + 3 * er + 2 * lr0;
    // u of the rows beyond the run and of the threads beyond the warp
    const T *const pS = !act ? P : run == 0 ? HU + c : P - q.P * VEC + (RR - 1) * S;
    const T *const pN = !act ? P : top ? HU + nth + c : P + q.P * VEC;
    const T *const pW = sm + (run * q.P + (atw ? q.ncg - 1 : cg - 1)) * VEC + VEC - 1;
    const T *const pE = sm + (run * q.P + (ate ? 0 : cg + 1)) * VEC;
    T *const pX = q.p + off;
    // (a whole warp's rows of its lane quarter; 128 columns a warp)
    const unsigned tv = tmem + ((unsigned)(wid & 3) << 21) + (unsigned)(wid >> 2) * 128u, tr = tv + 4 * RR;

    // coefficients of row rr (zero beyond the block's rows)
    const int most = nr > 0 ? nr - 1 : 0;
    const unsigned cat = act ? coff : (unsigned)q.cslot[cond] * (unsigned)q.n;
    auto coef = [&](const T *g, int rr, T(&x)[VEC]) {
        V::ldrw(g + (cat + (unsigned)(min(rr, most) * nth)), x);
#pragma unroll
        for (int e = 0; e < VEC; ++e) x[e] = rr < nr ? x[e] : T(0);
    };
    T *const PI = reinterpret_cast<T *>(g_res_smem + q.o_x) + tid * VEC;    // omega/D of the first q.ri rows
    auto get_I = [&](int rr, T(&x)[VEC]) {
        if (rr < q.ri)
            V::ldrw(PI + rr * S, x);
        else
            coef(q.invD, rr, x);
    };
    unsigned long long *const halo = q.halo + (size_t)blockIdx.x * 4 * q.halo_row + c;
    T aS0[VEC], hS[VEC], hN[VEC];
#pragma unroll
    for (int e = 0; e < VEC; ++e) aS0[e] = hS[e] = hN[e] = T(0);
    if (j0 + lr0 > 0 && act) V::ldrw(q.aN + coff - nth, aS0);
    auto fetch = [&](int s, int n) {
        bool ok = true;
        if (hasS) ok = ll_get<VEC>(halo + (s - 4) * q.halo_row, hS, ep, q.polls);
        if (hasN) ok = ll_get<VEC>(halo + (n + 4) * q.halo_row, hN, ep, q.polls) && ok;
        if (!ok) sh.halo_failed = 1;
        __syncwarp();
    };

    // b = r64 / ||r64||, x = 0
    {
        const double unit = sh.unit;
        ++ep;
#pragma unroll 1
        for (int rr = 0; rr < RR; ++rr) {
            T r[VEC], x[VEC];
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                r[e] = rr < nr ? (T)(q.r64[off + (size_t)rr * nth + e] * unit) : T(0);
                x[e] = T(0);
            }
            __syncwarp();
            tm_st(tr + 4 * rr, r);
            tm_st(tv + 4 * rr, x);
            if (rr < nr) V::st(pX + (size_t)rr * nth, x);
            if (hasS && rr == 0) ll_put<VEC>(halo, r, ep);
            if (hasN && rr == nr - 1) ll_put<VEC>(halo + q.halo_row, r, ep);
        }
        tm_wait_st();
        fetch(1, 0);
    }

    bool init = true;
    while (!sh.done) {
        // ------------------------------------------------ B: r -= alpha v; z = M^-1 r
        const T alpha = (T)sh.alpha;
        ResAcc<T> arz, arr;
        ++ep;
        T yN[VEC];
#pragma unroll
        for (int e = 0; e < VEC; ++e) yN[e] = T(0);
#pragma unroll 1
        for (int r0 = 0; r0 < RR; r0 += 4) {
            T od[4][VEC], v[4][VEC], r[4][VEC];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                tm_ld(tv + 4 * (r0 + k), v[k]);
                tm_ld(tr + 4 * (r0 + k), r[k]);
                get_I(r0 + k, od[k]);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) tm_wait_ld(v[k], r[k]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int rr = r0 + k;
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    r[k][e] -= alpha * v[k][e];
                    v[k][e] = r[k][e] * od[k][e];
                }
                tm_st(tr + 4 * rr, r[k]);
                tm_st(tv + 4 * rr, v[k]);
                if (rr == RR - 1 && act && !top) V::st(YR + (run + 1) * nth + c, v[k]);
                if (sege && rr < nr) EY[rr * NS] = v[k][VEC - 1];
                if (atw && rr < nr) EC[2 * rr] = v[k][0];
                __syncwarp();
            }
        }
        if (hasS) {
            T h[VEC], od[VEC];
            V::ldrw(HR + c, h);
            V::ldrw(HI + c, od);
#pragma unroll
            for (int e = 0; e < VEC; ++e) h[e] = init ? hS[e] : h[e] - alpha * hS[e];
            V::st(HR + c, h);
#pragma unroll
            for (int e = 0; e < VEC; ++e) h[e] *= od[e];
            V::st(YR + c, h);
        }
        if (hasN) {
            T h[VEC], od[VEC];
            V::ldrw(HR + nth + c, h);
            V::ldrw(HI + nth + c, od);
#pragma unroll
            for (int e = 0; e < VEC; ++e) h[e] = init ? hN[e] : h[e] - alpha * hN[e];
            V::st(HR + nth + c, h);
#pragma unroll
            for (int e = 0; e < VEC; ++e) yN[e] = h[e] * od[e];
            if (sege) EY[nr * NS] = yN[VEC - 1];
            if (atw) EC[2 * nr] = yN[0];
        }
        __syncwarp();
        tm_wait_st();
        if (assor) {
            bar_sync_n(1, TC);
            // first sweep: w = y + omega/D (lower couplings of y)
            T yp[VEC], nS[VEC], wN[VEC];
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                yp[e] = wN[e] = T(0);
                nS[e] = aS0[e];
            }
            if (act) V::ldrw(YR + run * nth + c, yp);
            T fe[G][VEC], fn[G][VEC], fi[G][VEC];
#pragma unroll
            for (int k = 0; k < G; ++k) {
                coef(q.aE, k, fe[k]);
                coef(q.aN, k, fn[k]);
                get_I(k, fi[k]);
            }
#pragma unroll 1
            for (int r0 = 0; r0 < RR; r0 += G) {
                T ev[G][VEC], nv[G][VEC], od[G][VEC], y[G][VEC];
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    tm_ld(tv + 4 * (r0 + k), y[k]);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        ev[k][e] = fe[k][e];
                        nv[k][e] = fn[k][e];
                        od[k][e] = fi[k][e];
                    }
                }
                if (r0 + G < RR) {
#pragma unroll
                    for (int k = 0; k < G; ++k) {
                        coef(q.aE, r0 + G + k, fe[k]);
                        coef(q.aN, r0 + G + k, fn[k]);
                        get_I(r0 + G + k, fi[k]);
                    }
                }
                tm_wait_ld(y[0], y[1]);
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    const int rr = r0 + k;
                    const bool in = rr < nr;
                    T w[VEC];
                    T yW = __shfl_up_sync(0xffffffffu, y[k][VEC - 1], 1);
                    T aW = __shfl_up_sync(0xffffffffu, ev[k][VEC - 1], 1);
                    if (segw) {
                        yW = in && !atw ? EYl[rr * NS] : T(0);
                        aW = in && !atw ? EYl[er + rr * NS] : T(0);
                    }
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        T sum = nS[e] * yp[e];
                        sum += (e > 0 ? ev[k][e - 1] : aW) * (e > 0 ? y[k][e - 1] : yW);
                        if (e == VEC - 1 && ate && in) sum += ev[k][e] * EC[2 * rr];
                        w[e] = y[k][e] + od[k][e] * sum;
                    }
                    if (rr == 0 && act && run > 0) V::st(WR + (run - 1) * nth + c, w);
                    if (segw && in) EY[2 * er + rr * NS] = w[0];
                    if (ate && in) EC[2 * rr + 1] = w[VEC - 1];
                    __syncwarp();
                    tm_st(tv + 4 * rr, w);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        yp[e] = in ? y[k][e] : yp[e];
                        nS[e] = in ? nv[k][e] : nS[e];
                    }
                }
            }
            // w on the row above the block, for z of its last row
            {
                T ev[VEC];
#pragma unroll
                for (int e = 0; e < VEC; ++e) ev[e] = T(0);
                if (hasN) V::ldrw(HE + c, ev);
                T yW = __shfl_up_sync(0xffffffffu, yN[VEC - 1], 1);
                T aW = __shfl_up_sync(0xffffffffu, ev[VEC - 1], 1);
                if (hasN) {
                    T od[VEC];
                    V::ldrw(HI + nth + c, od);
                    if (segw && !atw) {
                        yW = EYl[nr * NS];
                        aW = EYl[er + nr * NS];
                    }
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        T sum = nS[e] * yp[e];
                        if (e > 0)
                            sum += ev[e - 1] * yN[e - 1];
                        else if (!atw)
                            sum += aW * yW;
                        if (e == VEC - 1 && ate) sum += ev[e] * EC[2 * nr];
                        wN[e] = yN[e] + od[e] * sum;
                    }
                }
                __syncwarp();
            }
            tm_wait_st();
            bar_sync_n(1, TC);
            // second sweep: z = w + omega/D (upper couplings of w)
            if (act && !top) V::ldrw(WR + run * nth + c, wN);
#pragma unroll
            for (int k = 0; k < G; ++k) {
                coef(q.aE, RR - 1 - k, fe[k]);
                coef(q.aN, RR - 1 - k, fn[k]);
                get_I(RR - 1 - k, fi[k]);
            }
#pragma unroll 1
            for (int r0 = RR - 1; r0 >= 0; r0 -= G) {
                T ev[G][VEC], nv[G][VEC], od[G][VEC], w[G][VEC], r[G][VEC];
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    tm_ld(tv + 4 * (r0 - k), w[k]);
                    tm_ld(tr + 4 * (r0 - k), r[k]);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        ev[k][e] = fe[k][e];
                        nv[k][e] = fn[k][e];
                        od[k][e] = fi[k][e];
                    }
                }
                if (r0 - G >= 0) {
#pragma unroll
                    for (int k = 0; k < G; ++k) {
                        coef(q.aE, r0 - G - k, fe[k]);
                        coef(q.aN, r0 - G - k, fn[k]);
                        get_I(r0 - G - k, fi[k]);
                    }
                }
#pragma unroll
                for (int k = 0; k < G; ++k) tm_wait_ld(w[k], r[k]);
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    const int rr = r0 - k;
                    const bool in = rr < nr, north = !(last && rr == nr - 1);
                    T z[VEC];
                    T wE = __shfl_down_sync(0xffffffffu, w[k][0], 1);
                    if (sege) wE = in && !ate ? EWr[rr * NS] : T(0);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        T sum = north ? nv[k][e] * wN[e] : T(0);
                        sum += ev[k][e] * (e < VEC - 1 ? w[k][e + 1] : wE);
                        if (e == 0 && atw && in) sum += EYl[er + rr * NS] * EC[2 * rr + 1];
                        z[e] = w[k][e] + od[k][e] * sum;
                    }
#pragma unroll
                    for (int e = 0; e < VEC; ++e) wN[e] = in ? w[k][e] : wN[e];
                    if (hasS && rr == 0) ll_put<VEC>(halo + 2 * q.halo_row, z, ep);
                    if (hasN && rr == nr - 1) ll_put<VEC>(halo + 3 * q.halo_row, z, ep);
                    __syncwarp();
                    tm_st(tv + 4 * rr, z);
                    arz.add(r[k], z);
                    arr.add(r[k], r[k]);
                }
            }
            tm_wait_st();
        } else {
#pragma unroll 1
            for (int rr = 0; rr < RR; ++rr) {
                T r[VEC], z[VEC];
                tm_ld(tr + 4 * rr, r);
                tm_ld(tv + 4 * rr, z);
                tm_wait_ld(r, z);
                if (hasS && rr == 0) ll_put<VEC>(halo + 2 * q.halo_row, z, ep);
                if (hasN && rr == nr - 1) ll_put<VEC>(halo + 3 * q.halo_row, z, ep);
                __syncwarp();
                arz.add(r, z);
                arr.add(r, r);
            }
        }
        {
            const ResSum<T> x[2] = {arz.value(), arr.value()};
            ResTerm<T> t[2];
            res_warp_sums<2>(x, t);
            if (lane == 0) {
                sh.part[0][wid] = t[0];
                sh.part[1][wid] = t[1];
            }
            bar_sync_n(2, all);
        }
        // x += alpha u, and z on the neighbours' rows, while the sums travel
        if (!init) {
#pragma unroll 4
            for (int rr = 0; rr < RR; ++rr) {
                if (rr >= nr) break;
                T x[VEC], u[VEC];
                V::ldrw(pX + (size_t)rr * nth, x);
                V::ldrw(P + rr * S, u);
#pragma unroll
                for (int e = 0; e < VEC; ++e) x[e] += alpha * u[e];
                V::st(pX + (size_t)rr * nth, x);
            }
        }
        fetch(3, 2);
        bar_sync_n(2, all);
        if (sh.done) break;
        init = false;

        // ------------------------------------------------ A: u = z + beta u; v = A u
        ResAcc<T> auv;
        ++ep;
        const T beta = (T)sh.beta;
#pragma unroll 1
        for (int r0 = 0; r0 < RR; r0 += 4) {
            T z[4][VEC], u[4][VEC];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                tm_ld(tv + 4 * (r0 + k), z[k]);
                V::ldrw(P + (r0 + k) * S, u[k]);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                tm_wait_ld(z[k]);
#pragma unroll
                for (int e = 0; e < VEC; ++e) u[k][e] = z[k][e] + beta * u[k][e];
                V::st(P + (r0 + k) * S, u[k]);
            }
        }
        if (hasS) {
            T u[VEC];
            V::ldrw(HU + c, u);
#pragma unroll
            for (int e = 0; e < VEC; ++e) u[e] = hS[e] + beta * u[e];
            V::st(HU + c, u);
        }
        if (hasN) {
            T u[VEC];
            V::ldrw(HU + nth + c, u);
#pragma unroll
            for (int e = 0; e < VEC; ++e) u[e] = hN[e] + beta * u[e];
            V::st(HU + nth + c, u);
        }
        __syncwarp();
        T fe[G][VEC], fn[G][VEC];
#pragma unroll
        for (int k = 0; k < G; ++k) {
            coef(q.aE, k, fe[k]);
            coef(q.aN, k, fn[k]);
        }
        bar_sync_n(1, TC);
        T us[VEC], uc[VEC], nS[VEC];
#pragma unroll
        for (int e = 0; e < VEC; ++e) nS[e] = aS0[e];
        V::ldrw(pS, us);
        V::ldrw(P, uc);
#pragma unroll 1
        for (int r0 = 0; r0 < RR; r0 += G) {
            T ev[G][VEC], nv[G][VEC];
#pragma unroll
            for (int k = 0; k < G; ++k)
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    ev[k][e] = fe[k][e];
                    nv[k][e] = fn[k][e];
                }
            if (r0 + G < RR) {
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    coef(q.aE, r0 + G + k, fe[k]);
                    coef(q.aN, r0 + G + k, fn[k]);
                }
            }
#pragma unroll
            for (int k = 0; k < G; ++k) {
                const int rr = r0 + k;
                const bool in = rr < nr;
                T un[VEC], v[VEC], bnd[VEC];
                V::ldrw(rr == RR - 1 || rr == nr - 1 ? pN : P + (rr + 1) * S, un);
                T uW = __shfl_up_sync(0xffffffffu, uc[VEC - 1], 1);
                T uE = __shfl_down_sync(0xffffffffu, uc[0], 1);
                T aW = __shfl_up_sync(0xffffffffu, ev[k][VEC - 1], 1);
                if (segw) {
                    uW = in ? pW[rr * S] : T(0);
                    aW = in ? EYl[er + rr * NS] : T(0);
                }
                if (!in) aW = T(0);
                if (sege) uE = in ? pE[rr * S] : T(0);
                // the Dirichlet term of the first and last rows
                const bool end = last && rr == nr - 1;
#pragma unroll
                for (int e = 0; e < VEC; ++e) bnd[e] = T(0);
                if (in && (j0 + lr0 + rr == 0 || end))
                    V::ldrw(q.dbnd + ((size_t)q.cslot[cond] * 2 + (end ? 1 : 0)) * nth + c, bnd);
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    const T xE = e < VEC - 1 ? uc[e + 1] : uE;
                    const T xW = e > 0 ? uc[e - 1] : uW;
                    const T a = e > 0 ? ev[k][e - 1] : aW;
                    const T dg = (((ev[k][e] + a) + nv[k][e]) + nS[e]) + bnd[e];
                    const T up = end ? T(0) : nv[k][e] * un[e];
                    v[e] = dg * uc[e] - ev[k][e] * xE - a * xW - up - nS[e] * us[e];
                }
                auv.add(uc, v);
                if (hasS && rr == 0) ll_put<VEC>(halo, v, ep);
                if (hasN && rr == nr - 1) ll_put<VEC>(halo + q.halo_row, v, ep);
                __syncwarp();
                tm_st(tv + 4 * rr, v);
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    us[e] = uc[e];
                    uc[e] = un[e];
                    nS[e] = rr + 1 < nr ? nv[k][e] : T(0);
                }
            }
        }
        tm_wait_st();
        {
            const ResSum<T> x[1] = {auv.value()};
            ResTerm<T> t[1];
            res_warp_sums<1>(x, t);
            if (lane == 0) sh.part[0][wid] = t[0];
            bar_sync_n(2, all);
        }
        fetch(1, 0);
        bar_sync_n(2, all);
    }

    // p64 += x in its units
#pragma unroll 1
    for (int rr = 0; rr < nr; ++rr) {
        T x[VEC];
        V::ldrw(pX + (size_t)rr * nth, x);
        double *const p = q.p64 + off + (size_t)rr * nth;
#pragma unroll
        for (int e = 0; e < VEC; ++e) p[e] = fma(sh.back, (double)x[e], p[e]);
    }
    __syncwarp();
    return ep;
}

static __global__ void __launch_bounds__(kResThreads + 32, 1) k_resident_tm(const __grid_constant__ ResParams<float> q)
{
    using T = float;
    ResShared<T> &sh = res_shared<T>();
    __shared__ unsigned s_tmem;
    res_clear(sh);
    if ((int)threadIdx.x >= q.threads) {
        res_exchange_warp<T, false>(q, sh, q.sc, 0, 0, (int)gridDim.x, threadIdx.x & 31);
        return;
    }
    // omega/D of the first rows stays in shared memory
    {
        const ResRows<T, 4, kTmRows, false> w(q, sh);
        extern __shared__ __align__(16) unsigned char g_res_smem[];
        T *const PI = reinterpret_cast<T *>(g_res_smem + q.o_x) + w.tid * 4;
        for (int rr = 0; rr < q.ri; ++rr) {
            T t[4] = {0.0f, 0.0f, 0.0f, 0.0f};
            if (rr < w.nr) Vec<T, 4>::ldrw(q.invD + w.coff + (size_t)rr * w.nth, t);
            Vec<T, 4>::st(PI + rr * kResThreads * 4, t);
        }
    }
    if (threadIdx.x < 32) tm_alloc(&s_tmem);
    unsigned ep = q.epoch;
    res_setup<T, 4, kTmRows, false>(q);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    bar_sync_n(1, q.threads);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const unsigned tmem = s_tmem;
#pragma unroll 1
    for (;;) {
        res_residual<T, 4, kTmRows, false>(q, ++ep);
        res_decide<false>(q, sh);
        if (sh.stop) break;
        ep = res_iterate_tm(q, sh, ep, tmem);
    }
    bar_sync_n(1, q.threads);
    if (threadIdx.x < 32) tm_free(tmem);
}

ResKernel res_kernel_tm() { GMAF_RES_KERNEL((k_resident_tm)); }

}  // namespace gmaf
