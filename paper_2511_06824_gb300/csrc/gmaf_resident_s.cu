// The resident PCG with its vectors in tensor memory: runs of 8 rows, and in FP64 of 16.
//
// Above 64 bytes a thread the registers do not hold r beside the product.  Both then live in
// the SM's tensor memory (256 KB that nothing else here uses).  Runs of 8 rows keep the
// couplings there too (four fields of 32 words a thread), so that an iteration reads at most
// the diagonal, omega/D and x from L2; runs of 16 stream the couplings, one group of rows ahead
// of the one worked on.  u stays in shared memory.  Both sweeps of the preconditioner are one pass
// upwards, z following w by a row: a barrier and a reading of the couplings fewer than in two.
//
// FP64 is bound by its pipe (one warp instruction holds a quarter of the SM for 64 cycles), so
// the system is scaled: with s^2 = omega/D of the preconditioner, s A s has unit weights in both
// sweeps and a constant diagonal, which leaves 15 of 18 operations a cell and iteration; Q = 1/s^2
// gives r.r in the caller's units.  On 9 conditions of 512 x 256 cells an iteration takes 41.3 us
// (A 17.3, B 23.7; the pipe alone 30 us on 144 of 152 SMs) against 49.3 unscaled with r in shared
// memory and the couplings from L2; on 5 of 700 x 384 cells 56 us, the phase kernels 95.
// FP32 runs are bound by L2 and by instructions, and stay unscaled: they do the phase kernels'
// arithmetic in their order (see res_fma).  On 9 conditions of 640 x 256 cells 14.8 us an
// iteration, against 23.2 with r in shared memory and the couplings from L2.
#include "gmaf_resident.cuh"
#include "gmaf_tmem.cuh"

namespace gmaf {

// ------------------------------------------------------------------ rows

// What a thread that owns rows works on: its columns and rows, and the block's shared
// memory.  Built anew for each part of a solve (the thread's number is read again, volatile),
// so that nothing lives in registers across the iterations.
template <typename T, int RR>
struct ResGeom {
    static constexpr int VEC = 16 / (int)sizeof(T);
    static constexpr int S = kResThreads * VEC;     // private fields: [row][thread][VEC]
    int nth, nz, tid, lane, wid;
    int j0, R, run, cg, c, lr0, nr;                 // the block's rows; first local row and rows of the run
    bool act, top, last;                            // rows at all; the block's last rows; the run ends at row nz - 1
    bool hasS, hasN;                                // a block below, above
    int seg, nseg;                                  // segment of 32 threads in the row, and how many
    bool segw, sege, atw, ate;                      // edges of a segment, of the row
    unsigned off, coff;                             // first cell in the fields, in the coefficient slots
    T *P;                                           // u: P[rr * S]
    // rows: [2][nth] u and r on the halo rows; [nrr][nth] E, y north and y south of each run and
    // (without the scaling) omega/D north, and omega/D on the south halo row
    T *HU, *HR, *EN, *YN, *YS, *IN, *IS;
    // records of this thread's segment (ES values, the next row's are es further) and of a row (RS
    // values), for rows -1 .. R of the block, from this run's first row on
    T *eb, *rb;
    int es;
    enum { FY, EY, EL, NF, IF, WE, ES };    // first and last y, last E, first N and omega/D; w of the next
                                            // segment's first column
    enum { Y2, E2, N2, I2, WL, RS };        // y and E of column nth - 2; N, omega/D and w of column nth - 1

    __device__ __forceinline__ ResGeom(const ResParams<T> &q)
    {
        extern __shared__ __align__(16) unsigned char g_res_smem[];
        nth = q.nth;
        nz = q.nz;
        asm volatile("mov.u32 %0, %%tid.x;\n" : "=r"(tid));
        lane = tid & 31;
        wid = tid >> 5;
        const int cond = blockIdx.x / q.bpc, bc = blockIdx.x - cond * q.bpc;
        j0 = (int)((long long)bc * nz / q.bpc);
        R = (int)((long long)(bc + 1) * nz / q.bpc) - j0;
        run = tid / q.P;
        cg = tid - run * q.P;
        c = cg * VEC;
        lr0 = run * RR;
        nr = R - lr0;
        nr = cg >= q.ncg || nr < 0 ? 0 : (nr > RR ? RR : nr);
        act = nr > 0;
        top = act && lr0 + nr == R;
        last = top && j0 + R == nz;
        hasS = act && run == 0 && j0 > 0;
        hasN = top && !last;
        seg = cg >> 5;
        nseg = q.nseg;
        segw = (cg & 31) == 0;
        sege = (cg & 31) == 31 || cg == q.ncg - 1;
        atw = cg == 0;
        ate = cg == q.ncg - 1;
        // (whatever fits on the SMs has less than 2^32 cells)
        off = (unsigned)cond * (unsigned)q.n + (unsigned)((j0 + lr0) * nth + c);
        coff = (unsigned)q.cslot[cond] * (unsigned)q.n + (unsigned)((j0 + lr0) * nth + c);
        P = reinterpret_cast<T *>(g_res_smem) + tid * VEC;
        HU = reinterpret_cast<T *>(g_res_smem + q.o_rows);
        HR = HU + 2 * nth;
        EN = HR + 2 * nth;
        YN = EN + q.nrr * nth;
        YS = YN + q.nrr * nth;
        IN = YS + q.nrr * nth;
        IS = IN + q.nrr * nth;
        T *const edge = reinterpret_cast<T *>(g_res_smem + q.o_edge);
        es = nseg * ES;
        eb = edge + ((lr0 + 1) * nseg + seg) * ES;
        rb = edge + (q.rows + 2) * nseg * ES + (lr0 + 1) * RS;
    }
    __device__ __forceinline__ unsigned tm(unsigned base, int field) const
    {
        return base + ((unsigned)(wid & 3) << 21) + (unsigned)(wid >> 2) * 128u + (unsigned)(field * RR * 4);
    }
};

// The coefficients that stay on the SM, and zeros where no block lies beyond.
template <typename T, int RR, int TM>
__device__ __noinline__ void res_setup_s(const ResParams<T> &q, unsigned tmem)
{
    const ResGeom<T, RR> w(q);
    constexpr int VEC = w.VEC;
    constexpr bool kScaled = sizeof(T) == 8;
    using V = Vec<T, VEC>;
    constexpr int S = w.S;
    extern __shared__ __align__(16) unsigned char g_res_smem[];
    const int nth = w.nth, most = w.nr > 0 ? w.nr - 1 : 0;
    {
        T *const rows = w.HU;
        for (int i = w.tid; i < res_tm_rows(q.nrr, sizeof(T)) * nth; i += q.threads) rows[i] = T(0);
        T *const edge = reinterpret_cast<T *>(g_res_smem + q.o_edge);
        for (int i = w.tid; i < (q.rows + 2) * (w.ES * q.nseg + w.RS); i += q.threads) edge[i] = T(0);
    }
    bar_sync_n(1, q.threads);
    const unsigned base = w.act ? w.coff : (unsigned)q.cslot[blockIdx.x / q.bpc] * (unsigned)q.n;
    // (the rows of the block's halo give the edges only)
    for (int rr = -1; rr <= RR; ++rr) {
        const bool in = rr >= 0 && rr < w.nr;
        const bool edges = in || (rr == -1 && w.hasS) || (rr == w.nr && w.hasN);
        T e[VEC], n[VEC];
#pragma unroll
        for (int k = 0; k < VEC; ++k) e[k] = n[k] = T(0);
        const unsigned at = base + (unsigned)((edges ? rr : 0) * nth);
        if (edges) {
            T od[VEC];
            V::ldrw(q.aE + at, e);
            if (!(w.last && rr == w.nr - 1)) V::ldrw(q.aN + at, n);    // (a_N of row nz - 1 couples to nothing)
            if (w.sege) w.eb[rr * w.es + w.EL] = e[VEC - 1];
            if (w.segw) w.eb[rr * w.es + w.NF] = n[0];
            if (w.ate) w.rb[rr * w.RS + w.N2] = n[VEC - 1];
            if (w.ate) w.rb[rr * w.RS + w.E2] = e[VEC - 2];
            const bool above = rr == w.nr, first = rr == 0 && w.run > 0;
            if (above || first) V::st(w.EN + (w.run - (first ? 1 : 0)) * nth + w.c, e);
            if constexpr (!kScaled) {
                V::ldrw(q.invD + at, od);
                if (w.segw) w.eb[rr * w.es + w.IF] = od[0];
                if (w.ate) w.rb[rr * w.RS + w.I2] = od[VEC - 1];
                if (above || first) V::st(w.IN + (w.run - (first ? 1 : 0)) * nth + w.c, od);
                if (rr == -1) V::st(w.IS + w.c, od);
            }
        }
        if (rr < 0 || rr == RR) continue;
        T zero[VEC];
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            zero[k] = T(0);
            e[k] = in ? e[k] : T(0);
            n[k] = in ? n[k] : T(0);
        }
        V::st(w.P + rr * S, zero);
        if constexpr (TM == 2)
            if (rr < q.keep) V::st(reinterpret_cast<T *>(g_res_smem + q.o_keep) + w.tid * VEC + rr * S, e);
        if constexpr (TM == 1) {
            __syncwarp();
            tm_st(w.tm(tmem, 2) + 4 * rr, e);
            tm_st(w.tm(tmem, 3) + 4 * rr, n);
        }
        if (q.o_q >= 0) {
            V::ldrw((kScaled ? q.Q : q.invD) + base + (unsigned)(min(rr, most) * nth), e);
#pragma unroll
            for (int k = 0; k < VEC; ++k) e[k] = in ? e[k] : T(0);
            V::st(reinterpret_cast<T *>(g_res_smem + q.o_q) + w.tid * VEC + rr * S, e);
        }
    }
    if constexpr (TM == 1) tm_wait_st();
}

// One PCG run: the start (ep: the last exchange's number), the iterations, the result.
// Returns the last exchange's number.
//
// Every thread computes all RR rows: rows and threads beyond the block's have zero
// coefficients and only their stores are left out, so that the rows of a run are
// independent straight-line code.
template <typename T, int RR, int TM>
__device__ __forceinline__ unsigned res_iterate_s(const ResParams<T> &q, ResShared<T> &sh, unsigned ep,
                                                unsigned tmem)
{
    using Geom = ResGeom<T, RR>;
    constexpr int S = Geom::S, VEC = Geom::VEC;
    using V = Vec<T, VEC>;
    constexpr bool kMixed = sizeof(T) == 4;         // FP32 runs inside FP64 refinement
    constexpr bool kScaled = !kMixed;
    constexpr int G = 2, NG = RR / G;               // rows at a time, groups of them
    extern __shared__ __align__(16) unsigned char g_res_smem[];
    const Geom w(q);
    const int nth = w.nth, TC = q.threads, all = TC + 32, lane = w.lane, wid = w.wid;
    const int run = w.run, cg = w.cg, c = w.c, lr0 = w.lr0, nr = w.nr, seg = w.seg, nseg = w.nseg;
    const bool act = w.act, top = w.top, hasS = w.hasS, hasN = w.hasN;
    const bool segw = w.segw, sege = w.sege, atw = w.atw, ate = w.ate;
    const unsigned off = w.off;
    const bool assor = q.precond == 1;
    T *const P = w.P, *const HU = w.HU, *const HR = w.HR;
    // u of the rows beyond the run and of the threads beyond the warp
    T *const sm = reinterpret_cast<T *>(g_res_smem);
    const T *const pS = !act ? P : run == 0 ? HU + c : P - q.P * VEC + (RR - 1) * S;
    const T *const pN = !act ? P : top ? HU + nth + c : P + q.P * VEC;
    const T *const pW = sm + (run * q.P + (atw ? q.ncg - 1 : cg - 1)) * VEC + VEC - 1;
    const T *const pE = sm + (run * q.P + (ate ? 0 : cg + 1)) * VEC;
    T *const eb = w.eb, *const rb = w.rb;
    const int es = w.es;
    constexpr int ES = Geom::ES, RS = Geom::RS, FY = Geom::FY, EY = Geom::EY, EL = Geom::EL, NF = Geom::NF;
    constexpr int IF = Geom::IF, WE = Geom::WE, Y2 = Geom::Y2, E2 = Geom::E2, N2 = Geom::N2, I2 = Geom::I2;
    constexpr int WL = Geom::WL;
    // from this segment's record to the west neighbour's, the row's first and last
    const int toW = (atw ? nseg - 1 : -1) * ES, toF = -seg * ES, toL = (nseg - 1 - seg) * ES;
    T *const pX = q.o_x >= 0 ? reinterpret_cast<T *>(g_res_smem + q.o_x) + w.tid * VEC : q.x + off;
    const int stX = q.o_x >= 0 ? S : nth;
    // coefficients in global memory: rows beyond the block's read the last one's place
    const int most = nr > 0 ? nr - 1 : 0;
    const unsigned cat = act ? w.coff : (unsigned)q.cslot[blockIdx.x / q.bpc] * (unsigned)q.n;
    // Q (the scaled form) or omega/D
    const T *const gQ = kScaled ? q.Q : q.invD;
    const T *const pQ = q.o_q >= 0 ? reinterpret_cast<const T *>(g_res_smem + q.o_q) + w.tid * VEC : gQ + cat;
    const int stQ = q.o_q >= 0 ? S : nth, mostQ = q.o_q >= 0 ? RR - 1 : most;
    auto get_Q = [&](int rr, T(&x)[VEC]) {
        V::ldrw(pQ + min(rr, mostQ) * stQ, x);
#pragma unroll
        for (int e = 0; e < VEC; ++e) x[e] = rr < nr ? x[e] : T(0);
    };
    auto stream = [&](const T *g, int rr, T(&x)[VEC]) {
        V::ldrw(g + (cat + (unsigned)(min(rr, most) * nth)), x);
#pragma unroll
        for (int e = 0; e < VEC; ++e) x[e] = rr < nr ? x[e] : T(0);
    };
    auto get_E = [&](int rr, T(&x)[VEC]) {
        if (rr < q.keep)
            V::ldrw(reinterpret_cast<const T *>(g_res_smem + q.o_keep) + w.tid * VEC + rr * S, x);
        else
            stream(q.aE, rr, x);
    };
    auto get_N = [&](int rr, T(&x)[VEC]) {
        stream(q.aN, rr, x);
        if (w.last && rr == nr - 1) {
#pragma unroll
            for (int e = 0; e < VEC; ++e) x[e] = T(0);
        }
    };
    const unsigned tv = w.tm(tmem, 0), tr = w.tm(tmem, 1), te = w.tm(tmem, 2), tn = w.tm(tmem, 3);

    // rows of a block's halo area: 0, 1 = first and last row of v; 2, 3 = of z
    unsigned long long *const halo = q.halo + (size_t)blockIdx.x * 4 * q.halo_row + c * ((int)sizeof(T) / 4);
    T aS0[VEC], hS[VEC], hN[VEC];
    // G rows of N fields in tensor memory
    auto field = [&](int r0, unsigned a, T(&x)[G][VEC]) {
        TmRow t[G];
#pragma unroll
        for (int k = 0; k < G; ++k) tm_ld(a + 4 * (r0 + k), t[k]);
        tm_wait_ld(t);
#pragma unroll
        for (int k = 0; k < G; ++k) tm_get(t[k], x[k]);
    };
    auto fields = [&](int r0, unsigned a, T(&x)[G][VEC], unsigned b, T(&y)[G][VEC]) {
        TmRow t[2 * G];
#pragma unroll
        for (int k = 0; k < G; ++k) {
            tm_ld(a + 4 * (r0 + k), t[k]);
            tm_ld(b + 4 * (r0 + k), t[G + k]);
        }
        tm_wait_ld(t);
#pragma unroll
        for (int k = 0; k < G; ++k) {
            tm_get(t[k], x[k]);
            tm_get(t[G + k], y[k]);
        }
    };
    auto put_done = [&] {
        __syncwarp();
        tm_wait_st();
    };

    // the warps' sums, for the exchange warp
    auto publish = [&](const ResSum<T> &a) {
        const ResSum<T> x[1] = {a};
        ResTerm<T> t[1];
        res_warp_sums<1>(x, t);
        if (lane == 0) sh.part[0][wid] = t[0];
        bar_sync_n(2, all);
    };
    auto publish2 = [&](const ResSum<T> &a, const ResSum<T> &b) {
        const ResSum<T> x[2] = {a, b};
        ResTerm<T> t[2];
        res_warp_sums<2>(x, t);
        if (lane == 0) {
            sh.part[0][wid] = t[0];
            sh.part[1][wid] = t[1];
        }
        bar_sync_n(2, all);
    };
    // the neighbours' rows: `s`, the last row of the block below, `n`, the first of the one above
    auto fetch = [&](int s, int n) {
        bool ok = true;
        if (hasS) ok = ll_get<VEC>(halo + (s - 4) * q.halo_row, hS, ep, q.polls);
        if (hasN) ok = ll_get<VEC>(halo + (n + 4) * q.halo_row, hN, ep, q.polls) && ok;
        if (!ok) sh.halo_failed = 1;
        __syncwarp();
    };

#pragma unroll
    for (int e = 0; e < VEC; ++e) aS0[e] = hS[e] = hN[e] = T(0);
    if (w.j0 + lr0 > 0 && act) V::ldrw(q.aN + w.coff - nth, aS0);

    // ---- start: r = s (b - A p), or s times the residual handed in; x = 0
    {
        double unit = 1.0;
        ResAcc<double> acc;
        if constexpr (kMixed) unit = sh.unit;
        ++ep;
#pragma unroll 1
        for (int rr = 0; rr < RR; ++rr) {
            T r[VEC], x[VEC];
#pragma unroll
            for (int e = 0; e < VEC; ++e) r[e] = x[e] = T(0);
            if (rr < nr) {
                const unsigned go = off + (unsigned)(rr * nth), co = w.coff + (unsigned)(rr * nth);
                T s[VEC];
                if constexpr (kScaled) V::ldrw(q.s + co, s);
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    double b[1];
                    if constexpr (kMixed) {
                        b[0] = q.r64[go + e] * unit;
                    } else if (q.mode == kResRestart) {
                        b[0] = q.r_in[go + e];
                    } else {
                        b[0] = q.b[go + e];
                        acc.add(b, b);
                        if (!q.zero_init) {
                            const int j = w.j0 + lr0 + rr;
                            const int ie = c + e == nth - 1 ? 1 - nth + e : e + 1;
                            const int iw = c + e == 0 ? nth - 1 : e - 1;
                            const double *p = q.p64 + go, *aE = q.aE64 + co, *aN = q.aN64 + co;
                            double ap = q.D64[co + e] * p[e] - aE[e] * p[ie] - aE[iw] * p[iw];
                            if (j < w.nz - 1) ap -= aN[e] * p[nth + e];
                            if (j > 0) ap -= aN[e - nth] * p[e - nth];
                            b[0] -= ap;
                        }
                    }
                    r[e] = kScaled ? s[e] * (T)b[0] : (T)b[0];
                }
                if (hasS && rr == 0) ll_put<VEC>(halo, r, ep);
                if (hasN && rr == nr - 1) ll_put<VEC>(halo + q.halo_row, r, ep);
            }
            __syncwarp();
            tm_st(tr + 4 * (rr), r);
            tm_st(tv + 4 * (rr), x);
            if (q.o_x >= 0 || rr < nr) V::st(pX + rr * stX, x);
            asm volatile("" ::: "memory");      // (one row's doubles in registers at a time)
        }
        put_done();
        if constexpr (!kMixed) {
            // exchange 0: b.b
            publish(acc.value());
            fetch(1, 0);
            bar_sync_n(2, all);
        } else {
            fetch(1, 0);
        }
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
        for (int g = 0; g < NG; ++g) {
            const int r0 = g * G;
            T v[G][VEC], r[G][VEC];
            fields(r0, tv, v, tr, r);
#pragma unroll
            for (int k = 0; k < G; ++k) {
#pragma unroll
                for (int e = 0; e < VEC; ++e) r[k][e] = res_fnma(alpha, v[k][e], r[k][e]);
                tm_st(tr + 4 * (r0 + k), r[k]);
            }
            // y: r in the scaled form
            T y[G][VEC];
#pragma unroll
            for (int k = 0; k < G; ++k) {
                T od[VEC];
                if constexpr (!kScaled) get_Q(r0 + k, od);
#pragma unroll
                for (int e = 0; e < VEC; ++e) y[k][e] = kScaled ? r[k][e] : r[k][e] * od[e];
                if (!kScaled || !assor) tm_st(tv + 4 * (r0 + k), y[k]);
            }
#pragma unroll
            for (int k = 0; k < G; ++k) {
                const int rr = r0 + k;
                if (assor) {
                    if (rr == RR - 1 && act && !top) V::st(w.YS + (run + 1) * nth + c, y[k]);
                    if (rr == 0 && act && run > 0) V::st(w.YN + (run - 1) * nth + c, y[k]);
                    if (sege && rr < nr) eb[rr * es + EY] = y[k][VEC - 1];
                    if (segw && rr < nr) eb[rr * es + FY] = y[k][0];
                    if (ate && rr < nr) rb[rr * RS + Y2] = y[k][VEC - 2];
                } else {
                    // (without the sweeps z is y)
                    T t[VEC];
                    if constexpr (kScaled) get_Q(rr, t);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) t[e] = kScaled ? r[k][e] * t[e] : r[k][e];
                    arz.add(r[k], y[k]);
                    arr.add(r[k], t);
                    if (hasS && rr == 0) ll_put<VEC>(halo + 2 * q.halo_row, y[k], ep);
                    if (hasN && rr == nr - 1) ll_put<VEC>(halo + 3 * q.halo_row, y[k], ep);
                }
            }
            __syncwarp();
        }
        if (hasS) {
            T h[VEC], od[VEC];
            V::ldrw(HR + c, h);
#pragma unroll
            for (int e = 0; e < VEC; ++e) h[e] = init ? hS[e] : res_fnma(alpha, hS[e], h[e]);
            V::st(HR + c, h);
            if constexpr (!kScaled) {
                V::ldrw(w.IS + c, od);
#pragma unroll
                for (int e = 0; e < VEC; ++e) h[e] *= od[e];
            }
            V::st(w.YS + c, h);
            if (sege) eb[EY - es] = h[VEC - 1];
            if (segw) eb[FY - es] = h[0];
        }
        if (hasN) {
            T od[VEC];
            V::ldrw(HR + nth + c, yN);
#pragma unroll
            for (int e = 0; e < VEC; ++e) yN[e] = init ? hN[e] : res_fnma(alpha, hN[e], yN[e]);
            V::st(HR + nth + c, yN);
            if constexpr (!kScaled) {
                V::ldrw(w.IN + run * nth + c, od);
#pragma unroll
                for (int e = 0; e < VEC; ++e) yN[e] *= od[e];
            }
            if (sege) eb[nr * es + EY] = yN[VEC - 1];
            if (segw) eb[nr * es + FY] = yN[0];
        }
        put_done();
        if (assor) {
            T fe[G][VEC], fn[G][VEC], fq[G][VEC];
            if constexpr (TM == 2) {
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    get_E(k, fe[k]);
                    get_N(k, fn[k]);
                    get_Q(k, fq[k]);
                }
            }
            bar_sync_n(1, TC);
            // w where this warp needs it of columns that it does not hold: the next segment's
            // first column and, for column 0, column nth - 1
            {
                const int rows = min(RR, w.R - lr0), step = min(q.P, 32);
                for (int k = cg & 31; k < rows; k += step) {
                    T *const a = eb + k * es, *const n = a + ES, *const l = a + toL, *const t = rb + k * RS;
                    if (seg + 1 < nseg) {
                        const T sum = res_fma(a[EL], a[EY], n[NF - es] * n[FY - es]);
                        a[WE] = kScaled ? n[FY] + sum : res_fma(n[IF], sum, n[FY]);
                    }
                    if (seg == 0) {
                        T sum = t[N2 - RS] * l[EY - es];
                        sum = res_fma(l[EL], a[FY], res_fma(t[E2], t[Y2], sum));
                        t[WL] = kScaled ? l[EY] + sum : res_fma(t[I2], sum, l[EY]);
                    }
                }
                __syncwarp();
            }
            // Both sweeps in one pass upwards: w = y + (lower couplings of y) (Eq. 3.5) on a row,
            // then z = w + (upper couplings of w) (Eq. 3.6) on the one below it.
            // (rp: r of the row below, y itself in the scaled form; dp: its omega/D)
            T yp[VEC], wp[VEC], ev[VEC], nv[VEC], eN[VEC], rp[VEC], dp[VEC], dN[VEC];
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                yp[e] = wp[e] = ev[e] = eN[e] = rp[e] = dp[e] = dN[e] = T(0);
                nv[e] = aS0[e];
            }
            if (act) {
                V::ldrw(w.YS + run * nth + c, yp);
                V::ldrw(w.EN + run * nth + c, eN);
                if constexpr (!kScaled) V::ldrw(w.IN + run * nth + c, dN);
                if (!top) V::ldrw(w.YN + run * nth + c, yN);
            }
            auto step = [&](int rr, T(&y)[VEC], T(&e0)[VEC], const T(&n0)[VEC], const T(&r)[VEC], T(&od)[VEC]) {
                if (rr == nr) {                     // the row above the run
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        y[e] = yN[e];
                        e0[e] = eN[e];
                        od[e] = dN[e];
                    }
                }
                T yW = __shfl_up_sync(0xffffffffu, y[VEC - 1], 1);
                T aW = __shfl_up_sync(0xffffffffu, e0[VEC - 1], 1);
                const bool in = act && rr <= nr;
                if (segw) {
                    yW = in && !atw ? eb[rr * es + toW + EY] : T(0);
                    aW = in && !atw ? eb[rr * es + toW + EL] : T(0);
                }
                T wv[VEC];
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    T sum = kScaled ? res_fma(nv[e], yp[e], y[e]) : nv[e] * yp[e];
                    sum = res_fma(e > 0 ? e0[e - 1] : aW, e > 0 ? y[e - 1] : yW, sum);
                    if (e == VEC - 1 && ate && in) sum = res_fma(e0[e], eb[rr * es + toF + FY], sum);
                    wv[e] = kScaled ? sum : res_fma(od[e], sum, y[e]);
                }
                if (rr > 0) {
                    const int rz = rr - 1;
                    T wE = __shfl_down_sync(0xffffffffu, wp[0], 1);
                    if (sege) wE = rz < nr && !ate ? eb[rz * es + WE] : T(0);
                    T z[VEC];
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        T sum = kScaled ? res_fma(nv[e], wv[e], wp[e]) : nv[e] * wv[e];
                        // (column nth - 1 has no upper neighbour to the east: wE is 0 there)
                        sum = res_fma(ev[e], e < VEC - 1 ? wp[e + 1] : wE, sum);
                        if (e == 0 && atw && rz < nr) sum = res_fma(eb[rz * es + toL + EL], rb[rz * RS + WL], sum);
                        if (!kScaled) sum = res_fma(dp[e], sum, wp[e]);
                        z[e] = rz < nr ? sum : T(0);
                    }
                    arz.add(kScaled ? yp : rp, z);
                    if (hasS && rz == 0) ll_put<VEC>(halo + 2 * q.halo_row, z, ep);
                    if (hasN && rz == nr - 1) ll_put<VEC>(halo + 3 * q.halo_row, z, ep);
                    __syncwarp();
                    tm_st(tv + 4 * (rz), z);
                }
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    yp[e] = y[e];
                    wp[e] = wv[e];
                    ev[e] = e0[e];
                    nv[e] = n0[e];
                    rp[e] = r[e];
                    dp[e] = od[e];
                }
            };
#pragma unroll 1
            for (int g = 0; g < NG; ++g) {
                const int r0 = g * G;
                T y[G][VEC], r[G][VEC], e0[G][VEC], n0[G][VEC], od[G][VEC];
                {
                    constexpr int F = TM == 1 ? 3 : 1, M = F + (kScaled ? 0 : 1);
                    const unsigned at[4] = {kScaled ? tr : tv, TM == 1 ? te : tr, tn, tr};
                    TmRow t[M * G];
#pragma unroll
                    for (int f = 0; f < M; ++f)
#pragma unroll
                        for (int k = 0; k < G; ++k) tm_ld(at[f] + 4 * (r0 + k), t[f * G + k]);
                    tm_wait_ld(t);
#pragma unroll
                    for (int k = 0; k < G; ++k) {
                        tm_get(t[k], y[k]);
                        if constexpr (TM == 1) {
                            tm_get(t[G + k], e0[k]);
                            tm_get(t[2 * G + k], n0[k]);
                        }
                        tm_get(t[kScaled ? k : F * G + k], r[k]);
                    }
                }
#pragma unroll
                for (int k = 0; k < G; ++k) {
                    if constexpr (TM == 2) {
#pragma unroll
                        for (int e = 0; e < VEC; ++e) {
                            e0[k][e] = fe[k][e];
                            n0[k][e] = fn[k][e];
                            od[k][e] = fq[k][e];
                        }
                    } else {
                        get_Q(r0 + k, od[k]);
                    }
                    T t[VEC];
#pragma unroll
                    for (int e = 0; e < VEC; ++e) t[e] = kScaled ? r[k][e] * od[k][e] : r[k][e];
                    arr.add(r[k], t);
                }
                if constexpr (TM == 2) {
                    if (g + 1 < NG) {
#pragma unroll
                        for (int k = 0; k < G; ++k) {
                            get_E(r0 + G + k, fe[k]);
                            get_N(r0 + G + k, fn[k]);
                            get_Q(r0 + G + k, fq[k]);
                        }
                    }
                }
#pragma unroll
                for (int k = 0; k < G; ++k) step(r0 + k, y[k], e0[k], n0[k], r[k], od[k]);
            }
            {
                T y[VEC], e0[VEC], n0[VEC], od[VEC];
#pragma unroll
                for (int e = 0; e < VEC; ++e) y[e] = e0[e] = n0[e] = od[e] = T(0);
                step(RR, y, e0, n0, y, od);
            }
            put_done();
        }
        publish2(arz.value(), arr.value());
        // x += alpha u, and z on the neighbours' rows, while the sums travel
        if (!init) {
#pragma unroll 4
            for (int rr = 0; rr < RR; ++rr) {
                if (q.o_x < 0 && rr >= nr) continue;
                T x[VEC], u[VEC];
                V::ldrw(pX + rr * stX, x);
                V::ldrw(P + rr * S, u);
#pragma unroll
                for (int e = 0; e < VEC; ++e) x[e] = res_fma(alpha, u[e], x[e]);
                V::st(pX + rr * stX, x);
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
        for (int g = 0; g < NG; ++g) {
            const int r0 = g * G;
            T z[G][VEC];
            field(r0, tv, z);
#pragma unroll
            for (int k = 0; k < G; ++k) {
                T u[VEC];
                V::ldrw(P + (r0 + k) * S, u);
#pragma unroll
                for (int e = 0; e < VEC; ++e) u[e] = res_fma(beta, u[e], z[k][e]);
                V::st(P + (r0 + k) * S, u);
            }
        }
        if (hasS) {
            T u[VEC];
            V::ldrw(HU + c, u);
#pragma unroll
            for (int e = 0; e < VEC; ++e) u[e] = res_fma(beta, u[e], hS[e]);
            V::st(HU + c, u);
        }
        if (hasN) {
            T u[VEC];
            V::ldrw(HU + nth + c, u);
#pragma unroll
            for (int e = 0; e < VEC; ++e) u[e] = res_fma(beta, u[e], hN[e]);
            V::st(HU + nth + c, u);
        }
        __syncwarp();
        T fe[G][VEC], fn[G][VEC], gd[G][VEC];
        auto get_D = [&](int r0) {
            if constexpr (!kScaled) {
#pragma unroll
                for (int k = 0; k < G; ++k) stream(q.D, r0 + k, gd[k]);
            }
        };
        get_D(0);
        if constexpr (TM == 2) {
#pragma unroll
            for (int k = 0; k < G; ++k) {
                get_E(k, fe[k]);
                get_N(k, fn[k]);
            }
        }
        bar_sync_n(1, TC);
        const T dg0 = q.dg;
        T us[VEC], uc[VEC], nS[VEC];
#pragma unroll
        for (int e = 0; e < VEC; ++e) nS[e] = aS0[e];
        V::ldrw(pS, us);
        V::ldrw(P, uc);
#pragma unroll 1
        for (int g = 0; g < NG; ++g) {
            const int r0 = g * G;
            T e0[G][VEC], n0[G][VEC], fd[G][VEC];
#pragma unroll
            for (int k = 0; k < G; ++k)
#pragma unroll
                for (int e = 0; e < VEC; ++e) fd[k][e] = kScaled ? T(0) : gd[k][e];
            if (g + 1 < NG) get_D(r0 + G);
            if constexpr (TM == 1) {
                fields(r0, te, e0, tn, n0);
            } else if constexpr (TM == 2) {
#pragma unroll
                for (int k = 0; k < G; ++k)
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        e0[k][e] = fe[k][e];
                        n0[k][e] = fn[k][e];
                    }
                if (g + 1 < NG) {
#pragma unroll
                    for (int k = 0; k < G; ++k) {
                        get_E(r0 + G + k, fe[k]);
                        get_N(r0 + G + k, fn[k]);
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < G; ++k) {
                const int rr = r0 + k;
                T un[VEC], v[VEC], dg[VEC];
                V::ldrw(rr == RR - 1 || rr == nr - 1 ? pN : P + (rr + 1) * S, un);
                T uW = __shfl_up_sync(0xffffffffu, uc[VEC - 1], 1);
                T uE = __shfl_down_sync(0xffffffffu, uc[0], 1);
                T aW = __shfl_up_sync(0xffffffffu, e0[k][VEC - 1], 1);
                if (segw) {
                    uW = rr < nr ? pW[rr * S] : T(0);
                    aW = rr < nr ? eb[rr * es + toW + EL] : T(0);
                }
                if (rr >= nr) aW = T(0);        // (the last column's, next to a thread without columns)
                if (sege) uE = rr < nr ? pE[rr * S] : T(0);
#pragma unroll
                for (int e = 0; e < VEC; ++e) dg[e] = !kScaled ? fd[k][e] : rr < nr ? dg0 : T(0);
                if (kScaled && q.D && rr < nr) V::ldrw(q.D + (cat + (unsigned)(rr * nth)), dg);
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    const T xE = e < VEC - 1 ? uc[e + 1] : uE;
                    const T xW = e > 0 ? uc[e - 1] : uW;
                    const T a = e > 0 ? e0[k][e - 1] : aW;
                    T t = res_diff(dg[e], uc[e], e0[k][e], xE);
                    t = res_fnma(a, xW, t);
                    t = res_fnma(n0[k][e], un[e], t);
                    v[e] = res_fnma(nS[e], us[e], t);
                }
                auv.add(uc, v);
                if (hasS && rr == 0) ll_put<VEC>(halo, v, ep);
                if (hasN && rr == nr - 1) ll_put<VEC>(halo + q.halo_row, v, ep);
                __syncwarp();
                tm_st(tv + 4 * (rr), v);
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    us[e] = uc[e];
                    uc[e] = un[e];
                    nS[e] = rr + 1 < nr ? n0[k][e] : T(0);
                }
            }
        }
        put_done();
        publish(auv.value());
        fetch(1, 0);
        bar_sync_n(2, all);
    }

    // p += scale s x (mixed precision: in the run's units)
    {
        const double back = kMixed ? sh.back : *q.scale;
        const bool from0 = !kMixed && q.zero_init && q.mode != kResRestart;
        // (a restart that may be left out, and did not get there: p stays what it was)
        const bool leave = !kMixed && sh.done == 2 && ((q.optional >> (q.groups == 1 ? 0 : blockIdx.x / q.bpc)) & 1ull);
#pragma unroll 1
        for (int rr = 0; rr < (leave ? 0 : nr); ++rr) {
            T x[VEC], s[VEC];
            V::ldrw(pX + rr * stX, x);
            if constexpr (kScaled) V::ldrw(q.s + (w.coff + (unsigned)(rr * nth)), s);
            double *const p = q.p64 + off + (unsigned)(rr * nth);
#pragma unroll
            for (int e = 0; e < VEC; ++e) p[e] = fma(back, (double)(kScaled ? s[e] * x[e] : x[e]), from0 ? 0.0 : p[e]);
        }
        __syncwarp();
    }
    return ep;
}

template <typename T, int RR, int TM>
static __global__ void __launch_bounds__(kResThreads + 32, 1) k_resident_s(const __grid_constant__ ResParams<T> q)
{
    ResShared<T> &sh = res_shared<T>();
    __shared__ unsigned s_tmem;
    const int cond = blockIdx.x / q.bpc, grp = q.groups == 1 ? 0 : cond;
    if (!((q.mask >> grp) & 1ull)) return;                  // this group does not run
    res_clear(sh);
    if ((int)threadIdx.x >= q.threads) {
        res_exchange_warp<T>(q, sh, q.sc + grp, grp, q.groups == 1 ? 0 : cond * q.bpc,
                             q.groups == 1 ? (int)gridDim.x : q.bpc, threadIdx.x & 31);
        return;
    }
    if (threadIdx.x < 32) tm_alloc(&s_tmem);
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    bar_sync_n(1, q.threads);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const unsigned tmem = s_tmem;
    unsigned ep = q.epoch;
    res_setup_s<T, RR, TM>(q, tmem);
    if constexpr (sizeof(T) == 4) {
        // FP64 refinements around the FP32 run
#pragma unroll 1
        for (;;) {
            res_residual<T, 4, RR, false>(q, ++ep);
            res_decide<true>(q, sh);
            if (sh.stop) break;
            ep = res_iterate_s<T, RR, TM>(q, sh, ep, tmem);
        }
    } else {
        res_iterate_s<T, RR, TM>(q, sh, ep, tmem);
    }
    bar_sync_n(1, q.threads);
    if (threadIdx.x < 32) tm_free(tmem);
}

ResKernel res_kernel_s(int size, int rr)
{
    if (size == 4) GMAF_RES_KERNEL((k_resident_s<float, 8, 1>));
    if (rr == 8) GMAF_RES_KERNEL((k_resident_s<double, 8, 1>));
    GMAF_RES_KERNEL((k_resident_s<double, 16, 2>));
}

}  // namespace gmaf
