// Resident PCG: the whole joint solve in one cooperative launch, its vectors kept
// on the SMs.
//
// The phase kernels (gmaf_pcg_kernels.cuh) make two launches an iteration and pass
// every vector through memory between them.  On grids of up to about a million
// unknowns that costs far more than the arithmetic: 28 us an iteration on 2048
// unknowns and 31 us on 1.18 million (FP32), most of it launch boundaries, tasks
// marching rows one after the other and a last block adding all partial sums.
// Here every block owns whole rows of one condition for the whole solve: r and the
// product (v, later y, w and z in the same registers) live in registers, u in shared
// memory, x and the coefficients in shared memory as far as they fit (else they are
// streamed from L2), and an iteration is two exchanges between blocks:
//   after v = A u:     the sum u.v, and v on each block's first and last row;
//   after z = M^-1 r:  the sums r.z and r.r, and z on each block's first and last row.
// With a neighbour's v rows a block updates its copy of the neighbour's r rows, and
// with its z rows the copy of its u rows, so that no other field crosses blocks.
//
// The exchange needs no fences: every 8-byte word of a row that another block reads
// carries 4 bytes of payload and the 4-byte number of the exchange it belongs to, and
// readers poll the words themselves; sums are added up in L2 as integers, exactly and
// so in any order: all blocks take the same scalars and the same decisions, and a
// result does not depend on scheduling.  A block can write a word again only
// after an exchange that its readers entered after they had read it (v rows and u.v
// before the exchange of z, z rows and r.z before the next exchange of v).  All
// blocks are resident (cooperative launch); a wait that is not met after kResSpin
// polls ends the run with GMAF_TIMEOUT.
//
// Threads: lane groups of P threads (a power of two or a multiple of 32) cover a
// row, VEC columns each; every group marches a run of RR rows.  West and east
// neighbours come by shuffle, at the edges of a warp or row through shared memory.
// One more warp takes no rows: it adds the block's partial sums, publishes them,
// polls the others' and updates the scalars, while the other warps fetch the halo
// rows and add alpha u to x.
#pragma once

#include "gmaf_internal.cuh"
#include "gmaf_pcg_kernels.cuh"
#include "gmaf_resident.h"

namespace gmaf {

constexpr unsigned kResSpin = 1u << 21;     // polls (of about a microsecond) before a wait gives up

// ------------------------------------------------------------------ flagged words

__device__ __forceinline__ void ll_st2(unsigned long long *p, unsigned long long a,
                                       unsigned long long b)
{
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};\n" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void ll_st1(unsigned long long *p, unsigned long long a)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;\n" ::"l"(p), "l"(a) : "memory");
}
__device__ __forceinline__ void ll_ld2(const unsigned long long *p, unsigned long long &a,
                                       unsigned long long &b)
{
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];\n" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ unsigned long long ll_ld1(const unsigned long long *p)
{
    unsigned long long a;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];\n" : "=l"(a) : "l"(p) : "memory");
    return a;
}
__device__ __forceinline__ unsigned long long ll_word(unsigned payload, unsigned ep)
{
    return ((unsigned long long)ep << 32) | payload;
}

// VEC values as flagged words: one word a float, two a double.
template <int VEC>
__device__ __forceinline__ void ll_put(unsigned long long *p, const float (&x)[VEC], unsigned ep)
{
    if constexpr (VEC == 1) {
        ll_st1(p, ll_word(__float_as_uint(x[0]), ep));
    } else {
#pragma unroll
        for (int q = 0; q < VEC; q += 2)
            ll_st2(p + q, ll_word(__float_as_uint(x[q]), ep), ll_word(__float_as_uint(x[q + 1]), ep));
    }
}
template <int VEC>
__device__ __forceinline__ void ll_put(unsigned long long *p, const double (&x)[VEC], unsigned ep)
{
#pragma unroll
    for (int q = 0; q < VEC; ++q)
        ll_st2(p + 2 * q, ll_word((unsigned)__double2loint(x[q]), ep),
               ll_word((unsigned)__double2hiint(x[q]), ep));
}
// Polls until every word carries ep; false if that never happened.
template <int VEC>
__device__ __forceinline__ bool ll_get(const unsigned long long *p, float (&x)[VEC], unsigned ep)
{
    for (unsigned k = 0; k < kResSpin; ++k) {
        unsigned long long w[VEC];
        bool ok = true;
        if constexpr (VEC == 1) {
            w[0] = ll_ld1(p);
        } else {
#pragma unroll
            for (int q = 0; q < VEC; q += 2) ll_ld2(p + q, w[q], w[q + 1]);
        }
#pragma unroll
        for (int q = 0; q < VEC; ++q) ok = ok && (unsigned)(w[q] >> 32) == ep;
        if (ok) {
#pragma unroll
            for (int q = 0; q < VEC; ++q) x[q] = __uint_as_float((unsigned)w[q]);
            return true;
        }
    }
    return false;
}
template <int VEC>
__device__ __forceinline__ bool ll_get(const unsigned long long *p, double (&x)[VEC], unsigned ep)
{
    for (unsigned k = 0; k < kResSpin; ++k) {
        unsigned long long lo[VEC], hi[VEC];
        bool ok = true;
#pragma unroll
        for (int q = 0; q < VEC; ++q) ll_ld2(p + 2 * q, lo[q], hi[q]);
#pragma unroll
        for (int q = 0; q < VEC; ++q)
            ok = ok && (unsigned)(lo[q] >> 32) == ep && (unsigned)(hi[q] >> 32) == ep;
        if (ok) {
#pragma unroll
            for (int q = 0; q < VEC; ++q) x[q] = __hiloint2double((int)(unsigned)hi[q], (int)(unsigned)lo[q]);
            return true;
        }
    }
    return false;
}

// ------------------------------------------------------------------ sums
//
// A dependent FP64 addition takes 64 cycles here, a warp-wide butterfly of them 550, so
// sums over threads, warps and blocks are formed in integers: every term is put on a
// common power-of-two scale and the integers are added exactly, in any order.
//
// Within a warp (FP64) the scale is that of the largest term, 54 bits below its leading
// one: the quantum is half the last bit of the largest term, so the error is at most
// that of a chain of double additions.  FP32 keeps the two-float form of RowAcc through
// the warp's butterfly.  Across warps and blocks a value is an 80-bit integer in two
// limbs (44 bits and the rest), scaled so that the total expected (the last total of
// its kind) has 67 bits: a total may grow by 2^13, and one that shrank below 2^-12 of
// it would keep less than 54 bits; then, and the first time, the blocks first agree on
// the largest exponent among their terms.

constexpr int kResTop = 66;             // bit of the leading digit of the expected total
constexpr int kResLimb = 44;            // bits of the low limb
constexpr unsigned long long kResLimbMask = (1ull << kResLimb) - 1;

__device__ __forceinline__ int res_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// One warp's sum: FP64 v 2^(e - 1077) (e = 0x7ff: not finite), FP32 hi + lo.
template <typename T>
struct ResTerm;
template <>
struct ResTerm<double> {
    long long v;
    int e;
};
template <>
struct ResTerm<float> {
    float hi, lo;
};

// Warp sums of NV accumulators (in every lane).
template <int NV>
__device__ __forceinline__ void res_warp_sums(const double (&x)[NV], ResTerm<double> (&out)[NV])
{
    int e[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) e[q] = __reduce_max_sync(0xffffffffu, res_exp(x[q]));
    long long v[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        const int hi = __double2hiint(x[q]), ex = (hi >> 20) & 0x7ff, down = e[q] - ex;
        const unsigned long long m = ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) |
                                     (unsigned)__double2loint(x[q]);
        const long long t = ex == 0 || down > 56 ? 0ll : (long long)((m << 2) >> down);
        v[q] = hi < 0 ? -t : t;
    }
    // three limbs a value (24, 24 and 16 bits) by integer reductions over the warp
    unsigned s0[NV], s1[NV];
    int s2[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        s0[q] = __reduce_add_sync(0xffffffffu, (unsigned)v[q] & 0xffffffu);
        s1[q] = __reduce_add_sync(0xffffffffu, (unsigned)(v[q] >> 24) & 0xffffffu);
        s2[q] = __reduce_add_sync(0xffffffffu, (int)(v[q] >> 48));
    }
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        out[q].v = ((long long)s2[q] << 48) + (long long)(((unsigned long long)s1[q] << 24) + s0[q]);
        out[q].e = e[q];
    }
}
template <int NV>
__device__ __forceinline__ void res_warp_sums(const Acc<float> (&x)[NV], ResTerm<float> (&out)[NV])
{
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        out[q].hi = x[q].hi;
        out[q].lo = x[q].lo;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const float hi = out[q].hi;
            const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
            const float l2 = __shfl_xor_sync(0xffffffffu, out[q].lo, o);
            const float s = __fadd_rn(hi, h2);
            const float bb = __fsub_rn(s, hi);
            const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(h2, bb));
            out[q].lo = __fadd_rn(__fadd_rn(out[q].lo, l2), e);
            out[q].hi = s;
        }
    }
}

// The biased exponent (as of a double) of a term's leading bit; 0: zero, 0x7ff: not finite.
__device__ __forceinline__ int res_term_exp(const ResTerm<double> &t)
{
    if (t.e == 0x7ff) return 0x7ff;
    if (t.v == 0) return 0;
    return max(1, t.e - 54 + 63 - __clzll(t.v < 0 ? -t.v : t.v));
}
__device__ __forceinline__ int res_term_exp(const ResTerm<float> &t)
{
    const int e = (__float_as_uint(t.hi) >> 23) & 0xff;
    return e == 0 ? 0 : (e == 0xff ? 0x7ff : e + 896);
}

struct ResLimbs {
    long long lo, top;
    bool over;                          // too large for the scale
};
// m 2^up in units of the lowest bit (m of `bits` bits), added with its sign.
__device__ __forceinline__ void res_limbs_add(ResLimbs &x, unsigned long long m, int up, bool neg, int bits)
{
    unsigned long long lo, top;
    if (up >= kResLimb) {
        lo = 0;
        top = m << ((up - kResLimb) & 63);
    } else if (up >= 0) {
        lo = (m << up) & kResLimbMask;
        top = m >> (kResLimb - up);
    } else {
        m = up > -64 ? m >> -up : 0ull;
        lo = m & kResLimbMask;
        top = m >> kResLimb;
    }
    if (up + bits > kResTop + 14) {
        if (m != 0) x.over = true;
        lo = top = 0;
    }
    x.lo += neg ? -(long long)lo : (long long)lo;
    x.top += neg ? -(long long)top : (long long)top;
}
__device__ __forceinline__ ResLimbs res_limbs(const ResTerm<double> &t, int e)
{
    ResLimbs x{0, 0, t.e == 0x7ff};
    const bool neg = t.v < 0;
    const unsigned long long m = (unsigned long long)(neg ? -t.v : t.v);
    if (!x.over) res_limbs_add(x, m, t.e - e + kResTop - 54, neg, 64 - __clzll(m));
    return x;
}
__device__ __forceinline__ ResLimbs res_limbs(const ResTerm<float> &t, int e)
{
    ResLimbs x{0, 0, false};
    const float f[2] = {t.hi, t.lo};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const unsigned b = __float_as_uint(f[k]);
        const int ex = (b >> 23) & 0xff;
        if (ex == 0xff) x.over = true;
        if (ex > 0 && ex < 0xff)
            res_limbs_add(x, (b & 0x7fffffu) | 0x800000u, ex + 896 - e + kResTop - 23, (b >> 31) != 0, 24);
    }
    return x;
}

// ------------------------------------------------------------------ exchange of sums
//
// One line of words per group of blocks, which every block adds its limbs to (64-bit
// integer additions in L2) and every block polls: the total is there when the count in
// the words' low bits says so.  (Measured for 144 blocks: 0.73 us.  Reading every
// block's sum took 3.2 us, from one shared array or from an inbox a block, as each of
// the many lines read is taken away by writers in between; a grid barrier of
// cooperative groups takes 1.2 us without any sums.)
//
// The words are never reset during a run: readers keep what they held after the
// exchange before.  Words of one kind are added to again only after an exchange of
// another kind, which no block completes before all have read these.

enum ResWord { kWordUV = 0, kWordRZ = 4, kWordMaxCount = 8, kWordMax = 9 };
static_assert(kWordMax + 2 <= kResGroupWords, "words of a group");

struct ResSums {
    unsigned long long *w;              // the group's words (zero at the start of the run)
    unsigned long long prev[6], prev_max;
    int nb, e[3];                       // blocks; exponent expected of u.v, r.z, r.r (0: not known)
    unsigned turn;
};

__device__ __forceinline__ void res_red(unsigned long long *p, unsigned long long v)
{
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;\n" ::"l"(p), "l"(v) : "memory");
}

// The largest exponent of each of NV values over the group's blocks.
template <int NV>
__device__ __forceinline__ bool res_max_exp(ResSums &x, const int (&mine)[NV], int *e, int lane)
{
    ++x.turn;
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < NV; ++q)
            atomicMax(x.w + kWordMax + q, ((unsigned long long)x.turn << 16) | (unsigned)mine[q]);
        __threadfence();
        res_red(x.w + kWordMaxCount, 1ull);
    }
    for (unsigned k = 0; k < kResSpin; ++k) {
        if (ll_ld1(x.w + kWordMaxCount) - x.prev_max == (unsigned long long)x.nb) {
            x.prev_max += (unsigned long long)x.nb;
            __threadfence();
#pragma unroll
            for (int q = 0; q < NV; ++q) e[q] = (int)(ll_ld1(x.w + kWordMax + q) & 0xffffull);
            return true;
        }
    }
    return false;
}

// The totals over the group's blocks of NV values, of which each lane holds one term
// (in every lane); false if some block never came.  Values that are not finite or huge
// give NaN, ones next to zero give zero.
template <int NV, typename T>
__device__ __forceinline__ bool res_totals(ResSums &x, int kind, const ResTerm<T> (&term)[NV], int lane,
                                           double (&tot)[NV])
{
    unsigned long long *const w = x.w + (kind == 0 ? kWordUV : kWordRZ);
    unsigned long long *prev = x.prev + 2 * kind;
    int *e = x.e + kind;
    bool known = true;
#pragma unroll
    for (int q = 0; q < NV; ++q) known = known && e[q] != 0;
    for (int turn = 0; turn < 2; ++turn) {
        if (!known) {
            int ex[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) ex[q] = __reduce_max_sync(0xffffffffu, res_term_exp(term[q]));
            if (!res_max_exp<NV>(x, ex, e, lane)) return false;
        }
        int en[NV];
        unsigned long long word = 0;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            en[q] = e[q] > 80 && e[q] < 2030 ? e[q] : 1023;
            const ResLimbs l = res_limbs(term[q], en[q]);
            const unsigned l0 = __reduce_add_sync(0xffffffffu, (unsigned)l.lo & 0xffffffu);
            const int l1 = __reduce_add_sync(0xffffffffu, (int)(l.lo >> 24));
            const unsigned t0 = __reduce_add_sync(0xffffffffu, (unsigned)l.top & 0xffffffu);
            const int t1 = __reduce_add_sync(0xffffffffu, (int)(l.top >> 24));
            const bool over = __any_sync(0xffffffffu, l.over) != 0;
            const long long lo = ((long long)l1 << 24) + l0, top = ((long long)t1 << 24) + t0;
            // low limb: count in 8 bits; top limb: count and number of blocks with a term too large
            if (lane == 2 * q) word = ((unsigned long long)lo << 8) + 1ull;
            if (lane == 2 * q + 1) word = ((unsigned long long)top << 16) + (over ? 257ull : 1ull);
        }
        if (lane < 2 * NV) res_red(w + lane, word);
        unsigned long long d[2 * NV];
        bool ok = false;
        for (unsigned k = 0; k < kResSpin && !ok; ++k) {
            bool mine = true;
#pragma unroll
            for (int q = 0; q < NV; ++q) ll_ld2(w + 2 * q, d[2 * q], d[2 * q + 1]);
#pragma unroll
            for (int q = 0; q < 2 * NV; ++q)
                mine = mine && ((d[q] - prev[q]) & 0xffull) == (unsigned long long)x.nb;
            ok = __all_sync(0xffffffffu, mine);
        }
        if (!ok) return false;
        bool good = true;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const long long lo = (long long)(d[2 * q] - prev[2 * q]) >> 8;
            const unsigned long long t = d[2 * q + 1] - prev[2 * q + 1];
            const double s = fma((double)((long long)t >> 16), (double)(1ull << kResLimb), (double)lo);
            tot[q] = s == 0.0 ? 0.0 : __hiloint2double(__double2hiint(s) + ((en[q] - 1023 - kResTop) << 20),
                                                       __double2loint(s));
            good = good && ((t >> 8) & 0xffull) == 0 && res_exp(tot[q]) >= e[q] - 12;
            prev[2 * q] = d[2 * q];
            prev[2 * q + 1] = d[2 * q + 1];
        }
        if (!known || good) {
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                if (e[q] <= 80 || e[q] >= 2030)
                    tot[q] = e[q] <= 80 ? 0.0 : __longlong_as_double(0x7ff8000000000000ll);
                // (what the next total of the kind is expected to be)
                e[q] = res_exp(tot[q]);
                if (e[q] <= 80 || e[q] >= 2030) e[q] = 0;
            }
            return true;
        }
        known = false;
    }
    return false;
}

// a / b by Newton's iteration on the reciprocal from a single-precision start and one
// correction of the quotient by its residual (shorter than the general division: a
// dependent FP64 operation takes 64 cycles).
__device__ __forceinline__ double res_quotient(double a, double b)
{
    const float f = (float)b;
    if (!(fabsf(f) > 1e-30f && fabsf(f) < 1e30f)) return a / b;
    double y = (double)(1.0f / f);
    y = fma(y, fma(-b, y, 1.0), y);
    const double t = a * y;
    return fma(y, fma(-b, t, a), t);
}

// Barrier of the threads that own rows (the exchange warp does not take part).
__device__ __forceinline__ void bar_sync_n(int id, int threads)
{
    asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ unsigned long long res_time()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
    return t;
}

// ------------------------------------------------------------------ the exchange warp

// Shared state of a block.
template <typename T>
struct ResShared {
    ResTerm<T> part[2][kResThreads / 32];   // the warps' sums
    double alpha, beta;
    int done, halo_failed;
};

// The warp that takes no rows: adds the block's sums, exchanges them, updates the
// scalars (finish_a and finish_b of the phase kernels) and decides when to stop.
template <typename T>
__device__ __forceinline__ void res_exchange_warp(const ResParams<T> &q, ResShared<T> &sh, Scalars *sc,
                                                  int g0, int nb, int lane)
{
    const int all = q.threads + 32, warps = q.threads / 32;
    const int blk = blockIdx.x;
    int iter = q.keep_iter ? sc->iter : 0;
    double d = 0.0, normS = q.mode == kResRestart ? sc->normS : 0.0, rr_last = 0.0, alpha = 0.0;
    int status = 0, converged = 0, zero_rhs = 0, guard = 0, done = 0;
    const bool timed = q.times != nullptr && lane == 0 && blk == 0;
    unsigned long long t_mark = timed ? res_time() : 0ull;
    auto mark = [&](int k) {
        if (!timed) return;
        const unsigned long long t = res_time();
        q.times[k] += t - t_mark;
        t_mark = t;
    };
    auto gather = [&](int w) {
        ResTerm<T> t{};
        if (lane < warps) t = sh.part[w][lane];
        return t;
    };
    ResSums sums{};
    sums.w = q.words + (size_t)(q.groups == 1 ? 0 : blk / q.bpc) * kResGroupWords;
    sums.nb = nb;
    double d_inv = 0.0;
    bool d_plain = false;
    if (lane == 0) sh.done = sh.halo_failed = 0;

    // exchange 0: b.b (and r on the halo rows)
    bar_sync_n(2, all);
    {
        const ResTerm<T> mine[1] = {gather(0)};
        double tot[1];
        const bool got = res_totals<1, T>(sums, 0, mine, lane, tot);
        sums.e[0] = 0;
        if (!got) {
            status = GMAF_TIMEOUT;
            done = 1;
        } else if (q.mode != kResRestart) {
            normS = sqrt(tot[0]);
            zero_rhs = tot[0] == 0.0;
            if (!finite_d(tot[0])) {
                status = GMAF_NONFINITE;
                done = 1;
            }
        }
    }
    // a little above (eps ||b||)^2, compared as integers (r.r is not negative)
    const double thr = q.eps * normS;
    const long long thr2 = __double_as_longlong(thr * thr * (1.0 + 1e-10));
    if (lane == 0) {
        sh.alpha = sh.beta = 0.0;
        sh.done = done;
    }
    bar_sync_n(2, all);

    bool init = true;
    while (!done) {
        // after z = M^-1 r
        bar_sync_n(2, all);
        {
            const ResTerm<T> mine[2] = {gather(0), gather(1)};
            double tot[2], beta = 0.0;
            if (!res_totals<2, T>(sums, 1, mine, lane, tot) || sh.halo_failed) {
                status = GMAF_TIMEOUT;
                done = 1;
            } else {
                const double rz = tot[0], rr = tot[1];
                rr_last = rr;
                const bool fin = res_exp(rz) != 0x7ff && res_exp(rr) != 0x7ff;
                if (!init) {
                    ++iter;
                    // rz / d: the reciprocal was formed while the product ran
                    const double t = rz * d_inv;
                    beta = d_plain ? fma(d_inv, fma(-d, t, rz), t) : rz / d;
                } else if (q.mode == kResContinue) {
                    // a continued recurrence: u = z + beta u', the old direction in the new units
                    const double d_old = sc->d;
                    if (fin && finite_d(d_old) && d_old > 0.0 && q.cscale > 0.0)
                        beta = rz / (q.cscale * d_old);
                }
                if (zero_rhs) {
                    converged = 1;
                    done = 1;
                } else if (!fin) {
                    status = GMAF_NONFINITE;
                    done = 1;
                } else if (__double_as_longlong(rr) <= thr2 && sqrt(rr) / normS <= q.eps) {
                    // (Eq. 3.9; the root and the quotient are formed only near the tolerance)
                    converged = 1;
                    done = 1;
                } else if (iter >= q.max_iter) {
                    done = 1;
                }
                if (init || !done) d = rz;
                // loop guard: never more products than iterations (a host-set limit can lower it)
                if (!init && guard > (q.guard_limit > 0 ? (long long)q.guard_limit
                                                        : (long long)q.max_iter + 4)) {
                    status = GMAF_TIMEOUT;
                    done = 1;
                }
            }
            if (lane == 0) {
                sh.beta = beta;
                sh.done = done;
            }
        }
        mark(init ? 2 : 1);
        if (timed && !init) q.times[4] += 1;
        bar_sync_n(2, all);
        if (done) break;
        init = false;
        d_inv = 1.0 / d;
        d_plain = res_exp(d) > 100 && res_exp(d) < 1940;

        // after v = A u
        bar_sync_n(2, all);
        {
            const ResTerm<T> mine[1] = {gather(0)};
            double tot[1];
            ++guard;
            if (!res_totals<1, T>(sums, 0, mine, lane, tot) || sh.halo_failed) {
                status = GMAF_TIMEOUT;
                done = 1;
            } else if (res_exp(tot[0]) == 0x7ff || __double_as_longlong(tot[0]) <= 0 || res_exp(d) == 0x7ff) {
                status = GMAF_NONFINITE;
                done = 1;
            } else {
                alpha = res_quotient(d, tot[0]);
            }
            if (lane == 0) {
                sh.alpha = alpha;
                sh.done = done;
            }
        }
        mark(0);
        if (timed) q.times[3] += 1;
        bar_sync_n(2, all);
    }
    if (lane == 0 && blk == g0) {
        sc->iter = iter;
        sc->d = d;
        sc->normS = normS;
        sc->rel = sqrt(rr_last) / normS;
        sc->alpha = alpha;
        sc->converged = converged;
        sc->status = status;
        sc->zero_rhs = zero_rhs;
        sc->pending = 0;
        sc->done = 1;
    }
}

// ------------------------------------------------------------------ the solve

// Dot products: FP64 adds to the accumulator directly, FP32 a row's VEC products first.
template <typename T>
struct ResAcc;
template <>
struct ResAcc<double> {
    double s[1] = {0.0};
    template <int VEC>
    __device__ __forceinline__ void add(const double (&a)[VEC], const double (&b)[VEC])
    {
#pragma unroll
        for (int e = 0; e < VEC; ++e) s[0] = fma(a[e], b[e], s[0]);
    }
    __device__ __forceinline__ double value() const { return s[0]; }
};
template <>
struct ResAcc<float> {
    Acc<float> s;
    template <int VEC>
    __device__ __forceinline__ void add(const float (&a)[VEC], const float (&b)[VEC])
    {
        float t = 0.0f;
#pragma unroll
        for (int e = 0; e < VEC; ++e) t += a[e] * b[e];
        s.add_sum(t);
    }
    __device__ __forceinline__ Acc<float> value() const { return s; }
};
template <typename T>
using ResSum = decltype(ResAcc<T>{}.value());

// CS: the coefficients in shared memory (else read from global memory, i.e. L2).
template <typename T, int VEC, int RR, bool CS>
__global__ void __launch_bounds__(kResThreads + 32, 1) k_resident(const __grid_constant__ ResParams<T> q)
{
    using V = Vec<T, VEC>;
    constexpr int S = kResThreads * VEC;            // private fields: [row][thread][VEC]
    constexpr int NS = kResSegs;
    constexpr bool RS = res_r_shared(RR, VEC, sizeof(T));
    constexpr int FE = RR * S, FN = 2 * RR * S, FI = 3 * RR * S, FD = 4 * RR * S;
    constexpr int FR = CS ? 5 * RR * S : RR * S;
    extern __shared__ __align__(16) unsigned char g_res_smem[];
    __shared__ ResShared<T> sh;
    const int nth = q.nth, nz = q.nz;
    const int cond = blockIdx.x / q.bpc, bc = blockIdx.x - cond * q.bpc;
    const int grp = q.groups == 1 ? 0 : cond;
    if (!((q.mask >> grp) & 1ull)) return;                 // this group does not run
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int TC = q.threads;                               // threads that own rows
    if (tid >= TC) {
        res_exchange_warp<T>(q, sh, q.sc + grp, q.groups == 1 ? 0 : cond * q.bpc,
                             q.groups == 1 ? (int)gridDim.x : q.bpc, lane);
        return;
    }
    const int all = TC + 32;
    const int j0 = (int)((long long)bc * nz / q.bpc), j1 = (int)((long long)(bc + 1) * nz / q.bpc);
    const int R = j1 - j0;
    const bool assor = q.precond == 1;

    // ---- this thread's columns and rows
    const int run = tid / q.P, cg = tid - run * q.P, c = cg * VEC;
    const int lr0 = run * RR;                               // first local row
    int nr = R - lr0;
    nr = cg >= q.ncg || nr < 0 ? 0 : (nr > RR ? RR : nr);
    const bool act = nr > 0;
    const bool bot = act && run == 0, top = act && lr0 + nr == R;
    const bool hasS = bot && j0 > 0, hasN = top && j1 < nz;    // a block below, above
    const bool segw = (cg & 31) == 0, sege = (cg & 31) == 31 || cg == q.ncg - 1;
    const bool atw = cg == 0, ate = cg == q.ncg - 1;
    const bool last = top && j1 == nz;                      // this run ends at row nz - 1
    const size_t off = (size_t)cond * (size_t)q.n + (size_t)(j0 + lr0) * nth + c;
    const size_t coff = (size_t)q.cslot[cond] * (size_t)q.n + (size_t)(j0 + lr0) * nth + c;

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
    const T *const pS = run == 0 ? HU + c : P - q.P * VEC + (RR - 1) * S;
    const T *const pN = top ? HU + nth + c : P + q.P * VEC;
    const T *const pW = sm + (run * q.P + (atw ? q.ncg - 1 : cg - 1)) * VEC + VEC - 1;
    const T *const pE = sm + (run * q.P + (ate ? 0 : cg + 1)) * VEC;
    T *const pX = q.o_x >= 0 ? reinterpret_cast<T *>(g_res_smem + q.o_x) + tid * VEC : q.p + off;
    const int stX = q.o_x >= 0 ? S : nth;

    auto get_E = [&](int rr, T(&x)[VEC]) { V::ldrw(CS ? P + FE + rr * S : q.aE + coff + (size_t)rr * nth, x); };
    auto get_N = [&](int rr, T(&x)[VEC]) { V::ldrw(CS ? P + FN + rr * S : q.aN + coff + (size_t)rr * nth, x); };
    auto get_I = [&](int rr, T(&x)[VEC]) { V::ldrw(CS ? P + FI + rr * S : q.invD + coff + (size_t)rr * nth, x); };
    auto get_D = [&](int rr, T(&x)[VEC]) { V::ldrw(CS ? P + FD + rr * S : q.D + coff + (size_t)rr * nth, x); };

    // rows of a block's halo area: 0, 1 = first and last row of v; 2, 3 = of z
    unsigned long long *const halo = q.halo + (size_t)blockIdx.x * 4 * q.halo_row + c * ((int)sizeof(T) / 4);
    unsigned ep = q.epoch;

    T rg[RS ? 1 : RR][VEC], vz[RR][VEC], aS0[VEC], hS[VEC], hN[VEC];
    auto r_get = [&](int rr, T(&x)[VEC]) {
        if constexpr (RS) {
            V::ldrw(P + FR + rr * S, x);
        } else {
#pragma unroll
            for (int e = 0; e < VEC; ++e) x[e] = rg[rr][e];
        }
    };
    auto r_put = [&](int rr, const T(&x)[VEC]) {
        if constexpr (RS) {
            V::st(P + FR + rr * S, x);
        } else {
#pragma unroll
            for (int e = 0; e < VEC; ++e) rg[rr][e] = x[e];
        }
    };
#pragma unroll
    for (int rr = 0; rr < RR; ++rr)
#pragma unroll
        for (int e = 0; e < VEC; ++e) vz[rr][e] = T(0);
#pragma unroll
    for (int e = 0; e < VEC; ++e) aS0[e] = hS[e] = hN[e] = T(0);

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
        if (hasS) ok = ll_get<VEC>(halo + (s - 4) * q.halo_row, hS, ep);
        if (hasN) ok = ll_get<VEC>(halo + (n + 4) * q.halo_row, hN, ep) && ok;
        if (!ok) sh.halo_failed = 1;
    };

    // ---- set-up: coefficients, r, x, u
    for (int i = tid; i < 2 * nth; i += TC) HU[i] = HR[i] = T(0);
    for (int i = tid; i < nth; i += TC) YR[i] = T(0);
    bar_sync_n(1, TC);
    ResAcc<T> acc0;
    if (act) {
#pragma unroll
        for (int rr = 0; rr < RR; ++rr) {
            if (rr >= nr) continue;
            const size_t go = (size_t)rr * nth;
            T t[VEC];
            V::ldrw(q.aE + coff + go, t);
            if (CS) V::st(P + FE + rr * S, t);
            if (sege) EY[er + rr * NS] = t[VEC - 1];
            if (CS) {
                V::ldrw(q.aN + coff + go, t);
                V::st(P + FN + rr * S, t);
                V::ldrw(q.invD + coff + go, t);
                V::st(P + FI + rr * S, t);
                V::ldrw(q.D + coff + go, t);
                V::st(P + FD + rr * S, t);
            }
            // r = b (- A p), or the residual handed in; x = 0 or p
            T x[VEC], r[VEC];
#pragma unroll
            for (int e = 0; e < VEC; ++e) x[e] = T(0);
            if (q.mode == kResRestart) {
                V::ldrw(q.r_in + off + go, r);
                V::ldrw(q.p + off + go, x);
            } else {
                V::ldrw(q.b + off + go, r);
                acc0.add(r, r);
                if (!q.zero_init) {
                    V::ldrw(q.p + off + go, x);
                    const int j = j0 + lr0 + rr;
                    const T *p = q.p + off + go, *aE = q.aE + coff + go, *aN = q.aN + coff + go;
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        const int ie = c + e == nth - 1 ? 1 - nth + e : e + 1, iw = c + e == 0 ? nth - 1 : e - 1;
                        T ap = q.D[coff + go + e] * x[e] - aE[e] * p[ie] - aE[iw] * p[iw];
                        if (j < nz - 1) ap -= aN[e] * p[nth + e];
                        if (j > 0) ap -= aN[e - nth] * p[e - nth];
                        r[e] -= ap;
                    }
                }
            }
            r_put(rr, r);
            // (in global memory p itself is x, and a neighbour may still be reading it)
            if (q.o_x >= 0 || (q.mode != kResRestart && q.zero_init)) V::st(pX + rr * stX, x);
#pragma unroll
            for (int e = 0; e < VEC; ++e) t[e] = T(0);
            if (q.mode == kResContinue) V::ldrw(q.u + off + go, t);
            V::st(P + rr * S, t);
            // the rows that the neighbours keep a copy of
            if (hasS && rr == 0) ll_put<VEC>(halo, r, ep + 1);
            if (hasN && rr == nr - 1) ll_put<VEC>(halo + q.halo_row, r, ep + 1);
        }
        if (j0 + lr0 > 0) V::ldrw(q.aN + coff - nth, aS0);
        if (hasS) {
            T t[VEC];
            V::ldrw(q.invD + coff - nth, t);
            V::st(HI + c, t);
            if (q.mode == kResContinue) {
                V::ldrw(q.u + off - nth, t);
                V::st(HU + c, t);
            }
        }
        if (hasN) {
            T t[VEC];
            const size_t go = (size_t)nr * nth;
            V::ldrw(q.invD + coff + go, t);
            V::st(HI + nth + c, t);
            V::ldrw(q.aE + coff + go, t);
            V::st(HE + c, t);
            if (sege) EY[er + nr * NS] = t[VEC - 1];
            if (q.mode == kResContinue) {
                V::ldrw(q.u + off + go, t);
                V::st(HU + nth + c, t);
            }
        }
    }

    // exchange 0: b.b, and r on the halo rows
    publish(acc0.value());
    ++ep;
    fetch(1, 0);
    bar_sync_n(2, all);

    bool init = true;
    while (!sh.done) {
        // ------------------------------------------------ B: r -= alpha v; z = M^-1 r
        const T alpha = (T)sh.alpha;
        ResAcc<T> arz, arr;
        ++ep;
        T yN[VEC];
#pragma unroll
        for (int e = 0; e < VEC; ++e) yN[e] = T(0);
#pragma unroll
        for (int rr = 0; rr < RR; ++rr) {
            if (rr >= nr) continue;
            T od[VEC], r[VEC];
            get_I(rr, od);
            r_get(rr, r);
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                r[e] -= alpha * vz[rr][e];
                vz[rr][e] = r[e] * od[e];
            }
            r_put(rr, r);
            if (rr == RR - 1 && !top) V::st(YR + (run + 1) * nth + c, vz[rr]);
            if (sege) EY[rr * NS] = vz[rr][VEC - 1];
            if (atw) EC[2 * rr] = vz[rr][0];
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
        if (assor) {
            bar_sync_n(1, TC);
            // first sweep (Eq. 3.5): w = y + omega/D (lower couplings of y)
            T yp[VEC], nS[VEC], wN[VEC];
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                yp[e] = wN[e] = T(0);
                nS[e] = aS0[e];
            }
            if (act) V::ldrw(YR + run * nth + c, yp);
#pragma unroll
            for (int rr = 0; rr < RR; ++rr) {
                T ev[VEC];
#pragma unroll
                for (int e = 0; e < VEC; ++e) ev[e] = T(0);
                if (rr < nr) get_E(rr, ev);
                T yW = __shfl_up_sync(0xffffffffu, vz[rr][VEC - 1], 1);
                T aW = __shfl_up_sync(0xffffffffu, ev[VEC - 1], 1);
                if (rr < nr) {
                    if (segw && !atw) {
                        yW = EYl[rr * NS];
                        aW = EYl[er + rr * NS];
                    }
                    T w[VEC], od[VEC];
                    get_I(rr, od);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        T sum = nS[e] * yp[e];
                        if (e > 0)
                            sum += ev[e - 1] * vz[rr][e - 1];
                        else if (!atw)
                            sum += aW * yW;
                        if (e == VEC - 1 && ate) sum += ev[e] * EC[2 * rr];
                        w[e] = vz[rr][e] + od[e] * sum;
                    }
                    if (rr == 0 && run > 0) V::st(WR + (run - 1) * nth + c, w);
                    if (segw) EY[2 * er + rr * NS] = w[0];
                    if (ate) EC[2 * rr + 1] = w[VEC - 1];
                    get_N(rr, nS);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        yp[e] = vz[rr][e];
                        vz[rr][e] = w[e];
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
            }
            bar_sync_n(1, TC);
            // second sweep (Eq. 3.6 without its factor): z = w + omega/D (upper couplings of w)
            if (act && !top) V::ldrw(WR + run * nth + c, wN);
#pragma unroll
            for (int rr = RR - 1; rr >= 0; --rr) {
                T wE = __shfl_down_sync(0xffffffffu, vz[rr][0], 1);
                if (rr < nr) {
                    T ev[VEC], od[VEC], nv[VEC], z[VEC], r[VEC];
                    r_get(rr, r);
                    get_E(rr, ev);
                    get_I(rr, od);
                    get_N(rr, nv);
                    if (sege && !ate) wE = EWr[rr * NS];
                    const bool north = !(last && rr == nr - 1);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        T sum = north ? nv[e] * wN[e] : T(0);
                        if (e < VEC - 1)
                            sum += ev[e] * vz[rr][e + 1];
                        else if (!ate)
                            sum += ev[e] * wE;
                        if (e == 0 && atw) sum += EYl[er + rr * NS] * EC[2 * rr + 1];
                        z[e] = vz[rr][e] + od[e] * sum;
                    }
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        wN[e] = vz[rr][e];
                        vz[rr][e] = z[e];
                    }
                    if (hasS && rr == 0) ll_put<VEC>(halo + 2 * q.halo_row, z, ep);
                    if (hasN && rr == nr - 1) ll_put<VEC>(halo + 3 * q.halo_row, z, ep);
                    arz.add(r, z);
                    arr.add(r, r);
                }
            }
        } else {
#pragma unroll
            for (int rr = 0; rr < RR; ++rr) {
                if (rr >= nr) continue;
                T r[VEC];
                r_get(rr, r);
                if (hasS && rr == 0) ll_put<VEC>(halo + 2 * q.halo_row, vz[rr], ep);
                if (hasN && rr == nr - 1) ll_put<VEC>(halo + 3 * q.halo_row, vz[rr], ep);
                arz.add(r, vz[rr]);
                arr.add(r, r);
            }
        }
        publish2(arz.value(), arr.value());
        // x += alpha u, and z on the neighbours' rows, while the sums travel
        if (!init) {
#pragma unroll
            for (int rr = 0; rr < RR; ++rr) {
                if (rr >= nr) continue;
                T x[VEC], u[VEC];
                V::ldrw(pX + rr * stX, x);
                V::ldrw(P + rr * S, u);
#pragma unroll
                for (int e = 0; e < VEC; ++e) x[e] += alpha * u[e];
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
#pragma unroll
        for (int rr = 0; rr < RR; ++rr) {
            if (rr >= nr) continue;
            T u[VEC];
            V::ldrw(P + rr * S, u);
#pragma unroll
            for (int e = 0; e < VEC; ++e) u[e] = vz[rr][e] + beta * u[e];
            V::st(P + rr * S, u);
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
        bar_sync_n(1, TC);
        T us[VEC], uc[VEC], nS[VEC];
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            us[e] = uc[e] = T(0);
            nS[e] = aS0[e];
        }
        if (act) {
            V::ldrw(pS, us);
            V::ldrw(P, uc);
        }
#pragma unroll
        for (int rr = 0; rr < RR; ++rr) {
            T ev[VEC];
#pragma unroll
            for (int e = 0; e < VEC; ++e) ev[e] = T(0);
            if (rr < nr) get_E(rr, ev);
            T uW = __shfl_up_sync(0xffffffffu, uc[VEC - 1], 1);
            T uE = __shfl_down_sync(0xffffffffu, uc[0], 1);
            T aW = __shfl_up_sync(0xffffffffu, ev[VEC - 1], 1);
            if (rr < nr) {
                T un[VEC], nv[VEC], D[VEC];
                V::ldrw(rr == RR - 1 || rr == nr - 1 ? pN : P + (rr + 1) * S, un);
                get_N(rr, nv);
                get_D(rr, D);
                if (segw) {
                    uW = pW[rr * S];
                    aW = EYl[er + rr * NS];
                }
                if (sege) uE = pE[rr * S];
                if (last && rr == nr - 1) {
#pragma unroll
                    for (int e = 0; e < VEC; ++e) nv[e] = T(0);
                }
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    const T xE = e < VEC - 1 ? uc[e + 1] : uE;
                    const T xW = e > 0 ? uc[e - 1] : uW;
                    const T a = e > 0 ? ev[e - 1] : aW;
                    vz[rr][e] = D[e] * uc[e] - ev[e] * xE - a * xW - nv[e] * un[e] - nS[e] * us[e];
                }
                auv.add(uc, vz[rr]);
                if (hasS && rr == 0) ll_put<VEC>(halo, vz[rr], ep);
                if (hasN && rr == nr - 1) ll_put<VEC>(halo + q.halo_row, vz[rr], ep);
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    us[e] = uc[e];
                    uc[e] = un[e];
                    nS[e] = nv[e];
                }
            }
        }
        publish(auv.value());
        fetch(1, 0);
        bar_sync_n(2, all);
    }

    // ---- the solution, and the direction of a run to be continued
#pragma unroll
    for (int rr = 0; rr < RR; ++rr) {
        if (rr >= nr) continue;
        T t[VEC];
        if (q.o_x >= 0) {
            V::ldrw(pX + rr * stX, t);
            V::st(q.p + off + (size_t)rr * nth, t);
        }
        if (q.u) {
            V::ldrw(P + rr * S, t);
            V::st(q.u + off + (size_t)rr * nth, t);
        }
    }
}

}  // namespace gmaf
