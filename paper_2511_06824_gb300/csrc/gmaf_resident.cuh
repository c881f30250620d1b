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
// blocks are resident (cooperative launch), but other work on the GPU may keep some of
// them from running.  A wait that is not met after ResParams::polls polls (of about a
// microsecond) ends the run with kResLate, and the phase kernels, whose blocks wait for
// nothing, take the system.  A block that gives up adds no more sums, so the others give up
// too; where it did so in the last exchange of theirs, what they found is measured by the FP64
// residual after all, in mixed precision by the next one of the run, which is not formed without
// it.
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
// Polls until every word carries ep, `polls` times at most; false if that never happened.
template <int VEC>
__device__ __forceinline__ bool ll_get(const unsigned long long *p, float (&x)[VEC], unsigned ep, unsigned polls)
{
    for (unsigned k = 0; k < polls; ++k) {
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
__device__ __forceinline__ bool ll_get(const unsigned long long *p, double (&x)[VEC], unsigned ep, unsigned polls)
{
    for (unsigned k = 0; k < polls; ++k) {
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
// the warp's butterfly.  Across warps and blocks a value is an integer in two limbs (42
// bits and the rest), scaled so that the total expected (the last total of its kind) has
// 71 bits.  A warp's term may have 76; a total that shrank below 2^-8 of the expected one
// is formed again, as each warp's term is cut off at the lowest bit (FP32: both its parts)
// and all of them together may be short by 2^12.4 of it: 2^-49 of a total of 63 bits.  Then,
// and the first time, the blocks first agree on the largest exponent among their terms.

constexpr int kResTop = 70;             // bit of the leading digit of the expected total
constexpr int kResTermBits = 76;        // most bits of a term
constexpr int kResShrink = 8;           // most bits by which a total may fall short of the expected one
constexpr int kResLimb = 42;            // bits of the low limb
constexpr unsigned long long kResLimbMask = (1ull << kResLimb) - 1;
// Words of the exchange: the low limb beside a count of 8 bits, the rest beside two.  The sum over
// all blocks and warps (of FP32's two parts each) has to fit, with its sign.
constexpr long long kResTerms = 2ll * kResMaxBlocks * (kResThreads / 32);
static_assert(kResMaxBlocks < 256, "blocks are counted in a byte");
static_assert(kResTerms < 1ll << (55 - kResLimb), "low limbs");
static_assert(kResTerms < 1ll << (47 - (kResTermBits - kResLimb)), "high limbs");
// (and within a block, added up in pieces of 24 bits of 32 by integer reductions over a warp)
static_assert(kResTermBits - kResLimb - 24 < 26 && kResLimb - 24 < 26, "limbs of a block");

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
    for (int q = 0; q < NV; ++q) {
        // (1 where there are subnormal numbers only, whose sum is not formed: see res_totals)
        const bool some = (((unsigned)__double2hiint(x[q]) << 1) | (unsigned)__double2loint(x[q])) != 0u;
        e[q] = __reduce_max_sync(0xffffffffu, max(res_exp(x[q]), some ? 1 : 0));
    }
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

// The biased exponent (as of a double) of a term's leading bit; 0: zero, 1: perhaps less than that
// exponent, 0x7ff: not finite.
__device__ __forceinline__ int res_term_exp(const ResTerm<double> &t)
{
    if (t.e == 0x7ff) return 0x7ff;
    if (t.v == 0) return t.e == 1 ? 1 : 0;
    return max(1, t.e - 54 + 63 - __clzll(t.v < 0 ? -t.v : t.v));
}
__device__ __forceinline__ int res_term_exp(const ResTerm<float> &t)
{
    const int e = (__float_as_uint(t.hi) >> 23) & 0xff;
    return e == 0 ? (t.hi != 0.0f ? 1 : 0) : (e == 0xff ? 0x7ff : e + 896);
}

struct ResLimbs {
    long long lo, top;
    bool over;                          // too large for the scale
};
// m 2^up in units of the lowest bit (m of `bits` bits), added with its sign.
__device__ __forceinline__ void res_limbs_add(ResLimbs &x, unsigned long long m, int up, bool neg, int bits)
{
    const bool over = (up + bits > kResTermBits || up > 63) && m != 0;
    const int left = min(max(up, 0), 63);
    m = over ? 0ull : m >> min(max(-up, 0), 63);
    const unsigned long long low = m << left, high = left ? m >> (64 - left) : 0ull;
    const long long lo = (long long)(low & kResLimbMask);
    const long long top = (long long)((low >> kResLimb) | (high << (64 - kResLimb)));
    x.over = x.over || over;
    x.lo += neg ? -lo : lo;
    x.top += neg ? -top : top;
}
// (top 2^kResLimb + lo) 2^(e - 1023 - kResTop), the lowest bit's weight, rounded to a double.
__device__ __forceinline__ double res_value(long long top, long long lo, int e)
{
    top += lo >> kResLimb;
    unsigned long long l = (unsigned long long)lo & kResLimbMask;
    const bool neg = top < 0;
    unsigned long long h = (unsigned long long)top;
    if (neg) {
        h = 0ull - h - (l != 0);
        l = (0ull - l) & kResLimbMask;
    }
    // the leading 64 bits, the leading one on top
    const int hz = __clzll(h), lz = __clzll(l);
    const bool big = h != 0;
    unsigned long long m = big ? (hz >= kResLimb ? (h << hz) | (l << (hz - kResLimb))
                                                 : (h << hz) | (l >> (kResLimb - hz)))
                               : l << (lz & 63);
    int lead = big ? kResLimb + 63 - hz : 63 - lz;
    if (!big && l == 0) return 0.0;
    const unsigned long long r = m + 1024ull;            // to nearest
    if (r < m) ++lead;
    const unsigned long long bits = ((unsigned long long)(lead + e - kResTop) << 52) |
                                    ((r < m ? 0ull : r >> 11) & 0xfffffffffffffull);
    return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0ull)));
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

enum ResWord { kWordUV = 0, kWordRZ = 4, kWordMaxCount = 8, kWordMax = 9, kWordMeet = 11, kWordR64 = 12 };
static_assert(kWordR64 + 4 <= kResGroupWords, "words of a group");

struct ResSums {
    unsigned long long *w;              // the group's words (zero at the start of the run)
    unsigned long long prev[10], prev_max, prev_meet;
    int nb, e[5];                       // blocks; exponent expected of u.v, r.z, r.r, and of
                                        // r.r and S.S in FP64 (0: not known)
    unsigned turn;
};

__device__ __forceinline__ void res_red(unsigned long long *p, unsigned long long v)
{
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;\n" ::"l"(p), "l"(v) : "memory");
}

// The largest exponent of each of NV values over the group's blocks.
template <int NV>
__device__ __forceinline__ bool res_max_exp(ResSums &x, const int (&mine)[NV], int *e, int lane, unsigned polls)
{
    ++x.turn;
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < NV; ++q)
            atomicMax(x.w + kWordMax + q, ((unsigned long long)x.turn << 16) | (unsigned)mine[q]);
        __threadfence();
        res_red(x.w + kWordMaxCount, 1ull);
    }
    // (all lanes leave together: the caller goes on with operations of the whole warp)
    for (unsigned k = 0; k < polls; ++k) {
        if (__any_sync(0xffffffffu, ll_ld1(x.w + kWordMaxCount) - x.prev_max == (unsigned long long)x.nb)) {
            x.prev_max += (unsigned long long)x.nb;
            __threadfence();
#pragma unroll
            for (int q = 0; q < NV; ++q) e[q] = (int)(ll_ld1(x.w + kWordMax + q) & 0xffffull);
            return true;
        }
    }
    return false;
}

// All blocks of the group have come, and what their threads stored before is visible.
__device__ __forceinline__ bool res_meet(ResSums &x, int lane, unsigned polls)
{
    __threadfence();
    __syncwarp();
    if (lane == 0) res_red(x.w + kWordMeet, 1ull);
    bool ok = false;
    for (unsigned k = 0; k < polls && !ok; ++k)
        ok = ll_ld1(x.w + kWordMeet) - x.prev_meet == (unsigned long long)x.nb;
    x.prev_meet += (unsigned long long)x.nb;
    __threadfence();
    return __all_sync(0xffffffffu, ok) != 0;
}

// The totals over the group's blocks of NV values, of which each lane holds one term (in every
// lane).  Returns 0, kResLate if some block never came, or kResBeyond if the terms of a value
// leave the range of exponents that the fixed-point numbers are formed in, 2^-942 to 2^1006 (zero
// and what is not finite do not: they give 0 and NaN).
constexpr int kResMinExp = 80, kResMaxExp = 2030;

template <int NV, typename T>
__device__ __forceinline__ int res_totals(ResSums &x, int kind, const ResTerm<T> (&term)[NV], int lane,
                                          unsigned polls, double (&tot)[NV])
{
    // kind 0: u.v; 1: r.z and r.r; 2: the FP64 residual's and source's
    unsigned long long *const w = x.w + (kind == 0 ? kWordUV : kind == 1 ? kWordRZ : kWordR64);
    unsigned long long *prev = x.prev + (kind == 0 ? 0 : kind == 1 ? 2 : 6);
    int *e = x.e + (kind == 0 ? 0 : kind == 1 ? 1 : 3);
    bool known = true;
#pragma unroll
    for (int q = 0; q < NV; ++q) known = known && e[q] != 0;
    for (int turn = 0; turn < 2; ++turn) {
        if (!known) {
            int ex[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) ex[q] = __reduce_max_sync(0xffffffffu, res_term_exp(term[q]));
            if (!res_max_exp<NV>(x, ex, e, lane, polls)) return kResLate;
#pragma unroll
            for (int q = 0; q < NV; ++q)
                if ((e[q] > 0 && e[q] <= kResMinExp) || (e[q] >= kResMaxExp && e[q] < 0x7ff)) return kResBeyond;
        }
        int en[NV];
        unsigned long long word = 0;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            en[q] = e[q] > kResMinExp && e[q] < kResMaxExp ? e[q] : 1023;
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
        for (unsigned k = 0; k < polls && !ok; ++k) {
            bool mine = true;
#pragma unroll
            for (int q = 0; q < NV; ++q) ll_ld2(w + 2 * q, d[2 * q], d[2 * q + 1]);
#pragma unroll
            for (int q = 0; q < 2 * NV; ++q)
                mine = mine && ((d[q] - prev[q]) & 0xffull) == (unsigned long long)x.nb;
            ok = __all_sync(0xffffffffu, mine);
        }
        if (!ok) return kResLate;
        bool good = true;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const long long lo = (long long)(d[2 * q] - prev[2 * q]) >> 8;
            const unsigned long long t = d[2 * q + 1] - prev[2 * q + 1];
            tot[q] = res_value((long long)t >> 16, lo, en[q]);
            good = good && ((t >> 8) & 0xffull) == 0 && res_exp(tot[q]) >= e[q] - kResShrink;
            prev[2 * q] = d[2 * q];
            prev[2 * q + 1] = d[2 * q + 1];
        }
        if (!known || good) {
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                if (e[q] == 0) tot[q] = 0.0;
                if (e[q] == 0x7ff) tot[q] = __longlong_as_double(0x7ff8000000000000ll);
                // (what the next total of the kind is expected to be)
                e[q] = res_exp(tot[q]);
                if (e[q] <= kResMinExp || e[q] >= kResMaxExp) e[q] = 0;
            }
            return 0;
        }
        known = false;
    }
    return kResLate;
}

// Whether ||r||^2 stays in that range down to the tolerance (or to 1e-20, which no residual
// reaches): bb is ||b||^2.  If not, the phase kernels take the system from the start.
__device__ __forceinline__ bool res_in_range(double bb, double eps)
{
    return bb == 0.0 || res_exp(bb) + 2 * (max(res_exp(eps), 1023 - 67) - 1023) > kResMinExp + 40;
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

// Sums and products are written out as fused operations in the order of the phase kernels
// (gmaf_pcg_kernels.cuh), so that an FP32 run passes through their numbers: only the sums over
// the grid, which every scalar is rounded from, are added in another order.  A stopped
// refinement leaves rounding of 1e-13 in a solution, which a finite-difference Jacobian
// magnifies by 1e4: it must not depend on which kernels a grid takes.  (Left to the compiler,
// the two sweeps' sums were fused the other way round; on 9 conditions of 512 x 256 cells the
// Jacobian moved by up to 2.4e-9.)
__device__ __forceinline__ float res_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float res_fnma(float a, float b, float c) { return __fmaf_rn(-a, b, c); }
__device__ __forceinline__ float res_diff(float a, float b, float c, float d) { return __fmaf_rn(a, b, -__fmul_rn(c, d)); }
// (FP64 keeps the compiler's choice: it leaves no such trace)
__device__ __forceinline__ double res_fma(double a, double b, double c) { return a * b + c; }
__device__ __forceinline__ double res_fnma(double a, double b, double c) { return c - a * b; }
__device__ __forceinline__ double res_diff(double a, double b, double c, double d) { return a * b - c * d; }

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
    ResTerm<T> part[2][kResThreads / 32];           // the warps' sums
    ResTerm<double> part64[2][kResThreads / 32];    // (of the FP64 residual)
    double alpha, beta;
    double red64[kThreads / 32];        // (norm of the FP64 residual)
    double unit, back;                  // mixed precision: 1 / ||r64||; scale ||r64||, which takes x to p
    int done, stop, halo_failed;        // done: 1 converged, 2 not
};

// Before the threads part: row threads may find a halo row missing before the exchange warp runs.
template <typename T>
__device__ __forceinline__ void res_clear(ResShared<T> &sh)
{
    if (threadIdx.x == 0) sh.done = sh.stop = sh.halo_failed = 0;
    __syncthreads();
}

// (one object per block: a function's own shared variable)
template <typename T>
__device__ __forceinline__ ResShared<T> &res_shared()
{
    __shared__ ResShared<T> sh;
    return sh;
}

// The warp that takes no rows: adds the block's sums, exchanges them, updates the
// scalars (finish_a and finish_b of the phase kernels) and decides when to stop.
// NORM: ||r64|| in k_resid64's order (res_norm_warps).
template <typename T, bool NORM>
struct ResExchange {
    const ResParams<T> &q;
    ResShared<T> &sh;
    const int all, warps, lane;
    ResSums sums;
    int iter, status, converged, zero_rhs, done;
    double d, normS, rr_last, alpha;
    bool timed;
    unsigned long long t_mark;

    __device__ __forceinline__ void mark(int k)
    {
        if (!timed) return;
        const unsigned long long t = res_time();
        q.times[k] += t - t_mark;
        t_mark = t;
    }
    __device__ __forceinline__ ResTerm<T> gather(int w) const
    {
        ResTerm<T> t{};
        if (lane < warps) t = sh.part[w][lane];
        return t;
    }
    __device__ __forceinline__ ResTerm<double> gather64(int w) const
    {
        ResTerm<double> t{};
        if (lane < warps) t = sh.part64[w][lane];
        return t;
    }

    // Limit of this warp's waits: constant in FP32 (as a parameter it cost k_resident_s<float> 4 %:
    // 15.3 -> 15.9 us an iteration on 9 conditions of 640 x 200 cells).
    __device__ __forceinline__ unsigned polls() const { return sizeof(T) == 4 ? kResPolls : q.polls; }
    // res_totals; kResLate if a row of a neighbour is missing.
    template <int NV, typename U>
    __device__ __forceinline__ int totals(int kind, const ResTerm<U> (&mine)[NV], double (&tot)[NV])
    {
        const int got = res_totals<NV, U>(sums, kind, mine, lane, polls(), tot);
        return got ? got : sh.halo_failed ? kResLate : 0;
    }

    // One PCG run from the residual that the row threads hold, to ||r|| <= eps normS or
    // max_iter (of the running count).  cscale > 0: a continued recurrence (mixed
    // precision), whose old direction is cscale times smaller in the new units.
    __device__ __forceinline__ void run(double eps, int max_iter, double cscale)
    {
        const double thr = eps * normS;
        // a little above (eps ||b||)^2, compared as integers (r.r is not negative)
        const long long thr2 = __double_as_longlong(thr * thr * (1.0 + 1e-10));
        double d_inv = 0.0;
        bool d_plain = false, init = true;
        int guard = 0;
        while (!done) {
            // after z = M^-1 r
            bar_sync_n(2, all);
            {
                const ResTerm<T> mine[2] = {gather(0), gather(1)};
                double tot[2], beta = 0.0;
                const int got = totals<2, T>(1, mine, tot);
                if (got) {
                    status = got;
                    done = 2;
                } else {
                    const double rz = tot[0], rr = tot[1];
                    rr_last = rr;
                    const bool fin = res_exp(rz) != 0x7ff && res_exp(rr) != 0x7ff;
                    if (!init) {
                        ++iter;
                        // rz / d: the reciprocal was formed while the product ran
                        const double t = rz * d_inv;
                        beta = d_plain ? fma(d_inv, fma(-d, t, rz), t) : rz / d;
                    } else if (cscale > 0.0) {
                        // u = z + beta u', the old direction in the new units
                        if (fin && finite_d(d) && d > 0.0) beta = rz / (cscale * d);
                    }
                    if (zero_rhs) {
                        converged = 1;
                        done = 1;
                    } else if (!fin) {
                        status = GMAF_NONFINITE;
                        done = 2;
                    } else if (__double_as_longlong(rr) <= thr2 && sqrt(rr) / normS <= eps) {
                        // (Eq. 3.9; the root and the quotient are formed only near the tolerance)
                        converged = 1;
                        done = 1;
                    } else if (iter >= max_iter) {
                        done = 2;
                    }
                    if (init || !done) d = rz;
                    // loop guard: never more products than iterations (a host-set limit can lower it)
                    if (!init && guard > (q.guard_limit > 0 ? (long long)q.guard_limit
                                                            : (long long)max_iter + 4)) {
                        status = GMAF_TIMEOUT;
                        done = 2;
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
                const int got = totals<1, T>(0, mine, tot);
                if (got) {
                    status = got;
                    done = 2;
                } else if (res_exp(tot[0]) == 0x7ff || __double_as_longlong(tot[0]) <= 0 ||
                           res_exp(d) == 0x7ff) {
                    status = GMAF_NONFINITE;
                    done = 2;
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
    }

    // FP64: one run (Table 1, or its restart).
    __device__ __forceinline__ void solve(Scalars *sc)
    {
        iter = q.mode == kResRestart ? sc->iter : 0;
        normS = q.mode == kResRestart ? sc->normS : 0.0;
        // exchange 0: b.b (and r on the halo rows)
        bar_sync_n(2, all);
        {
            const ResTerm<T> mine[1] = {gather(0)};
            double tot[1];
            const int got = totals<1, T>(0, mine, tot);
            sums.e[0] = 0;
            if (got) {
                status = got;
                done = 2;
            } else if (q.mode != kResRestart) {
                normS = sqrt(tot[0]);
                zero_rhs = tot[0] == 0.0;
                if (!finite_d(tot[0])) {
                    status = GMAF_NONFINITE;
                    done = 2;
                } else if (!res_in_range(tot[0], q.eps)) {
                    status = kResBeyond;
                    done = 2;
                }
            }
        }
        if (lane == 0) {
            sh.alpha = sh.beta = 0.0;
            sh.done = done;
        }
        bar_sync_n(2, all);
        run(q.eps, q.max_iter, 0.0);
    }

    // Mixed precision: FP64 refinement around the FP32 run (the loop of solve_joint_device).
    __device__ __forceinline__ void refine(Scalars *sc)
    {
        const double scale = *q.scale;
        int total = 0, outer = 0, longest = 0, last_iter = 0, verdict = GMAF_NOT_CONVERGED;
        bool stalled = false, stop = false;
        double rnorm_prev = 0.0, true_rel = 0.0;
        for (;;) {
            // after r64 = S - A p64
            bar_sync_n(2, all);
            double cscale = 0.0, eps_in = 0.5, rnorm = 0.0;
            int max_iter = 0;
            {
                const ResTerm<double> mine[2] = {gather64(0), gather64(1)};
                double tot[2];
                int got = sh.halo_failed ? kResLate : totals<2, double>(2, mine, tot);
                // ||r64|| in the order of k_resid64, to the last bit: it is the unit of the FP32
                // run and the factor of x in p (see res_norm_warps)
                double nn = tot[0];
                if constexpr (NORM) {
                    if (!got && !res_meet(sums, lane, polls())) got = kResLate;
                    bar_sync_n(2, all);
                    bar_sync_n(2, all);
                    if (!got && !res_meet(sums, lane, polls())) got = kResLate;
                    bar_sync_n(2, all);
                    bar_sync_n(2, all);
                    nn = 0.0;
                    for (int w = 0; w < kThreads / 32; ++w) nn += sh.red64[w];
                }
                rnorm = sqrt(nn);
                if (got) {
                    verdict = got;
                    stop = true;
                } else {
                    const double nS = sqrt(tot[1]);
                    true_rel = nS > 0.0 ? rnorm / nS : 0.0;
                    if (!finite_d(tot[0]) || !finite_d(tot[1]) || !finite_d(true_rel)) {
                        verdict = GMAF_NONFINITE;
                        stop = true;
                    } else if (outer == 0 && !res_in_range(tot[1], q.eps)) {
                        verdict = kResBeyond;
                        stop = true;
                    } else if (nS == 0.0 || true_rel <= q.eps) {
                        verdict = GMAF_OK;
                        stop = true;
                    } else if (stop || outer >= q.max_outer || total >= q.max_iter) {
                        stop = true;
                    } else {
                        // a fixed reduction, but no further than the outer target needs
                        eps_in = fmin(fmax(0.5 * q.eps / true_rel, q.inner_floor), 0.5);
                        const bool cont = outer > 0 && q.continued && rnorm_prev > 0.0 && !stalled;
                        // a continued run that needs more than max(1000, 4 x the longest so
                        // far) is cut off, and the next one restarts from its residual
                        const int left = q.max_iter - total, cap = max(1000, 4 * longest);
                        if (!cont) iter = last_iter = 0;
                        max_iter = cont ? last_iter + min(left, cap) : left;
                        cscale = cont ? rnorm_prev / rnorm : 0.0;
                        rnorm_prev = rnorm;
                    }
                }
            }
            done = status = converged = 0;
            normS = 1.0;                // b is r64 / ||r64||
            if (lane == 0) {
                sh.alpha = sh.beta = 0.0;
                sh.unit = 1.0 / rnorm;
                sh.back = scale * rnorm;
                sh.done = 0;
                sh.stop = stop;
            }
            mark(5);
            if (timed) q.times[6] += 1;
            bar_sync_n(2, all);
            if (stop) break;
            // the scales of the sums change with the units
            if (cscale == 0.0) sums.e[0] = sums.e[1] = sums.e[2] = 0;
            run(eps_in, max_iter, cscale);
            const int seg = iter - last_iter;
            last_iter = iter;
            total += seg;
            longest = max(longest, seg);
            stalled = q.continued && !converged;
            ++outer;
            if (status != 0) verdict = status;
            if (lane == 0 && status == kResLate) sh.halo_failed = 1;    // (the row threads wait no further)
            stop = status != 0 || seg == 0;     // (the row threads still add x to p)
            if (stop) {
                for (int k = 0; k < (NORM ? 5 : 1); ++k) bar_sync_n(2, all);    // the residual's sums: not wanted
                if (lane == 0) sh.stop = 1;
                bar_sync_n(2, all);
                break;
            }
        }
        if (lane == 0 && blockIdx.x == 0) {
            sc->iter = total;
            sc->guard = outer;
            sc->status = verdict;
            sc->true_rel = true_rel;
        }
    }
};

template <typename T, bool NORM = true>
__device__ __forceinline__ void res_exchange_warp(const ResParams<T> &q, ResShared<T> &sh, Scalars *sc,
                                                  int grp, int g0, int nb, int lane)
{
    ResExchange<T, NORM> x{q, sh, q.threads + 32, q.threads / 32, lane};
    x.sums = ResSums{};
    x.sums.w = q.words + (size_t)grp * kResGroupWords;
    x.sums.nb = nb;
    x.iter = x.status = x.converged = x.zero_rhs = x.done = 0;
    x.d = x.normS = x.rr_last = x.alpha = 0.0;
    x.timed = q.times != nullptr && lane == 0 && blockIdx.x == 0;
    x.t_mark = x.timed ? res_time() : 0ull;
    if constexpr (sizeof(T) == 4) {
        x.refine(sc);
    } else {
        x.solve(sc);
        if (lane == 0 && (int)blockIdx.x == g0) {
            sc->iter = x.iter;
            sc->d = x.d;
            sc->normS = x.normS;
            sc->rel = sqrt(x.rr_last) / x.normS;
            sc->alpha = x.alpha;
            sc->converged = x.converged;
            sc->status = x.status;
            sc->zero_rhs = x.zero_rhs;
            sc->pending = 0;
            sc->done = 1;
        }
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
        for (int e = 0; e < VEC; ++e) t = res_fma(a[e], b[e], t);
        s.add_sum(t);
    }
    __device__ __forceinline__ Acc<float> value() const { return s; }
};
template <typename T>
using ResSum = decltype(ResAcc<T>{}.value());

// What a thread that owns rows works on.  Built anew for each part of a mixed-precision
// solve, and set-up and residual are not inlined: the iterations would otherwise pay
// registers for values that live across them.
// CS: the coefficients in shared memory (else read from global memory, i.e. L2).
template <typename T, int VEC, int RR, bool CS>
struct ResRows {
    using V = Vec<T, VEC>;
    static constexpr int S = kResThreads * VEC;     // private fields: [row][thread][VEC]
    static constexpr int NS = kResSegs;
    static constexpr int FE = RR * S, FN = 2 * RR * S, FI = 3 * RR * S, FD = 4 * RR * S;

    const ResParams<T> &q;
    ResShared<T> &sh;
    int nth, nz, TC, tid, lane, wid;
    int j0, run, cg, c, lr0, nr;                    // the block's first row; first local row and rows of the run
    bool act, top, hasS, hasN;                      // rows at all; the block's last rows; a block below, above
    bool segw, sege, atw, ate, last;                // edges of a segment, of the row; the run ends at row nz - 1
    size_t off, coff;                               // first cell in the fields, in the coefficient slots
    // shared memory that setup() fills, laid out as res_iterate describes it
    T *P, *HU, *HR, *HI, *HE, *YR, *EY;
    int er;

    __device__ __forceinline__ ResRows(const ResParams<T> &q_, ResShared<T> &sh_) : q(q_), sh(sh_)
    {
        extern __shared__ __align__(16) unsigned char g_res_smem[];
        nth = q.nth;
        nz = q.nz;
        TC = q.threads;
        // (volatile: formed anew where it is used, not kept in registers across refinements)
        asm volatile("mov.u32 %0, %%tid.x;\n" : "=r"(tid));
        lane = tid & 31;
        wid = tid >> 5;
        const int cond = blockIdx.x / q.bpc, bc = blockIdx.x - cond * q.bpc;
        j0 = (int)((long long)bc * nz / q.bpc);
        const int j1 = (int)((long long)(bc + 1) * nz / q.bpc), R = j1 - j0;
        run = tid / q.P;
        cg = tid - run * q.P;
        c = cg * VEC;
        lr0 = run * RR;
        nr = R - lr0;
        nr = cg >= q.ncg || nr < 0 ? 0 : (nr > RR ? RR : nr);
        act = nr > 0;
        top = act && lr0 + nr == R;
        hasS = act && run == 0 && j0 > 0;
        hasN = top && j1 < nz;
        segw = (cg & 31) == 0;
        sege = (cg & 31) == 31 || cg == q.ncg - 1;
        atw = cg == 0;
        ate = cg == q.ncg - 1;
        last = top && j1 == nz;
        off = (size_t)cond * (size_t)q.n + (size_t)(j0 + lr0) * nth + c;
        coff = (size_t)q.cslot[cond] * (size_t)q.n + (size_t)(j0 + lr0) * nth + c;
        P = reinterpret_cast<T *>(g_res_smem) + tid * VEC;
        HU = reinterpret_cast<T *>(g_res_smem + q.o_rows);
        HR = HU + 2 * nth;
        HI = HR + 2 * nth;
        HE = HI + 2 * nth;
        YR = HE + nth;
        er = (q.rows + 1) * NS;
        EY = reinterpret_cast<T *>(g_res_smem + q.o_edge) + lr0 * NS + (cg >> 5);
    }

    // The coefficients, and zeros for u and where no block lies beyond.
    __device__ __forceinline__ void setup()
    {
        for (int i = tid; i < 2 * nth; i += TC) HU[i] = HR[i] = T(0);
        for (int i = tid; i < nth; i += TC) YR[i] = T(0);
        bar_sync_n(1, TC);
#pragma unroll
        for (int rr = 0; rr < RR; ++rr) {
            const size_t go = (size_t)rr * nth;
            const bool in = rr < nr;
            T t[VEC], zero[VEC];
#pragma unroll
            for (int e = 0; e < VEC; ++e) t[e] = zero[e] = T(0);
            V::st(P + rr * S, zero);
            if (in) V::ldrw(q.aE + coff + go, t);
            if (CS) V::st(P + FE + rr * S, t);
            if (in && sege) EY[er + rr * NS] = t[VEC - 1];
            if (CS) {
                // (a_N of the last row is not read: it couples to nothing)
                if (in && !(last && rr == nr - 1)) V::ldrw(q.aN + coff + go, t);
                V::st(P + FN + rr * S, in && !(last && rr == nr - 1) ? t : zero);
                if (in) V::ldrw(q.invD + coff + go, t);
                V::st(P + FI + rr * S, in ? t : zero);
                if (in) V::ldrw(q.D + coff + go, t);
                V::st(P + FD + rr * S, in ? t : zero);
            }
        }
        if (!act) return;
        T t[VEC];
        if (hasS) {
            V::ldrw(q.invD + coff - nth, t);
            V::st(HI + c, t);
        }
        if (hasN) {
            V::ldrw(q.invD + coff + (size_t)nr * nth, t);
            V::st(HI + nth + c, t);
            V::ldrw(q.aE + coff + (size_t)nr * nth, t);
            V::st(HE + c, t);
            if (sege) EY[er + nr * NS] = t[VEC - 1];
        }
    }

    // VEC doubles from global memory: 16 bytes at a time where every row allows it.
    __device__ __forceinline__ void ld64(const double *p, double (&x)[VEC]) const
    {
        if (VEC > 1 && q.pairs64) {
#pragma unroll
            for (int e = 0; e + 1 < VEC; e += 2) {
                const double2 t = *reinterpret_cast<const double2 *>(p + e);
                x[e] = t.x;
                x[e + 1] = t.y;
            }
        } else {
#pragma unroll
            for (int e = 0; e < VEC; ++e) x[e] = p[e];
        }
    }

    // Mixed precision: this thread's rows of r64 = S - A p64, and the warps' sums of r64 r64 and
    // S S.  The rows of the blocks below and above come as flagged words.  A row of p serves three
    // rows' equations from registers, its neighbours' columns come by shuffle: 5 values a cell are
    // loaded, not 11 (1024 x 512 x 9 cells: 145 us before, 123 us so; its FP64 operations take 70).
    __device__ __forceinline__ void residual(unsigned ep)
    {
        const double *const p64 = q.p64 + off;
        unsigned long long *const row64 = q.halo64 + ((size_t)blockIdx.x * 2 * nth + c) * 2;
        double pS64[VEC], pN64[VEC], rr = 0.0, ss = 0.0;
        if (hasS) {
            ld64(p64, pS64);
            ll_put<VEC>(row64, pS64, ep);
        }
        if (hasN) {
            ld64(p64 + (size_t)(nr - 1) * nth, pN64);
            ll_put<VEC>(row64 + 2 * nth, pN64, ep);
        }
        // (a run that ended late waits no further)
        const unsigned polls = sh.halo_failed ? 1u : q.polls;
        bar_sync_n(1, TC);                          // p64 of the block's other threads
#pragma unroll
        for (int e = 0; e < VEC; ++e) pS64[e] = pN64[e] = 0.0;
        bool ok = true;
        if (hasS) ok = ll_get<VEC>(row64 - 2 * nth, pS64, ep, polls);
        if (hasN) ok = ll_get<VEC>(row64 + 4 * nth, pN64, ep, polls) && ok;
        if (!ok) sh.halo_failed = 1;
        // p on this row and the one below, a_N of the row below
        double pc[VEC], ps[VEC], nS[VEC];
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
            pc[e] = nS[e] = 0.0;
            ps[e] = pS64[e];
        }
        const int jl = j0 + lr0;
        if (act) {
            ld64(p64, pc);
            if (jl > 0) ld64(q.aN64 + coff - nth, nS);
            if (jl > 0 && !hasS) ld64(p64 - nth, ps);
        }
        __syncwarp();
#pragma unroll 1
        for (int k = 0; k < RR; ++k) {
            const int j = jl + k;
            const bool in = k < nr;
            const size_t go = (size_t)k * nth;
            double pn[VEC], aE[VEC], aN[VEC], D[VEC], S[VEC];
#pragma unroll
            for (int e = 0; e < VEC; ++e) aE[e] = aN[e] = D[e] = S[e] = pn[e] = 0.0;
            double pW = 0.0, pE = 0.0, aW = 0.0;
            if (in) {
                ld64(q.aE64 + coff + go, aE);
                ld64(q.aN64 + coff + go, aN);
                ld64(q.D64 + coff + go, D);
                ld64(q.S64 + off + go, S);
                if (hasN && k == nr - 1) {
#pragma unroll
                    for (int e = 0; e < VEC; ++e) pn[e] = pN64[e];
                } else if (j < nz - 1) {
                    ld64(p64 + go + nth, pn);
                }
                if (segw) {
                    const int iw = atw ? nth - 1 : -1;
                    pW = p64[go + iw];
                    aW = q.aE64[coff + go + iw];
                }
                if (sege) pE = p64[go + (ate ? 1 - nth + VEC - 1 : VEC)];
            }
            const double wp = __shfl_up_sync(0xffffffffu, pc[VEC - 1], 1);
            const double wa = __shfl_up_sync(0xffffffffu, aE[VEC - 1], 1);
            const double ep_ = __shfl_down_sync(0xffffffffu, pc[0], 1);
            if (!segw) {
                pW = wp;
                aW = wa;
            }
            if (!sege) pE = ep_;
            if (in) {
                double r64[VEC];
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    double ap = D[e] * pc[e] - aE[e] * (e < VEC - 1 ? pc[e + 1] : pE) -
                                (e > 0 ? aE[e - 1] : aW) * (e > 0 ? pc[e - 1] : pW);
                    if (j < nz - 1) ap -= aN[e] * pn[e];
                    if (j > 0) ap -= nS[e] * ps[e];
                    const double rv = S[e] - ap;
                    r64[e] = rv;
                    rr = fma(rv, rv, rr);
                    ss = fma(S[e], S[e], ss);
                }
#pragma unroll
                for (int e = 0; e < VEC; ++e) q.r64[off + go + e] = r64[e];
            }
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                ps[e] = pc[e];
                pc[e] = pn[e];
                nS[e] = aN[e];
            }
        }
        const double x[2] = {rr, ss};
        ResTerm<double> t[2];
        res_warp_sums<2>(x, t);
        if (lane == 0) {
            sh.part64[0][wid] = t[0];
            sh.part64[1][wid] = t[1];
        }
    }
};

// One PCG run: the start (ep: the last exchange's number), the iterations, the result.
// Returns the last exchange's number.
//
// Every thread computes all RR rows: rows and threads beyond the block's have zero
// coefficients and only their stores are left out, so that the rows of a run are
// independent straight-line code.
template <typename T, int VEC, int RR, bool CS>
__device__ __forceinline__ unsigned res_iterate(const ResParams<T> &q, ResShared<T> &sh, unsigned ep)
{
    using V = Vec<T, VEC>;
    constexpr int S = kResThreads * VEC;            // private fields: [row][thread][VEC]
    constexpr int NS = kResSegs;
    constexpr bool kMixed = sizeof(T) == 4;         // FP32 runs inside FP64 refinement
    constexpr int FE = RR * S, FN = 2 * RR * S, FI = 3 * RR * S, FD = 4 * RR * S;
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
    T *const pX = q.o_x >= 0 ? reinterpret_cast<T *>(g_res_smem + q.o_x) + tid * VEC : q.p + off;
    const int stX = q.o_x >= 0 ? S : nth;

    // a row's coefficients; in global memory rows beyond the block's read the last one's place
    const int most = nr > 0 ? nr - 1 : 0;
    const unsigned cat = act ? coff : (unsigned)q.cslot[cond] * (unsigned)q.n;
    auto coef = [&](int field, const T *g, int rr, T(&x)[VEC]) {
        if constexpr (CS) {
            V::ldrw(P + field + rr * S, x);
        } else {
            V::ldrw(g + (cat + (unsigned)(min(rr, most) * nth)), x);
            const bool none = rr >= nr || (field == FN && last && rr == nr - 1);
#pragma unroll
            for (int e = 0; e < VEC; ++e) x[e] = none ? T(0) : x[e];
        }
    };
    auto get_E = [&](int rr, T(&x)[VEC]) { coef(FE, q.aE, rr, x); };
    auto get_N = [&](int rr, T(&x)[VEC]) { coef(FN, q.aN, rr, x); };
    auto get_I = [&](int rr, T(&x)[VEC]) { coef(FI, q.invD, rr, x); };
    auto get_D = [&](int rr, T(&x)[VEC]) { coef(FD, q.D, rr, x); };

    // rows of a block's halo area: 0, 1 = first and last row of v; 2, 3 = of z
    unsigned long long *const halo = q.halo + (size_t)blockIdx.x * 4 * q.halo_row + c * ((int)sizeof(T) / 4);
    T rg[RR][VEC], vz[RR][VEC], aS0[VEC], hS[VEC], hN[VEC];
    auto r_get = [&](int rr, T(&x)[VEC]) {
#pragma unroll
        for (int e = 0; e < VEC; ++e) x[e] = rg[rr][e];
    };
    auto r_put = [&](int rr, const T(&x)[VEC]) {
#pragma unroll
        for (int e = 0; e < VEC; ++e) rg[rr][e] = x[e];
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
        if (hasS) ok = ll_get<VEC>(halo + (s - 4) * q.halo_row, hS, ep, q.polls);
        if (hasN) ok = ll_get<VEC>(halo + (n + 4) * q.halo_row, hN, ep, q.polls) && ok;
        if (!ok) sh.halo_failed = 1;
    };

    if (j0 + lr0 > 0 && act) V::ldrw(q.aN + coff - nth, aS0);
    if constexpr (kMixed) {
        // b = r64 / ||r64||, x = 0
        const double unit = sh.unit;
        ++ep;
#pragma unroll
        for (int rr = 0; rr < RR; ++rr) {
            T r[VEC], x[VEC];
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                r[e] = rr < nr ? (T)(q.r64[off + (size_t)rr * nth + e] * unit) : T(0);
                x[e] = T(0);
            }
            r_put(rr, r);
            if (q.o_x >= 0 || rr < nr) V::st(pX + rr * stX, x);
            if (hasS && rr == 0) ll_put<VEC>(halo, r, ep);
            if (hasN && rr == nr - 1) ll_put<VEC>(halo + q.halo_row, r, ep);
            asm volatile("" ::: "memory");      // (one row's doubles in registers at a time)
        }
        fetch(1, 0);
    } else {
        // r = b (- A p), or the residual handed in; x = 0 or p; exchange 0: b.b, and r on the
        // halo rows
        ResAcc<T> acc;
        ++ep;
#pragma unroll
        for (int rr = 0; rr < RR; ++rr) {
            const size_t go = (size_t)rr * nth;
            T x[VEC], r[VEC];
#pragma unroll
            for (int e = 0; e < VEC; ++e) x[e] = r[e] = T(0);
            if (rr >= nr) {
                r_put(rr, r);
                if (q.o_x >= 0) V::st(pX + rr * stX, x);
                continue;
            }
            if (q.mode == kResRestart) {
                V::ldrw(q.r_in + off + go, r);
                V::ldrw(q.p + off + go, x);
            } else {
                V::ldrw(q.b + off + go, r);
                acc.add(r, r);
                if (!q.zero_init) {
                    V::ldrw(q.p + off + go, x);
                    const int j = j0 + lr0 + rr;
                    const T *p = q.p + off + go, *aE = q.aE + coff + go, *aN = q.aN + coff + go;
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        const int ie = c + e == nth - 1 ? 1 - nth + e : e + 1;
                        const int iw = c + e == 0 ? nth - 1 : e - 1;
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
            // the rows that the neighbours keep a copy of
            if (hasS && rr == 0) ll_put<VEC>(halo, r, ep);
            if (hasN && rr == nr - 1) ll_put<VEC>(halo + q.halo_row, r, ep);
        }
        publish(acc.value());
        fetch(1, 0);
        bar_sync_n(2, all);
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
#pragma unroll
        for (int rr = 0; rr < RR; ++rr) {
            T od[VEC], r[VEC];
            get_I(rr, od);
            r_get(rr, r);
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                r[e] -= alpha * vz[rr][e];
                vz[rr][e] = r[e] * od[e];
            }
            r_put(rr, r);
            if (rr == RR - 1 && act && !top) V::st(YR + (run + 1) * nth + c, vz[rr]);
            if (sege && rr < nr) EY[rr * NS] = vz[rr][VEC - 1];
            if (atw && rr < nr) EC[2 * rr] = vz[rr][0];
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
                const bool in = rr < nr;
                T ev[VEC], od[VEC], nv[VEC], w[VEC];
                get_E(rr, ev);
                get_I(rr, od);
                get_N(rr, nv);
                T yW = __shfl_up_sync(0xffffffffu, vz[rr][VEC - 1], 1);
                T aW = __shfl_up_sync(0xffffffffu, ev[VEC - 1], 1);
                if (segw) {
                    yW = in && !atw ? EYl[rr * NS] : T(0);
                    aW = in && !atw ? EYl[er + rr * NS] : T(0);
                }
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    T sum = nS[e] * yp[e];
                    sum = res_fma(e > 0 ? ev[e - 1] : aW, e > 0 ? vz[rr][e - 1] : yW, sum);
                    if (e == VEC - 1 && ate && in) sum = res_fma(ev[e], EC[2 * rr], sum);
                    w[e] = res_fma(od[e], sum, vz[rr][e]);
                }
                if (rr == 0 && act && run > 0) V::st(WR + (run - 1) * nth + c, w);
                if (segw && in) EY[2 * er + rr * NS] = w[0];
                if (ate && in) EC[2 * rr + 1] = w[VEC - 1];
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    yp[e] = in ? vz[rr][e] : yp[e];
                    nS[e] = in ? nv[e] : nS[e];
                    vz[rr][e] = w[e];
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
                            sum = res_fma(ev[e - 1], yN[e - 1], sum);
                        else if (!atw)
                            sum = res_fma(aW, yW, sum);
                        if (e == VEC - 1 && ate) sum = res_fma(ev[e], EC[2 * nr], sum);
                        wN[e] = res_fma(od[e], sum, yN[e]);
                    }
                }
            }
            bar_sync_n(1, TC);
            // second sweep (Eq. 3.6 without its factor): z = w + omega/D (upper couplings of w)
            if (act && !top) V::ldrw(WR + run * nth + c, wN);
#pragma unroll
            for (int rr = RR - 1; rr >= 0; --rr) {
                const bool in = rr < nr;
                T ev[VEC], od[VEC], nv[VEC], z[VEC], r[VEC];
                r_get(rr, r);
                get_E(rr, ev);
                get_I(rr, od);
                get_N(rr, nv);
                T wE = __shfl_down_sync(0xffffffffu, vz[rr][0], 1);
                if (sege) wE = in && !ate ? EWr[rr * NS] : T(0);
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    T sum = nv[e] * wN[e];
                    // (column nth - 1 has no upper neighbour to the east: wE is 0 there)
                    sum = res_fma(ev[e], e < VEC - 1 ? vz[rr][e + 1] : wE, sum);
                    if (e == 0 && atw && in) sum = res_fma(EYl[er + rr * NS], EC[2 * rr + 1], sum);
                    z[e] = res_fma(od[e], sum, vz[rr][e]);
                }
#pragma unroll
                for (int e = 0; e < VEC; ++e) {
                    wN[e] = in ? vz[rr][e] : wN[e];
                    vz[rr][e] = z[e];
                }
                if (hasS && rr == 0) ll_put<VEC>(halo + 2 * q.halo_row, z, ep);
                if (hasN && rr == nr - 1) ll_put<VEC>(halo + 3 * q.halo_row, z, ep);
                arz.add(r, z);
                arr.add(r, r);
                }
        } else {
#pragma unroll
            for (int rr = 0; rr < RR; ++rr) {
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
                if (q.o_x < 0 && rr >= nr) continue;
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
        V::ldrw(pS, us);
        V::ldrw(P, uc);
#pragma unroll
        for (int rr = 0; rr < RR; ++rr) {
            T ev[VEC], un[VEC], nv[VEC], D[VEC];
            get_E(rr, ev);
            get_N(rr, nv);
            get_D(rr, D);
            V::ldrw(rr == RR - 1 || rr == nr - 1 ? pN : P + (rr + 1) * S, un);
            T uW = __shfl_up_sync(0xffffffffu, uc[VEC - 1], 1);
            T uE = __shfl_down_sync(0xffffffffu, uc[0], 1);
            T aW = __shfl_up_sync(0xffffffffu, ev[VEC - 1], 1);
            if (segw) {
                uW = rr < nr ? pW[rr * S] : T(0);
                aW = rr < nr ? EYl[er + rr * NS] : T(0);
            }
            if (rr >= nr) aW = T(0);        // (the last column's, next to a thread without columns)
            if (sege) uE = rr < nr ? pE[rr * S] : T(0);
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                const T xE = e < VEC - 1 ? uc[e + 1] : uE;
                const T xW = e > 0 ? uc[e - 1] : uW;
                const T a = e > 0 ? ev[e - 1] : aW;
                T t = res_diff(D[e], uc[e], ev[e], xE);
                t = res_fnma(a, xW, t);
                t = res_fnma(nv[e], un[e], t);
                vz[rr][e] = res_fnma(nS[e], us[e], t);
            }
            auv.add(uc, vz[rr]);
            if (hasS && rr == 0) ll_put<VEC>(halo, vz[rr], ep);
            if (hasN && rr == nr - 1) ll_put<VEC>(halo + q.halo_row, vz[rr], ep);
#pragma unroll
            for (int e = 0; e < VEC; ++e) {
                us[e] = uc[e];
                uc[e] = un[e];
                nS[e] = rr + 1 < nr ? nv[e] : T(0);
            }
        }
        publish(auv.value());
        fetch(1, 0);
        bar_sync_n(2, all);
    }

    // the solution: x, or p64 += x in its units
#pragma unroll
    for (int rr = 0; rr < RR; ++rr) {
        if (rr >= nr) continue;
        T x[VEC];
        V::ldrw(pX + rr * stX, x);
        if constexpr (kMixed) {
            double *const p = q.p64 + off + (size_t)rr * nth;
#pragma unroll
            for (int e = 0; e < VEC; ++e) p[e] = fma(sh.back, (double)x[e], p[e]);
            asm volatile("" ::: "memory");
        } else if (q.o_x >= 0) {
            V::st(q.p + off + (size_t)rr * nth, x);
        }
    }
    return ep;
}

template <typename T, int VEC, int RR, bool CS>
__device__ __noinline__ void res_setup(const ResParams<T> &q)
{
    ResRows<T, VEC, RR, CS>(q, res_shared<T>()).setup();
}
// The norm of r64 as k_resid64 adds it up: a run of the refinement then works on the numbers that
// it would have with the phase kernels, bit for bit on every grid tested (the last bit of the norm is a bit of p, whose
// rounding is all that r64 is made of towards the end; with the norm as the blocks' exact sum a
// Picard step's Jacobian on 512 x 256 cells moved by 1e-10 to 1e-9, so it does by 1e-12).  First the sums of that kernel's warps,
// then, in every block, what its blocks and its last block add: 16 us a refinement on 256 x 128 x 9
// cells, 19 on 512 x 256 x 9 (several warps of that kernel at a time: no faster).
static __device__ __noinline__ void res_norm_warps(const ResParams<float> &q)
{
    const int warps = q.threads >> 5, lane = threadIdx.x & 31, total = q.grid64 * (kThreads / 32);
    const long long N = q.n * (long long)(gridDim.x / q.bpc), stride = (long long)q.grid64 * kThreads;
    for (int w = blockIdx.x * warps + (threadIdx.x >> 5); w < total; w += gridDim.x * warps) {
        double s = 0.0;
        for (long long g = (long long)w * 32 + lane; g < N; g += 4 * stride) {
            double v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = g + k * stride < N ? __ldcg(q.r64 + g + k * stride) : 0.0;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (g + k * stride < N) s = fma(v[k], v[k], s);
        }
        s = warp_sum_d(s);
        if (lane == 0) __stcg(q.warps64 + w, s);
    }
    __threadfence();
}
static __device__ __noinline__ void res_norm_total(const ResParams<float> &q, double *red)
{
    constexpr int W = kThreads / 32;
    const int warps = q.threads >> 5, lane = threadIdx.x & 31;
    for (int w = threadIdx.x >> 5; w < W; w += warps) {
        double s = 0.0;
        for (int b = w * 32 + lane; b < q.grid64; b += kThreads) {
            double x[W], t = 0.0;
#pragma unroll
            for (int k = 0; k < W; ++k) x[k] = __ldcg(q.warps64 + b * W + k);
#pragma unroll
            for (int k = 0; k < W; ++k) t += x[k];
            s += t;
        }
        s = warp_sum_d(s);
        if (lane == 0) red[w] = s;
    }
}

template <typename T, int VEC, int RR, bool CS>
__device__ __noinline__ void res_residual(const ResParams<T> &q, unsigned ep)
{
    ResRows<T, VEC, RR, CS>(q, res_shared<T>()).residual(ep);
}

// The meetings of the row threads with refine() between a residual and the next run.
template <bool NORM>
__device__ __forceinline__ void res_decide(const ResParams<float> &q, ResShared<float> &sh)
{
    const int all = q.threads + 32;
    if constexpr (NORM) {
        __threadfence();
        bar_sync_n(2, all);
        bar_sync_n(2, all);
        res_norm_warps(q);
        bar_sync_n(2, all);
        bar_sync_n(2, all);
        res_norm_total(q, sh.red64);
    }
    bar_sync_n(2, all);
    bar_sync_n(2, all);
}

template <typename T, int VEC, int RR, bool CS>
__global__ void __launch_bounds__(kResThreads + 32, 1) k_resident(const __grid_constant__ ResParams<T> q)
{
    ResShared<T> &sh = res_shared<T>();
    const int cond = blockIdx.x / q.bpc, grp = q.groups == 1 ? 0 : cond;
    if (!((q.mask >> grp) & 1ull)) return;                  // this group does not run
    res_clear(sh);
    if ((int)threadIdx.x >= q.threads) {
        res_exchange_warp<T>(q, sh, q.sc + grp, grp, q.groups == 1 ? 0 : cond * q.bpc,
                             q.groups == 1 ? (int)gridDim.x : q.bpc, threadIdx.x & 31);
        return;
    }
    unsigned ep = q.epoch;
    if constexpr (sizeof(T) == 4) {
        // FP64 refinements around the FP32 run
        res_setup<T, VEC, RR, CS>(q);
#pragma unroll 1
        for (;;) {
            res_residual<T, VEC, RR, CS>(q, ++ep);
            res_decide<true>(q, sh);
            if (sh.stop) break;
            ep = res_iterate<T, VEC, RR, CS>(q, sh, ep);
        }
    } else {
        res_setup<T, VEC, RR, CS>(q);
        res_iterate<T, VEC, RR, CS>(q, sh, ep);
    }
}

// Returns a kernel, named in parentheses, with its record of devices.
#define GMAF_RES_KERNEL(fn)                                                                          \
    do {                                                                                             \
        static std::atomic<unsigned long long> opted{0};                                             \
        return ResKernel{(const void *)fn, &opted};                                                  \
    } while (0)

}  // namespace gmaf
