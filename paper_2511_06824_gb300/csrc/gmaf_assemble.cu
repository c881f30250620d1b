// Geometry, FVM assembly, load integration and the Picard update on the GPU.
//
//  - film thickness: Eq. 2.3 with h_Text from a hexagonal dimple lattice;
//  - assembly: Sec. 2.1 (Eq. 2.1, 2.4-2.7) and Sec. 2.4-I, one thread per column
//    marching down the rows, for all conditions of the same eccentricities at once;
//  - loads: Sec. 2.4-III, pressure and viscous shear, the same way;
//  - Picard: Eq. 2.12-2.19 with the backward-difference closure of Eq. 2.22.
#include <cmath>
#include <cstring>

#include "gmaf_internal.cuh"

namespace gmaf {

// ------------------------------------------------------------------ host: geometry set-up

Lattice make_lattice(const gmaf_texture *tex, double Rk)
{
    Lattice lt{};
    if (tex == nullptr || tex->kind == 0 || tex->depth == 0.0) return lt;
    lt.on = 1;
    lt.r = tex->radius;
    lt.depth = tex->depth;
    lt.oth = tex->offset_theta;
    lt.oz = tex->offset_z;
    const double rho = tex->area_density;
    const double circ = 2.0 * kPi * Rk;
    // column count: nearest whole number to the ideal hexagonal pitch for density rho
    const double a0 = lt.r * std::sqrt(2.0 * kPi / (std::sqrt(3.0) * rho));
    double ncol = std::round(circ / a0);
    if (ncol < 1.0) ncol = 1.0;
    lt.ath = circ / ncol;
    lt.az = kPi * lt.r * lt.r / (rho * lt.ath);   // one dimple per ath x az cell
    return lt;
}

Geom make_geom(const gmaf_grid *g, const gmaf_physics *ph, const gmaf_texture *tex)
{
    Geom G{};
    G.nth = g->n_theta;
    G.nz = g->n_z;
    G.Rk = ph->R_k;
    G.L = ph->L;
    G.c = ph->c;
    G.mu = ph->mu;
    G.v = ph->v_slide;
    G.pch = ph->p_chamber;
    G.pcase = ph->p_case;
    G.dth = 2.0 * kPi / (double)G.nth;
    G.dx = G.Rk * G.dth;
    G.dz = G.L / (double)G.nz;
    G.invL = 1.0 / G.L;
    G.lt = make_lattice(tex, G.Rk);
    return G;
}

// ------------------------------------------------------------------ device: film thickness

// A point at unwrapped (x, z) is inside a dimple if its distance to the nearest centre
// of one of four lattice rows is below r.  The lattice decision is an integer one, so
// it is written with explicitly rounded operations (no contraction into fused
// multiply-adds) to take the same decision as a plain IEEE evaluation, (dx dx) + (dz dz)
// < r r for the centres left and right of the point.  It separates: dz depends on the
// level z and the lattice row only, dx on the column and on the row's parity (odd rows
// are shifted) only.  A block therefore tables the rows that reach each of its levels
// (those with dz dz < r r: the sum cannot be smaller), a thread the smaller dx dx of its
// column for either parity, and a cell is left with one addition and one comparison
// per row in reach instead of two divisions and eight squares (rounding is monotonic,
// so the smaller square decides).
struct Reach {
    double dz2[4];      // squared distances to the lattice rows in reach
    int n, odd;         // how many; bit q: row q is odd
};

__device__ __forceinline__ void lattice_reach(const Lattice &lt, double z, Reach &out)
{
    out.n = out.odd = 0;
    if (!lt.on) return;
    const double k0 = floor(__ddiv_rn(__dsub_rn(z, lt.oz), lt.az));
    const double r2 = __dmul_rn(lt.r, lt.r);
    for (int dk = -1; dk <= 2; ++dk) {
        const double k = __dadd_rn(k0, (double)dk);
        const double zc = __dadd_rn(lt.oz, __dmul_rn(k, lt.az));
        const double dz = __dsub_rn(z, zc);
        const double dz2 = __dmul_rn(dz, dz);
        if (!(dz2 < r2)) continue;
        if ((long long)k & 1LL) out.odd |= 1 << out.n;
        out.dz2[out.n++] = dz2;
    }
}

// The smaller squared distance of column x to the centres of an even (q[0]) or odd (q[1]) row.
__device__ __forceinline__ void lattice_column(const Lattice &lt, double x, double (&q)[2])
{
    q[0] = q[1] = 0.0;
    if (!lt.on) return;
#pragma unroll
    for (int odd = 0; odd < 2; ++odd) {
        const double shift = odd ? __dmul_rn(0.5, lt.ath) : 0.0;
        const double u = __dsub_rn(__dsub_rn(x, lt.oth), shift);
        const double m = floor(__ddiv_rn(u, lt.ath));
        const double dxa = __dsub_rn(u, __dmul_rn(m, lt.ath));
        const double dxb = __dsub_rn(u, __dmul_rn(__dadd_rn(m, 1.0), lt.ath));
        const double a = __dmul_rn(dxa, dxa), b = __dmul_rn(dxb, dxb);
        q[odd] = a < b ? a : b;
    }
}

__device__ __forceinline__ double texture_depth(const Lattice &lt, const Reach &z, const double (&q)[2])
{
    const double r2 = __dmul_rn(lt.r, lt.r);
    bool in = false;
    // (squares: not negative, so that the integers compare as they do, off the FP64 pipe)
    for (int c = 0; c < z.n; ++c)
        in = in || __double_as_longlong(__dadd_rn((z.odd >> c) & 1 ? q[1] : q[0], z.dz2[c])) < __double_as_longlong(r2);
    return in ? lt.depth : 0.0;
}

// Smooth part of Eq. 2.3 for a condition: sqrt((Rc cos - ex)^2 + (Rc sin - ey)^2) - Rk.
// t = z / L along the gap; e = state[0..3].
struct FilmPt {
    double X, Y, rho;
};

__device__ __forceinline__ FilmPt film_at(double Rc, double ex, double ey, double ct, double st)
{
    FilmPt f;
    f.X = Rc * ct - ex;
    f.Y = Rc * st - ey;
    f.rho = sqrt(f.X * f.X + f.Y * f.Y);
    return f;
}

__device__ __forceinline__ FilmPt film_pt(const Geom &g, const double *e, double ct, double st,
                                          double t)
{
    return film_at(g.Rk + g.c, e[0] + (e[2] - e[0]) * t, e[1] + (e[3] - e[1]) * t, ct, st);
}

// ------------------------------------------------------------------ trig table

// trig = [cos(theta_c), sin(theta_c), cos(theta_e), sin(theta_e)] x nth with
// theta_c = (i + 1/2) dth (cell centres) and theta_e = (i + 1) dth (east faces).
__global__ void k_trig(int nth, double dth, double *trig)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nth) return;
    const double tc = ((double)i + 0.5) * dth;
    const double te = ((double)i + 1.0) * dth;
    double s, c;
    sincos(tc, &s, &c);
    trig[i] = c;
    trig[nth + i] = s;
    sincos(te, &s, &c);
    trig[2 * nth + i] = c;
    trig[3 * nth + i] = s;
}

int launch_trig(const Geom &g, double *trig, cudaStream_t s)
{
    k_trig<<<(g.nth + 127) / 128, 128, 0, s>>>(g.nth, g.dth, trig);
    return cuda_status(cudaGetLastError());
}

// ------------------------------------------------------------------ condition fan-out (Eq. 2.17-2.19)

// conds[k] = base for k = 0; e_{k-1} + d_e for k = 1..4; edot_{k-5} + d_edot for k = 5..8.
// cslot_write[k] = k for k <= 4 (own coefficients), -1 for k >= 5: the ė-perturbed
// conditions share the coefficients of condition 0 because A depends on e only.
// General scheme (Eq. 2.13-2.19): condition 0 = (e, edot), 1..4 = e_j + d_e,
// 5..8 = edot_j + d_edot; coefficient slots 0..4 (A does not depend on edot).
// Simplified scheme (Eq. 2.20): 0 = (e, edot), 1..4 = edot_j + d_edot, all in slot 0.
__global__ void k_fanout(const double base0, const double base1, const double base2,
                         const double base3, const double base4, const double base5,
                         const double base6, const double base7, double d_e, double d_edot,
                         double *conds, int *cslot_write, int simplified)
{
    const int k = threadIdx.x;
    if (k >= (simplified ? 5 : 9)) return;
    double s[8] = {base0, base1, base2, base3, base4, base5, base6, base7};
    if (simplified) {
        if (k >= 1) s[4 + (k - 1)] += d_edot;
        cslot_write[k] = (k == 0) ? 0 : -1;
    } else {
        if (k >= 1 && k <= 4) s[k - 1] += d_e;
        if (k >= 5) s[4 + (k - 5)] += d_edot;
        cslot_write[k] = (k <= 4) ? k : -1;
    }
    for (int q = 0; q < 8; ++q) conds[k * 8 + q] = s[q];
}

int launch_fanout(const double *b, double d_e, double d_edot, double *conds, int *cslot_write,
                  cudaStream_t s, int simplified)
{
    k_fanout<<<1, 32, 0, s>>>(b[0], b[1], b[2], b[3], b[4], b[5], b[6], b[7], d_e, d_edot, conds,
                              cslot_write, simplified);
    return cuda_status(cudaGetLastError());
}

// ------------------------------------------------------------------ conditions of one film
//
// The film thickness depends on the eccentricities only, so conditions that differ in
// their rates share it (a Picard step's base and its four rate perturbations).  A batch
// is up to kBatch of them; the kernels below evaluate the film once for a batch.

constexpr int kBatch = 5;

struct Batches {
    int n;
    unsigned char cnt[kMaxCond], idx[kMaxCond][kBatch];
};

// Conditions 0 .. ncond - 1 with the same e (e == nullptr: of a Picard step's fan-out).
static Batches make_batches(int ncond, const gmaf_state *conds, bool simplified)
{
    Batches b{};
    auto same = [&](int k, int l) {
        if (conds) return std::memcmp(conds[k].e, conds[l].e, sizeof conds[k].e) == 0;
        return simplified || ((k == 0 || k >= 5) && (l == 0 || l >= 5));
    };
    for (int k = 0; k < ncond; ++k) {
        int at = -1;
        for (int q = 0; q < b.n && at < 0; ++q)
            if (b.cnt[q] < kBatch && same(b.idx[q][0], k)) at = q;
        if (at < 0) at = b.n++;
        b.idx[at][b.cnt[at]++] = (unsigned char)k;
    }
    return b;
}

// ------------------------------------------------------------------ assembly
//
// Bound by the FP64 pipe (one warp instruction in 16 cycles an SM): every film point
// costs a square root, every cell two quotients more.  A thread marches down its column
// for one batch of conditions, so the film at the south face is the one at the north
// face of the row before, and per row there are three film points for the whole batch.
// Lane 0 of a warp works on the column west of the warp's 31 others: its a_E is the
// neighbour's a_W, so that the diagonal is complete without a second pass.  The
// results are bitwise those of evaluating every cell and condition by itself.
// 1024 x 512 x 9 cells of a Picard step's conditions: 1486 us that way, 703 us now (738 before
// what depends on the row only was formed once a block, and conditions of one film shared a
// reciprocal).

// a / b, correctly rounded, from y = 1 / b (correctly rounded): the product and two
// corrections by the residual (Markstein), for a divisor that is the same for all cells.
__device__ __forceinline__ double quotient(double a, double b, double y)
{
    double t = a * y;
    t = fma(y, fma(-b, t, a), t);
    return fma(y, fma(-b, t, a), t);
}

// Far from the ends of the exponent's range, where quotient() is that of the division.
__device__ __forceinline__ bool mid_range(double x)
{
    const int e = (__double2hiint(x) >> 20) & 0x7ff;
    return e > 300 && e < 1700;
}

constexpr int kAsmWarps = 4, kAsmRows = 32;

// Per row of a block: the axial coordinate of its centre and north face, and what of the
// texture is in reach of them; the eccentricities there, and the rates of each condition at
// the centre.
struct AsmRow {
    double tc, exc, eyc, exn, eyn;
    double exd[kBatch], eyd[kBatch];
    Reach c, n;
};

__global__ void __launch_bounds__(kAsmWarps * 32) k_assemble(Geom g, Batches bt,
                                                             const double *__restrict__ conds,
                                                             const int *__restrict__ coef_slot,
                                                             double *__restrict__ D,
                                                             double *__restrict__ aE,
                                                             double *__restrict__ aN,
                                                             double *__restrict__ S,
                                                             const double *__restrict__ trig,
                                                             int rows, double inv_dx, double inv_dz,
                                                             int *__restrict__ flags)
{
    __shared__ AsmRow row[kAsmRows];
    __shared__ Reach south;
    __shared__ double st[kBatch][8];
    __shared__ int slot[kBatch];
    const long long n = (long long)g.nth * g.nz;
    const int nb = bt.cnt[blockIdx.z];
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid < 8 * nb) st[tid >> 3][tid & 7] = conds[8 * bt.idx[blockIdx.z][tid >> 3] + (tid & 7)];
    if (tid < nb) slot[tid] = coef_slot[bt.idx[blockIdx.z][tid]];
    const int i0 = (blockIdx.x * kAsmWarps + (tid >> 5)) * 31;      // the warp's first own column
    int i = i0 + lane - 1;
    const bool own = lane > 0 && i < g.nth;
    if (i < 0) i = g.nth - 1;
    if (i >= g.nth) i = g.nth - 1;

    const double Ub = -g.v;
    const double inv12mu = 1.0 / (12.0 * g.mu), Rc = g.Rk + g.c;
    int contact = 0;
    const double cc = trig[i], sc = trig[g.nth + i];
    const double ce = trig[2 * g.nth + i], se = trig[3 * g.nth + i];
    double qc[2], qe[2];
    lattice_column(g.lt, __dmul_rn(g.Rk, ((double)i + 0.5) * g.dth), qc);
    lattice_column(g.lt, __dmul_rn(g.Rk, ((double)i + 1.0) * g.dth), qe);
    const int segs = (g.nz + rows - 1) / rows;
    for (int seg = blockIdx.y; seg < segs; seg += gridDim.y) {
        const int j0 = seg * rows, j1 = min(j0 + rows, g.nz);
        __syncthreads();
        for (int q = tid; q < 2 * (j1 - j0) + 1; q += blockDim.x) {
            if (q == 2 * (j1 - j0)) {
                lattice_reach(g.lt, (double)j0 * g.dz, south);
            } else {
                const int j = j0 + q / 2;
                const double z = q & 1 ? ((double)j + 1.0) * g.dz : ((double)j + 0.5) * g.dz;
                AsmRow &r = row[q / 2];
                const double t = z * g.invL;
                (q & 1 ? r.exn : r.exc) = st[0][0] + (st[0][2] - st[0][0]) * t;
                (q & 1 ? r.eyn : r.eyc) = st[0][1] + (st[0][3] - st[0][1]) * t;
                if (!(q & 1)) r.tc = t;
                lattice_reach(g.lt, z, q & 1 ? r.n : r.c);
            }
        }
        __syncthreads();
        // (the multiply-adds of S are written out, so that it does not depend on how the
        // compiler pairs these terms)
        for (int q = tid; q < nb * (j1 - j0); q += blockDim.x) {
            const int k = q / (j1 - j0);
            AsmRow &r = row[q - k * (j1 - j0)];
            const double rest = 1.0 - r.tc;
            r.exd[k] = __fma_rn(st[k][4], rest, __dmul_rn(st[k][6], r.tc));
            r.eyd[k] = __fma_rn(st[k][5], rest, __dmul_rn(st[k][7], r.tc));
        }
        __syncthreads();
        if (i0 >= g.nth) continue;                                  // (a whole warp)
        // the south face of the first row
        double hs, south_n = 0.0;
        {
            const FilmPt fs = film_pt(g, st[0], cc, sc, ((double)j0 * g.dz) * g.invL);
            hs = (fs.rho - g.Rk) + texture_depth(g.lt, south, qc);
            contact |= hs <= 0.0;
            if (j0 > 0) south_n = quotient(hs * hs * hs * inv12mu * g.dx, g.dz, inv_dz);
        }
        for (int j = j0; j < j1; ++j) {
            const AsmRow &rw = row[j - j0];
            const FilmPt fe = film_at(Rc, rw.exc, rw.eyc, ce, se);
            const FilmPt fn = film_at(Rc, rw.exn, rw.eyn, cc, sc);
            const FilmPt fc = film_at(Rc, rw.exc, rw.eyc, cc, sc);
            const double he = (fe.rho - g.Rk) + texture_depth(g.lt, rw.c, qe);
            const double hn = (fn.rho - g.Rk) + texture_depth(g.lt, rw.n, qc);
            contact |= (he <= 0.0) | (hn <= 0.0);
            const double gn = hn * hn * hn * inv12mu;
            const double ge = he * he * he * inv12mu;
            const double east = quotient(ge * g.dz, g.dx, inv_dx);
            const double north = j < g.nz - 1 ? quotient(gn * g.dx, g.dz, inv_dz) : 0.0;
            const double west = __shfl_up_sync(0xffffffffu, east, 1);
            double aB = 0.0, sB = 0.0;
            if (j == 0) {
                const double gs = hs * hs * hs * inv12mu;
                const double a = gs * g.dx / (0.5 * g.dz);
                aB += a;
                sB += a * g.pch;
            }
            if (j == g.nz - 1) {
                const double a = gn * g.dx / (0.5 * g.dz);
                aB += a;
                sB += a * g.pcase;
            }
            // D = a_E + a_W + a_N + a_S + a_B, with a_W(i) = a_E(i - 1) (periodic) and
            // a_S(j) = a_N(j - 1), so that the stored diagonals describe a symmetric matrix
            const double diag = east + west + north + south_n + aB;
            if (own) {
                const size_t P = (size_t)j * g.nth + i;
                const double wedge = __dmul_rn(-(Ub / 2.0), __dsub_rn(hn, hs));
                // (several conditions: one reciprocal for their quotients)
                const bool shared = nb > 1 && mid_range(fc.rho);
                const double inv_rho = shared ? 1.0 / fc.rho : 0.0;
                for (int k = 0; k < nb; ++k) {
                    // dh/dt = -(X/rho) dex/dt - (Y/rho) dey/dt at the cell centre
                    const double a = __fma_rn(fc.X, rw.exd[k], __dmul_rn(fc.Y, rw.eyd[k]));
                    const bool zero = (__double_as_longlong(a) << 1) == 0;
                    const double hdot = -(shared && (mid_range(a) || zero) ? quotient(a, fc.rho, inv_rho) : a / fc.rho);
                    const double squeeze = __dmul_rn(__dmul_rn(hdot, g.dx), g.dz);
                    S[(size_t)bt.idx[blockIdx.z][k] * (size_t)n + P] =
                        __dadd_rn(__fma_rn(wedge, g.dx, -squeeze), sB);
                    if (slot[k] >= 0) {
                        const size_t at = (size_t)slot[k] * (size_t)n + P;
                        aE[at] = east;
                        aN[at] = north;
                        D[at] = diag;
                    }
                }
            }
            hs = hn;
            south_n = north;
        }
    }
    if (contact) atomicOr(flags, 1);
}

// conds_host: the conditions' states (null: a Picard step's fan-out, general or simplified).
int launch_assemble(const Geom &g, int ncond, const double *conds, const int *coef_slot,
                    double *D, double *aE, double *aN, double *S, const double *trig, int *flags,
                    const gmaf_state *conds_host, bool simplified, cudaStream_t s)
{
    const Batches bt = make_batches(ncond, conds_host, simplified);
    const int strips = (g.nth + 31 * kAsmWarps - 1) / (31 * kAsmWarps);
    // rows a block marches: 32, fewer while there are fewer than about 4 blocks an SM (512 x 256
    // x 9: 247 us a call, with 8 blocks an SM 275, with 1 330)
    int rows = kAsmRows;
    while (rows > 2 && (long long)strips * ((g.nz + rows - 1) / rows) * bt.n < 152 * 4) rows /= 2;
    const int segs = (g.nz + rows - 1) / rows;
    const dim3 grid(strips, segs < 65535 ? segs : 65535, bt.n);
    k_assemble<<<grid, kAsmWarps * 32, 0, s>>>(g, bt, conds, coef_slot, D, aE, aN, S, trig, rows,
                                              1.0 / g.dx, 1.0 / g.dz, flags);
    return cuda_status(cudaGetLastError());
}

// ------------------------------------------------------------------ loads
//
// Pressure: the element-wise 2-D trapezoid (mean of the 4 corners times the
// element area) summed over elements equals a sum over pressure nodes with
// weight R_k dth (dz_below + dz_above)/2, dz_e = dz/2 for the two boundary
// element rows.  Shear: per element at its centre, dp/dz and dp/dtheta from
// differences of edge means.  Node rows r = 0 .. nz+1 (0: z = 0 with p_ch,
// nz+1: z = L with p_case, else cell centres); element rows er = 0 .. nz.
//
// Bound by the FP64 pipe.  The directions (cos, sin) depend on the column only, so a
// thread marches down its column and keeps five sums for each condition, of p w,
// z p w, tau_theta A, z tau_theta A and tau_z A; the twelve forces and moments are
// formed from them once, at the end of the column.  The film of an element is formed
// once for a batch of conditions of the same eccentricities.  1024 x 512 x 9 cells: 347 us,
// 2107 us when every thread added up the twelve sums of one condition cell by cell.
//
// Grid: blocks (each takes units of a strip of columns x a segment of rows) x batches.
// Each block writes 12 partial sums a condition; the last block of a batch (by ticket) adds them in block order.

constexpr int kLoadThreads = 128, kLoadRows = 64;
constexpr int kSums = 12, kShare = 8;           // sums; threads that add up one sum of a block

struct LoadRow {
    double w, zw;           // weight of node row r = er, and z times it
    double t, zc;           // z / L and z of the element's centre
    double cs, ct, cv;      // factors: h dp/dz A, h dp/dtheta / R_k A, 1 / h (Couette) A
    Reach reach;
};

// Adds part[b * kSums + c], b = 0 .. nblk - 1, for c = tid / kShare: its kShare threads take
// every kShare-th block and are added in order.  Threads from kSums * kShare on idle.
template <typename F>
__device__ __forceinline__ void add_up(int tid, int nblk, F &&get, double *out)
{
    const int c = tid / kShare, l = tid % kShare;
    double s = 0.0;
    if (tid < kSums * kShare) {
#pragma unroll 4
        for (int b = l; b < nblk; b += kShare) s += get(b, c);
    }
    // (whole warps: kSums * kShare is a multiple of 32)
    if (tid < kSums * kShare) {
#pragma unroll
        for (int o = 1; o < kShare; o *= 2) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (l == 0) out[c] = s;
    }
}

__global__ void __launch_bounds__(kLoadThreads) k_loads(Geom g, Batches bt,
                                                        const double *__restrict__ conds,
                                                        const double *__restrict__ p,
                                                        const double *__restrict__ trig,
                                                        double *__restrict__ partials,
                                                        unsigned int *__restrict__ tickets,
                                                        double *__restrict__ loads, int rows,
                                                        int *flags)
{
    __shared__ LoadRow row[kLoadRows];
    __shared__ double red[kSums][kLoadThreads + 1], total[kBatch][kSums], one[kSums];
    __shared__ int s_last;
    const int nth = g.nth, nz = g.nz;
    const long long n = (long long)nth * nz;
    const int nb = bt.cnt[blockIdx.y];
    const unsigned char *idx = bt.idx[blockIdx.y];
    const int nblk = gridDim.x, blk = blockIdx.x;
    const int tid = threadIdx.x;
    const double Ub = -g.v;
    const int strips = (nth + kLoadThreads - 1) / kLoadThreads, segs = (nz + 1 + rows - 1) / rows;
    double e4[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) e4[q] = conds[8 * idx[0] + q];
    if (tid < kBatch * kSums) total[tid / kSums][tid % kSums] = 0.0;
    int contact = 0;
    for (long long unit = blk; unit < (long long)strips * segs; unit += nblk) {
        const int seg = (int)(unit / strips), strip = (int)(unit - (long long)seg * strips);
        const int e0 = seg * rows, e1 = min(e0 + rows, nz + 1);             // element rows
        __syncthreads();
        for (int q = tid; q < e1 - e0; q += blockDim.x) {
            const int er = e0 + q;
            LoadRow &w = row[q];
            const double zr = (er == 0) ? 0.0 : ((double)er - 0.5) * g.dz;
            const double dzb = (er == 0) ? 0.0 : (er == 1 ? 0.5 * g.dz : g.dz);
            const double dza = (er == 0 || er == nz) ? 0.5 * g.dz : g.dz;
            w.w = g.Rk * g.dth * (0.5 * (dzb + dza));
            w.zw = zr * w.w;
            const double dze = (er == 0 || er == nz) ? 0.5 * g.dz : g.dz;
            const double zhi = (er == nz) ? g.L : ((double)er + 0.5) * g.dz;
            w.zc = 0.5 * (zr + zhi);
            w.t = w.zc * g.invL;
            // with A = R_k dth dze: -(h/2) dp/dz A = h cs (north - south edge sums),
            // -(h/2) dp/dtheta / R_k A = h ct (east - west edge sums), mu U_b / h A = cv / h
            w.cs = -0.25 * g.Rk * g.dth;
            w.ct = -0.25 * dze;
            w.cv = g.mu * Ub * (g.Rk * g.dth * dze);
            lattice_reach(g.lt, w.zc, w.reach);
        }
        __syncthreads();
        const int i = strip * kLoadThreads + tid;
        double sum[kBatch][5];
#pragma unroll
        for (int k = 0; k < kBatch; ++k)
#pragma unroll
            for (int q = 0; q < 5; ++q) sum[k][q] = 0.0;
        double ct = 0.0, sn = 0.0, ce = 0.0, se = 0.0;
        if (i < nth) {
            const int i2 = (i + 1 == nth) ? 0 : i + 1;
            ct = trig[i];
            sn = trig[nth + i];
            ce = trig[2 * nth + i];
            se = trig[3 * nth + i];
            double qe[2];
            lattice_column(g.lt, __dmul_rn(g.Rk, ((double)i + 1.0) * g.dth), qe);
            // pressure of node row r at columns i and i + 1
            auto node = [&](int k, int r, double &a, double &b) {
                if (r == 0) {
                    a = b = g.pch;
                } else if (r == nz + 1) {
                    a = b = g.pcase;
                } else {
                    const double *pk = p + (size_t)idx[k] * (size_t)n + (size_t)(r - 1) * nth;
                    a = pk[i];
                    b = pk[i2];
                }
            };
            double pa[kBatch], pb[kBatch];
#pragma unroll
            for (int k = 0; k < kBatch; ++k)
                if (k < nb) node(k, e0, pa[k], pb[k]);
            for (int er = e0; er < e1; ++er) {
                const LoadRow &w = row[er - e0];
                double na[kBatch], nc[kBatch];
#pragma unroll
                for (int k = 0; k < kBatch; ++k)
                    if (k < nb) node(k, er + 1, na[k], nc[k]);
                const FilmPt f = film_pt(g, e4, ce, se, w.t);
                const double h = (f.rho - g.Rk) + texture_depth(g.lt, w.reach, qe);
                contact |= (h <= 0.0);
                const double couette = w.cv / h, hcs = h * w.cs, hct = h * w.ct;
#pragma unroll
                for (int k = 0; k < kBatch; ++k) {
                    if (k >= nb) continue;
                    const double tz = fma(hcs, (na[k] + nc[k]) - (pa[k] + pb[k]), couette);
                    const double tt = hct * ((pb[k] + nc[k]) - (pa[k] + na[k]));
                    sum[k][0] = fma(pa[k], w.w, sum[k][0]);
                    sum[k][1] = fma(pa[k], w.zw, sum[k][1]);
                    sum[k][2] += tt;
                    sum[k][3] = fma(w.zc, tt, sum[k][3]);
                    sum[k][4] += tz;
                    pa[k] = na[k];
                    pb[k] = nc[k];
                }
            }
            if (e1 == nz + 1) {
                // the last node row, z = L
                const double wl = g.Rk * g.dth * (0.5 * (0.5 * g.dz));
#pragma unroll
                for (int k = 0; k < kBatch; ++k)
                    if (k < nb) {
                        sum[k][0] = fma(pa[k], wl, sum[k][0]);
                        sum[k][1] = fma(pa[k], g.L * wl, sum[k][1]);
                    }
            }
        }
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            if (k >= nb) continue;
            const double P = sum[k][0], Pz = sum[k][1], T = sum[k][2], Tz = sum[k][3], Z = sum[k][4];
            const double fx = -P * ct, fy = -P * sn;
            red[0][tid] = fx;
            red[1][tid] = fy;
            red[2][tid] = 0.0;
            red[3][tid] = Pz * sn;
            red[4][tid] = -Pz * ct;
            red[5][tid] = g.Rk * ct * fy - g.Rk * sn * fx;
            red[6][tid] = -T * se;
            red[7][tid] = T * ce;
            red[8][tid] = Z;
            red[9][tid] = g.Rk * se * Z - Tz * ce;
            red[10][tid] = -Tz * se - g.Rk * ce * Z;
            red[11][tid] = g.Rk * ce * (T * ce) + g.Rk * se * (T * se);
            __syncthreads();
            add_up(tid, kLoadThreads, [&](int b, int c) { return red[c][b]; }, one);
            __syncthreads();
            if (tid < kSums) total[k][tid] += one[tid];
        }
    }
    if (contact) atomicOr(flags, 1);
    __syncthreads();
    for (int q = tid; q < nb * kSums; q += blockDim.x)
        partials[((size_t)idx[q / kSums] * nblk + blk) * kSums + q % kSums] = total[q / kSums][q % kSums];
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        const unsigned t = atomicAdd(&tickets[idx[0]], 1u);
        s_last = (t == (unsigned)nblk - 1u);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int k = 0; k < nb; ++k) {
        const double *part = partials + (size_t)idx[k] * nblk * kSums;
        add_up(tid, nblk, [&](int b, int c) { return __ldcg(part + (size_t)b * kSums + c); },
               loads + (size_t)idx[k] * kSums);
    }
    if (tid == 0) tickets[idx[0]] = 0u;
}

// Blocks a condition may have (its partial sums): two an SM.
size_t loads_partials_bytes(int ncond, int num_sms)
{
    return (size_t)ncond * (size_t)num_sms * 2 * kSums * sizeof(double) + kMaxCond * sizeof(unsigned);
}

// conds_host: as in launch_assemble.
int launch_loads(const Geom &g, int ncond, const double *conds, const double *p,
                 const double *trig, double *partials, unsigned int *tickets, double *loads,
                 int *flags, int num_sms, const gmaf_state *conds_host, bool simplified,
                 cudaStream_t s)
{
    const Batches bt = make_batches(ncond, conds_host, simplified);
    const int er = g.nz + 1, strips = (g.nth + kLoadThreads - 1) / kLoadThreads;
    // segments of rows: short ones on small grids, so that every SM has work, but no more
    // blocks a condition than there are partial sums (512 x 256 x 9: 116 us a call with 4 blocks
    // an SM, 134 with 8, 188 with 1)
    const long long most = 2LL * num_sms;
    int rows = kLoadRows;
    while (rows > 2 && (long long)strips * ((er + rows - 1) / rows) * bt.n < 4LL * num_sms &&
           (long long)strips * ((er + rows / 2 - 1) / (rows / 2)) <= most)
        rows /= 2;
    const long long units = (long long)strips * ((er + rows - 1) / rows);
    k_loads<<<dim3((unsigned)(units < most ? units : most), bt.n), kLoadThreads, 0, s>>>(
        g, bt, conds, p, trig, partials, tickets, loads, rows, flags);
    return cuda_status(cudaGetLastError());
}

// ------------------------------------------------------------------ Picard update

// result layout (doubles): [0..11] loads of condition 0, [12..59] J (6 x 8),
// [60..63] G, [64..71] new state, [72] status (0 ok, -4 singular).
//
// One warp: the entries of a step side by side, the 4 x 4 system eliminated a row and column a
// lane.  All of it is chains of FP64 divisions (570 cycles) and multiply-adds (64): 43 us on one
// thread, 9 us so.
__global__ void k_picard(const double *__restrict__ loads, PicardIn in, double dt, double d_e,
                         double d_edot, double L, double *__restrict__ result)
{
    __shared__ double F[9][6], J[6][8], Je[4][4], Jd[4][4], G[4], A[4][5];
    const int lane = threadIdx.x;
    const double *base = in.base, *e_prev = in.e_prev, *F_ext = in.F_ext;
    const bool simp = in.simplified != 0;
    const int K = simp ? 5 : 9;
    for (int q = lane; q < K * 6; q += 32) F[q / 6][q % 6] = loads[q / 6 * 12 + q % 6] + loads[q / 6 * 12 + 6 + q % 6];
    __syncwarp();
    // load Jacobian by forward differences (Eq. 2.13-2.14); the simplified scheme
    // forms only the rate columns, from its conditions 1..4
    for (int q = lane; q < 48; q += 32) {
        const int r = q / 8, c = q % 8;
        if (simp)
            J[r][c] = c < 4 ? 0.0 : (F[1 + (c - 4)][r] - F[0][r]) / d_edot;
        else
            J[r][c] = (F[1 + c][r] - F[0][r]) / (c < 4 ? d_e : d_edot);
    }
    __syncwarp();
    // generalized force of the linear tilt: (Fx - My/L, Fy + Mx/L, My/L, -Mx/L)
    auto gen = [L](int r, double fx, double fy, double mx, double my) {
        const double t = (r == 0 || r == 2 ? my : mx) / L;
        return r == 0 ? fx - t : r == 1 ? fy + t : r == 2 ? t : -t;
    };
    {
        const int r = lane & 3, c = (lane >> 2) & 3, at = c + (lane < 16 ? 0 : 4);
        (lane < 16 ? Je : Jd)[r][c] = gen(r, J[0][at], J[1][at], J[3][at], J[4][at]);
        if (lane < 4) G[r] = gen(r, F[0][0], F[0][1], F[0][3], F[0][4]) + F_ext[r];
    }
    __syncwarp();
    // general: (J_edot + dt J_e) delta = -G - J_e (e_prev + dt edot - e);
    // simplified (Eq. 2.20-2.21): J_edot delta = -G
    if (lane < 16) {
        const int r = lane >> 2, c = lane & 3;
        A[r][c] = simp ? Jd[r][c] : Jd[r][c] + dt * Je[r][c];
    } else if (lane < 20) {
        const int r = lane - 16;
        double s = 0.0;
        if (!simp)
            for (int c = 0; c < 4; ++c) s += Je[r][c] * (e_prev[c] + dt * base[4 + c] - base[c]);
        A[r][4] = -G[r] - s;
    }
    __syncwarp();
    int status = 0;
    // Gaussian elimination with partial pivoting
    const int row = lane / 5, col = lane - 5 * row;
    for (int k = 0; k < 4 && status == 0; ++k) {
        int best = k;
        for (int r = k + 1; r < 4; ++r)
            if (fabs(A[r][k]) > fabs(A[best][k])) best = r;
        if (A[best][k] == 0.0 || !isfinite(A[best][k])) {
            status = -4;
            break;
        }
        double a = 0.0;
        if (lane < 20) a = A[row == k ? best : row == best ? k : row][col];
        __syncwarp();
        if (lane < 20) A[row][col] = a;
        __syncwarp();
        if (lane < 20 && row > k && col >= k) {
            const double f = A[row][k] / A[k][k];
            a -= f * A[k][col];
        }
        __syncwarp();
        if (lane < 20) A[row][col] = a;
        __syncwarp();
    }
    for (int q = lane; q < 12; q += 32) result[q] = loads[q];
    for (int q = lane; q < 48; q += 32) result[12 + q] = J[q / 8][q % 8];
    if (lane < 4) result[60 + lane] = G[lane];
    double delta[4] = {0, 0, 0, 0};
    if (status == 0) {
#pragma unroll
        for (int r = 3; r >= 0; --r) {
            double s = A[r][4];
#pragma unroll
            for (int c = r + 1; c < 4; ++c) s -= A[r][c] * delta[c];
            delta[r] = s / A[r][r];
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (lane != q) continue;
        const double ed = base[4 + q] + delta[q];
        result[64 + 4 + q] = ed;
        // general: e = e_prev + dt edot_new; simplified: e += dt delta (Eq. 2.22)
        result[64 + q] = simp ? base[q] + dt * delta[q] : e_prev[q] + dt * ed;
    }
    if (lane == 0) result[72] = (double)status;
}

int launch_picard_update(const double *loads, const PicardIn &in, double dt, double d_e,
                         double d_edot, double L, double *result, cudaStream_t s)
{
    k_picard<<<1, 32, 0, s>>>(loads, in, dt, d_e, d_edot, L, result);
    return cuda_status(cudaGetLastError());
}

}  // namespace gmaf
