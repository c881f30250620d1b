// Launch shapes of the resident PCG, the scaled matrix (gmaf_resident_s.cu) and the FP64 kernels
// of gmaf_resident.cuh.
#include "gmaf_resident.cuh"
#include "gmaf_pcg_host.cuh"

#include <algorithm>
#include <cstdlib>

namespace gmaf {

ResKernel res_kernel_f64(int vec, int rr, bool cs)
{
#define GMAF_RES(V, R)                                              \
    if (vec == V && rr == R) {                                      \
        if (cs) GMAF_RES_KERNEL((k_resident<double, V, R, true>));  \
        GMAF_RES_KERNEL((k_resident<double, V, R, false>));         \
    }
    GMAF_RES(1, 1) GMAF_RES(1, 2) GMAF_RES(1, 4) GMAF_RES(1, 8)
    GMAF_RES(2, 1) GMAF_RES(2, 2) GMAF_RES(2, 4)
#undef GMAF_RES
    return {};
}

// ------------------------------------------------------------------ scaled matrix

static size_t pad256(size_t b) { return (b + 255) / 256 * 256; }

// s^2 = minv (of scale A): aE and aN of s A s, Q = 1 / s^2, s, and the diagonal where it is not
// the constant w.
static __global__ void __launch_bounds__(kThreads)
k_res_scaled(const double *__restrict__ D, const double *__restrict__ aE, const double *__restrict__ aN,
             const double *__restrict__ minv, double w, int nth, int nz, unsigned m, double *__restrict__ E,
             double *__restrict__ N, double *__restrict__ Q, double *__restrict__ s, double *__restrict__ diag,
             double *__restrict__ scale_out)
{
    const double scale = ldexp(1.0, -ilogb(D[0])), root = sqrt(w);
    if (blockIdx.x == 0 && threadIdx.x == 0) *scale_out = scale;
    for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < m; q += gridDim.x * blockDim.x) {
        const unsigned row = q / (unsigned)nth, i = q - row * (unsigned)nth;
        const unsigned e = i + 1 == (unsigned)nth ? q - i : q + 1;
        const unsigned n = row % (unsigned)nz + 1 < (unsigned)nz ? q + nth : q;     // (aN of the last row is not read)
        if (minv) {
            const double mi = minv[q];
            E[q] = aE[q] * sqrt(mi) * sqrt(minv[e]);
            N[q] = aN[q] * sqrt(mi) * sqrt(minv[n]);
            s[q] = sqrt(mi / scale);
            Q[q] = scale / mi;
            diag[q] = D[q] * mi;
        } else {
            const double d = D[q] * scale;
            E[q] = aE[q] * scale * w * rsqrt(d * (D[e] * scale));
            N[q] = aN[q] * scale * w * rsqrt(d * (D[n] * scale));
            s[q] = root * rsqrt(d);
            Q[q] = d / w;
        }
    }
}

size_t res_scaled_bytes(long long m, bool with_d)
{
    return (size_t)(with_d ? 5 : 4) * pad256((size_t)m * sizeof(double)) + 256;
}

int res_scaled(const double *D, const double *aE, const double *aN, const double *minv, double w, int nth, int nz,
               long long m, void *coef, int num_sms, cudaStream_t s, ResParams<double> *q)
{
    double *f[5];
    for (int k = 0; k < 5; ++k) f[k] = (double *)((char *)coef + 256 + k * pad256((size_t)m * sizeof(double)));
    q->scale = (const double *)coef;
    q->aE = f[0];
    q->aN = f[1];
    q->Q = f[2];
    q->s = f[3];
    q->D = minv ? f[4] : nullptr;
    q->dg = w;
    k_res_scaled<<<stream_grid(m, num_sms), kThreads, 0, s>>>(D, aE, aN, minv, w, nth, nz, (unsigned)m, f[0], f[1],
                                                              f[2], f[3], f[4], (double *)coef);
    return cuda_status(cudaGetLastError());
}

// ------------------------------------------------------------------ launch shapes

unsigned res_polls()
{
    const char *v = std::getenv("GMAF_RESIDENT_POLLS");
    const long long n = v ? std::atoll(v) : 0;
    return n >= 1 && n < (long long)kResPolls ? (unsigned)n : kResPolls;
}

static long long round16(long long b) { return (b + 15) / 16 * 16; }

// Shared memory of a plan: u, rows and edges; then, as far as there is room, the coefficients and
// x; the tensor memory forms keep x and 1 / s^2 (1), the first rows' aE (2) or omega/D (3).
static bool layout(ResPlan &pl, int nth, int sz, bool *cs)
{
    const int kMax = kResSmem;
    const bool scaled = pl.tm == 1 || pl.tm == 2;
    const long long row = (long long)kResThreads * pl.vec * sz, field = pl.rr * row;
    const long long rows = (long long)(scaled ? res_tm_rows(pl.nrr, sz) : 6 + 2 * pl.nrr) * nth * sz;
    const long long edges = scaled ? (long long)(pl.rows + 2) * (6 * pl.nseg + 5) * sz
                                   : (long long)(pl.rows + 1) * (3 * kResSegs + 2) * sz;
    const long long need = field + round16(rows) + round16(edges);
    if (rows > kMax || edges > kMax || need > kMax) return false;
    *cs = !pl.tm && need + 4 * field <= kMax;
    long long o = field * (*cs ? 5 : 1);
    pl.o_rows = (int)o;
    o += round16(rows);
    pl.o_edge = (int)o;
    o += round16(edges);
    pl.o_x = pl.o_q = -1;
    pl.o_keep = pl.keep = pl.ri = 0;
    const int left = (int)std::min<long long>(pl.rr, (kMax - o) / row);
    if (pl.tm == 2) {
        pl.o_keep = (int)o;
        pl.keep = left;
        o += left * row;
    } else if (pl.tm == 3) {
        pl.o_x = (int)o;
        pl.ri = left;
        o += left * row;
    } else if (left == pl.rr) {
        pl.o_x = (int)o;
        o += field;
        if (pl.tm == 1 && o + field <= kMax) {
            pl.o_q = (int)o;
            o += field;
        }
    }
    pl.smem = (int)o;
    return true;
}

template <typename T>
bool res_plan(int nth, int nz, int K, bool vec_ok, int num_sms, ResPlan *out)
{
    const int sz = (int)sizeof(T);
    ResPlan pl{};
    const int blocks = std::min(num_sms, kResMaxBlocks);
    if (K < 1 || K > blocks) return false;
    // whole rows, spread over as many blocks as there are: an exchange costs the same
    // for 32 blocks as for 152, and rows shared among more blocks take less time
    pl.bpc = std::min(nz, blocks / K);
    pl.rows = (nz + pl.bpc - 1) / pl.bpc;
    pl.bpc = (nz + pl.rows - 1) / pl.rows;
    pl.grid = pl.bpc * K;
    // columns a thread and rows a run: in FP64, where one warp instruction holds a
    // quarter of the SM's FP64 pipe for 64 cycles, the pair that gives the fullest
    // quarter the fewest cells; in FP32 16-byte columns; the shortest runs that fit.
    // Whatever fits is faster here than in the phase kernels, up to the largest: us an
    // iteration in FP32 on 9 conditions of 640 x 256 cells 14.8 against 54, of 700 x 300
    // 33 against 57, of 1024 x 512 39 against 68; in FP64 on 9 of 512 x 256 41 against 76,
    // on 5 of 700 x 384 56 against 95
    long long best = 0;
    for (int vec : {16 / sz, 1}) {
        if (vec > 1 && !vec_ok) continue;
        if (best && sz == 4) break;
        const long long ncg = nth / vec;
        if (ncg > kResThreads) continue;
        int P = 1;
        while (P < ncg && P < 32) P *= 2;
        if (ncg > 32) P = (int)((ncg + 31) / 32 * 32);
        for (int rr : {1, 2, 4, 8, 16}) {
            // (tensor memory takes 16 bytes a row and thread)
            if (rr == 16 && vec * sz != 16) break;
            ResPlan t = pl;
            t.nrr = (pl.rows + rr - 1) / rr;
            if ((long long)P * t.nrr > kResThreads) continue;
            t.tm = res_tm(rr, vec, sz);
            t.vec = vec;
            t.rr = rr;
            t.ncg = (int)ncg;
            t.P = P;
            t.nseg = (int)((ncg + 31) / 32);
            bool cs = false;
            if (!layout(t, nth, sz, &cs)) continue;
            t.k = t.tm == 3   ? res_kernel_tm()
                  : t.tm      ? res_kernel_s(sz, rr)
                  : sz == 4   ? res_kernel_f32(vec, rr, cs)
                              : res_kernel_f64(vec, rr, cs);
            const long long warps = ((long long)P * t.nrr + 31) / 32;
            const long long cells = (warps + 3) / 4 * vec * rr;
            if (t.k.fn && (!best || cells < best)) {
                best = cells;
                pl = t;
            }
            break;
        }
    }
    if (!best) return false;
    pl.threads = (pl.P * pl.nrr + 31) / 32 * 32;
    // flagged rows: four of T, and for FP32 two of doubles behind them
    pl.halo_bytes = (size_t)pl.grid * 4 * nth * 2 * sz + (sz == 4 ? (size_t)pl.grid * 2 * nth * 16 : 0);
    *out = pl;
    return true;
}

template <typename T>
void res_fill(const ResPlan &pl, ResParams<T> *q)
{
    q->bpc = pl.bpc;
    q->threads = pl.threads;
    q->P = pl.P;
    q->ncg = pl.ncg;
    q->nrr = pl.nrr;
    q->rows = pl.rows;
    q->o_rows = pl.o_rows;
    q->o_edge = pl.o_edge;
    q->o_x = pl.o_x;
    q->nseg = pl.nseg;
    q->o_q = pl.o_q;
    q->o_keep = pl.o_keep;
    q->keep = pl.keep;
    q->ri = pl.ri;
    q->halo_row = q->nth * ((int)sizeof(T) / 4);
    q->halo64 = q->halo + (size_t)pl.grid * 4 * q->halo_row;
}

template <typename T>
cudaError_t res_launch(const ResPlan &pl, ResParams<T> &q, cudaStream_t s)
{
    smem_optin(*pl.k.opted, pl.k.fn, kResSmem);
    void *args[] = {(void *)&q};
    return cudaLaunchCooperativeKernel(pl.k.fn, dim3(pl.grid), dim3(pl.threads + 32), args, pl.smem, s);
}

cudaError_t res_preload64(cudaStream_t s)
{
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, (const void *)k_res_scaled);
    for (int k = 0; k < 18 && e == cudaSuccess; ++k) {
        const int vec = 1 + (k & 1), rr = 1 << (k >> 2);
        ResPlan pl{};
        pl.k = k >= 16 ? res_kernel_s(8, k == 16 ? 8 : 16) : res_kernel_f64(vec, rr, (k & 2) != 0);
        if (!pl.k.fn) continue;
        pl.grid = 1;
        pl.threads = 32;
        pl.smem = kResSmem;
        ResParams<double> q{};
        q.bpc = q.groups = 1;           // (mask 0: the group does not run)
        q.threads = pl.threads;
        e = res_launch<double>(pl, q, s);
    }
    return e;
}

template bool res_plan<float>(int, int, int, bool, int, ResPlan *);
template bool res_plan<double>(int, int, int, bool, int, ResPlan *);
template void res_fill<float>(const ResPlan &, ResParams<float> *);
template void res_fill<double>(const ResPlan &, ResParams<double> *);
template cudaError_t res_launch<float>(const ResPlan &, ResParams<float> &, cudaStream_t);
template cudaError_t res_launch<double>(const ResPlan &, ResParams<double> &, cudaStream_t);

}  // namespace gmaf
