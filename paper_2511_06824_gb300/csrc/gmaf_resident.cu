// Launch shapes of the resident PCG (gmaf_resident.cuh) and its FP64 kernels.
#include "gmaf_resident.cuh"

#include <algorithm>

namespace gmaf {

const void *res_kernel_f64(int vec, int rr, bool cs)
{
#define GMAF_RES(V, R)                                                              \
    if (vec == V && rr == R)                                                        \
        return cs ? (const void *)k_resident<double, V, R, true>                    \
                  : (const void *)k_resident<double, V, R, false>;
    GMAF_RES(1, 1) GMAF_RES(1, 2) GMAF_RES(1, 4) GMAF_RES(1, 8)
    GMAF_RES(2, 1) GMAF_RES(2, 2) GMAF_RES(2, 4) GMAF_RES(2, 8)
#undef GMAF_RES
    return nullptr;
}

static long long round16(long long b) { return (b + 15) / 16 * 16; }

template <typename T>
bool res_plan(int nth, int nz, int K, bool vec_ok, int num_sms, ResPlan *out)
{
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
    // quarter the fewest cells; in FP32 16-byte columns; the shortest runs that fit
    long long best = 0;
    for (int vec : {16 / (int)sizeof(T), 1}) {
        if (vec > 1 && !vec_ok) continue;
        if (best && sizeof(T) == 4) break;
        const long long ncg = nth / vec;
        if (ncg > kResThreads) continue;
        int P = 1;
        while (P < ncg && P < 32) P *= 2;
        if (ncg > 32) P = (int)((ncg + 31) / 32 * 32);
        for (int rr : {1, 2, 4, 8}) {
            const int nrr = (pl.rows + rr - 1) / rr;
            if ((long long)P * nrr > kResThreads) continue;
            const long long warps = ((long long)P * nrr + 31) / 32;
            const long long cells = (warps + 3) / 4 * vec * rr;
            if (!best || cells < best) {
                best = cells;
                pl.vec = vec;
                pl.rr = rr;
                pl.nrr = nrr;
                pl.ncg = (int)ncg;
                pl.P = P;
            }
            break;
        }
    }
    if (!best && sizeof(T) == 4 && vec_ok && nth / 4 <= kResThreads) {
        // the largest systems (one joint system, 4 columns a thread): with an iteration on 9
        // conditions of 700 x 300 cells in 33 us against 57 of the phase kernels and of 1024 x
        // 512 in 39 against 68, whatever fits comes here
        pl.tm = true;
        pl.vec = 4;
        pl.rr = kTmRows;
        pl.ncg = nth / 4;
        pl.P = 1;
        while (pl.P < pl.ncg && pl.P < 32) pl.P *= 2;
        if (pl.ncg > 32) pl.P = (pl.ncg + 31) / 32 * 32;
        pl.nrr = (pl.rows + kTmRows - 1) / kTmRows;
        best = (long long)pl.P * pl.nrr <= kResThreads;
    }
    if (!best) return false;
    pl.threads = (pl.P * pl.nrr + 31) / 32 * 32;
    // shared memory: u, rows and edges, r for the longest runs; then, as far as there is
    // room, the coefficients, then x
    const int kMax = 226 * 1024;         // of the 227 KB a block can have (a little is static)
    const int sz = (int)sizeof(T);
    const long long field = (long long)pl.rr * kResThreads * pl.vec * sz;
    const long long rows = (long long)(6 + 2 * pl.nrr) * nth * sz;
    const long long edges = (long long)(pl.rows + 1) * (3 * kResSegs + 2) * sz;
    const bool rs = !pl.tm && res_r_shared(pl.rr, pl.vec, sz);
    const long long need = field * (rs ? 2 : 1) + round16(rows) + round16(edges);
    if (rows > kMax || edges > kMax || need > kMax) return false;
    const bool cs = !pl.tm && need + 4 * field <= kMax;
    long long o = field * ((rs ? 2 : 1) + (cs ? 4 : 0));
    pl.o_rows = (int)o;
    o += round16(rows);
    pl.o_edge = (int)o;
    o += round16(edges);
    pl.o_x = -1;
    if (pl.tm) {
        // omega/D of as many rows of a run as there is room for
        pl.o_x = (int)o;
        pl.ri = (int)std::min<long long>(kTmRows, (kMax - o) / (field / kTmRows));
        o += pl.ri * (field / kTmRows);
    } else if (o + field <= kMax) {
        pl.o_x = (int)o;
        o += field;
    }
    pl.smem = (int)o;
    pl.fn = pl.tm ? res_kernel_tm() : sz == 4 ? res_kernel_f32(pl.vec, pl.rr, cs) : res_kernel_f64(pl.vec, pl.rr, cs);
    if (!pl.fn) return false;
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
    q->ri = pl.ri;
    q->halo_row = q->nth * ((int)sizeof(T) / 4);
    q->halo64 = q->halo + (size_t)pl.grid * 4 * q->halo_row;
}

template <typename T>
cudaError_t res_launch(const ResPlan &pl, ResParams<T> &q, cudaStream_t s)
{
    cudaError_t e = cudaFuncSetAttribute(pl.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, pl.smem);
    if (e != cudaSuccess) return e;
    void *args[] = {(void *)&q};
    return cudaLaunchCooperativeKernel(pl.fn, dim3(pl.grid), dim3(pl.threads + 32), args, pl.smem, s);
}

template bool res_plan<float>(int, int, int, bool, int, ResPlan *);
template bool res_plan<double>(int, int, int, bool, int, ResPlan *);
template void res_fill<float>(const ResPlan &, ResParams<float> *);
template void res_fill<double>(const ResPlan &, ResParams<double> *);
template cudaError_t res_launch<float>(const ResPlan &, ResParams<float> &, cudaStream_t);
template cudaError_t res_launch<double>(const ResPlan &, ResParams<double> &, cudaStream_t);

}  // namespace gmaf
