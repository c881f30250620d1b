// Host-visible part of the resident PCG (gmaf_resident.cuh): the shape of a launch
// and the launch itself, used by the joint solver (gmaf_pcg.cu) and the
// allocation-free solve (gmaf_noalloc.cu).  Internal; not part of the ABI.
#pragma once

#include <atomic>
#include <cstddef>

#include "gmaf_internal.cuh"

namespace gmaf {

constexpr int kResThreads = 512;        // most threads that own rows (one more warp exchanges)
constexpr int kResMaxBlocks = 160;      // most blocks of a launch (they are counted in a byte)
constexpr int kResSmem = 225 * 1024;    // shared memory of a block (of 227 KB; 1.1 KB more is static)
constexpr int kResGroupWords = 16;      // 8-byte words of a group of blocks for its sums
constexpr int kResSegs = kResThreads / 32;   // segments of 32 threads in a row, at most
constexpr int kResVariant = 50000000;   // gmaf_solve_info.kernel_variant: + 1000 VEC + 10 RR

// Where a kernel keeps r and the product: in registers (0), or, with over 64 bytes a thread, in
// tensor memory: with the couplings there too (1, runs of 8 rows), or in runs of 16 with the
// couplings streamed from L2 (FP64: 2, FP32: 3).
__host__ __device__ constexpr int res_tm(int rr, int vec, int size)
{
    return rr * vec * size <= 64 ? 0 : rr == 8 ? 1 : size == 8 ? 2 : 3;
}
// How far above the tolerance the true residual of a first FP64 run may be.  In the scaled forms
// the recurrence is that of a matrix rounded to the last bits and drifts from the true residual
// (by 4e-14 of the right-hand side on 512 x 256 cells, 2e-13 on 1000 x 250, 1e-11 on 511 x 5,
// where the unscaled forms drift by a tenth of it), so a run that ends well above is restarted
// from its true residual, which takes that out; the unscaled forms keep the phase kernels' limit.
// (Below ten times the tolerance the first run's solution is good, and stays if the restart finds no
// room for its residual or no iterations left.)
constexpr double res_limit(int tm) { return tm ? 1.25 : 10.0; }

// Rows of n_theta values that a block of form 1 or 2 keeps in shared memory.
__host__ __device__ constexpr int res_tm_rows(int nrr, int size) { return size == 8 ? 4 + 3 * nrr : 5 + 4 * nrr; }

// Scalars.status of a run that the phase kernels have to take over (not statuses of the ABI): a sum
// of squares outside the range that the exchange forms sums in; a wait for another block that ran out.
constexpr int kResBeyond = 1, kResLate = 2;
inline bool res_gives_way(int status) { return status > 0; }

// Polls of about a microsecond before a wait runs out, unless the host sets fewer: about 2 s.
constexpr unsigned kResPolls = 1u << 21;
// The limit: GMAF_RESIDENT_POLLS (fault injection: a test can make a wait run out) or kResPolls.
unsigned res_polls();

// FP64 (T = double): one run.  FP32: the whole mixed-precision solve.
enum ResMode {
    kResFresh = 0,      // r = b - A p (p = 0 with zero_init)
    kResRestart = 1     // r handed in, p continued, the count and the norm of b kept from the last run
};

// Kernel parameters.  o_*: byte offsets in shared memory (-1: the array stays in
// global memory).
template <typename T>
struct ResParams {
    int nth, nz, bpc, groups;           // bpc blocks a condition; groups: 1 joint system or K
    int threads, P, ncg, nrr, rows, nseg;
    int precond, mode, zero_init, max_iter, guard_limit;
    int o_rows, o_edge, o_x, o_q, o_keep, keep;     // keep: rows of a run whose E stays on the SM
    unsigned polls;                     // limit of a wait (FP32: for a neighbour's row)
    unsigned epoch;                     // exchanges of this run are epoch + 1, epoch + 2, ...
    unsigned long long mask;            // groups that run
    unsigned long long optional;        // scaled: groups whose p is within the limit already: a restart
                                        // that ends without meeting the tolerance leaves it
    long long n;
    const T *D, *invD, *aE, *aN;        // (scaled: of s A s; D null where it is the constant dg)
    const int *cslot;
    const T *b, *r_in;
    T *p;                               // (FP32: scratch for x when it does not fit on the SM)
    // scaled FP64: 1 / s^2, s, and scratch for x; the system is D64 ..., p64
    const T *Q, *s;
    T *x;
    T dg;
    Scalars *sc;                        // [groups]
    double eps;
    // FP32: the FP64 system and its refinement
    const double *D64, *aE64, *aN64, *S64, *scale;   // scale: FP32 or scaled matrix: of scale A
    double *p64, *r64;
    unsigned long long *halo64;         // flagged FP64 rows, [blocks][2]
    const float *dbnd;                  // the largest systems: Dirichlet term of the diagonal, [slots][2][nth]
    int ri;                             //   and rows of a run whose omega/D is in shared memory
    double inner_floor;                 // reduction of a run
    int continued, max_outer;
    int grid64;                         // blocks of k_resid64 on this system, and sums of
    double *warps64;                    // its warps: the norm is added up in that kernel's order
    int pairs64;                        // the rows of the FP64 arrays start on 16-byte boundaries
    unsigned long long *words;          // [groups][kResGroupWords], zero at the start of the run
    unsigned long long *halo;           // flagged rows, [blocks][4]
    int halo_row;                       // 8-byte words of one flagged row
    unsigned long long *times;          // ns in A, B and set-up, counts of A and B, ns and count
                                        // of FP64 residuals (added to; or null)
};

// A kernel and the devices on which it is opted in to kResSmem.  (The attribute is the kernel's,
// not the launch's: set to a plan's own size before each launch, it was lowered between another
// thread's setting and launch, which then failed.)
struct ResKernel {
    const void *fn;
    std::atomic<unsigned long long> *opted;
};

struct ResPlan {
    ResKernel k;
    int grid, smem, vec, rr;
    int bpc, threads, P, ncg, nrr, rows, nseg;
    int o_rows, o_edge, o_x, o_q, o_keep, keep, ri;
    int tm;                             // res_tm
    size_t halo_bytes;                  // flagged rows, zero before the first launch
};

// Whether (and how) a solve of K conditions on nth x nz fits on the SMs: vec_ok says
// that rows can be read 16 bytes at a time.
template <typename T>
bool res_plan(int nth, int nz, int K, bool vec_ok, int num_sms, ResPlan *out);

// Fills the plan's part of the parameters.
template <typename T>
void res_fill(const ResPlan &pl, ResParams<T> *q);

// Kernel of a plan (compiled for T in a translation unit of its own).
ResKernel res_kernel_f32(int vec, int rr, bool cs);
ResKernel res_kernel_f64(int vec, int rr, bool cs);
ResKernel res_kernel_tm();
constexpr int kTmRows = 16;             // rows of a run of k_resident_tm
ResKernel res_kernel_s(int size, int rr);

// The scaled FP64 matrix of m cells: coef (res_scaled_bytes) receives aE, aN, Q, s and (with minv)
// D.  minv: the preconditioner's diagonal, null for w / D.
size_t res_scaled_bytes(long long m, bool with_d);
int res_scaled(const double *D, const double *aE, const double *aN, const double *minv, double w, int nth, int nz,
               long long m, void *coef, int num_sms, cudaStream_t s, ResParams<double> *q);

// Loads every FP64 kernel on the current device and launches it once without work, so that later
// launches allocate neither code nor local memory.
cudaError_t res_preload64(cudaStream_t s);

// Cooperative launch; cudaErrorCooperativeLaunchTooLarge when the blocks cannot all
// be resident (a partitioned GPU): the caller then takes the phase kernels.
template <typename T>
cudaError_t res_launch(const ResPlan &pl, ResParams<T> &q, cudaStream_t s);

}  // namespace gmaf
