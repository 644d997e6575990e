// Declarations of the CG / multigrid kernels' launchers (rhi_linear.cu).
#pragma once

#include "rhi_internal.cuh"

namespace rhi {

// One level's 7-point operator, stored per face: the face below cell c along axis ax carries
// W[ax][c], the coupling of row c to its lower neighbour, and Wp[ax][c], the coupling of the
// lower neighbour's row to c:
//   (A x)_c = diag_c x_c - sum_ax (W[ax]_c x_lo(ax) + Wp[ax]_hi(ax) x_hi(ax)).
// A symmetric operator has Wp = W (the same arrays); the Newton matrix that keeps dD/dE has
// Wp != W.  Both are 0 on zero-flux boundary faces.
template <typename T>
struct Op {
    int nx, ny, nz;
    long long N;
    FastDiv fd_nx, fd_nxy;
    int per[3];
    const T* diag;
    const T* W[3];       // per lower face: the coupling of the upper cell's row
    const T* Wp[3];      // per lower face: the coupling of the lower cell's row (= W: symmetric)
    const T* wid;        // omega / diag, read by the multigrid smoothers
    const T* loc;        // diag - the sum of the row's six couplings; symmetric FP64 levels only
    const double* skip;  // when not null and *skip != 0 the kernel returns at once (the second
                         // half of a BiCGStab iteration after the solve converged at its middle)
};

// Non-symmetric 7-point operator (the Schur matrix with dD/dE kept):
// (A x)_c = diag_c x_c - sum_ax (Q[ax]_c x_lo + P[ax]_hi x_hi), P and Q per lower face.
struct OpNS {
    int nx, ny, nz;
    long long N;
    FastDiv fd_nx, fd_nxy;
    int per[3];
    const double* diag;
    const double* P[3];
    const double* Q[3];
    const double* skip;  // as Op::skip
};

// The coarse end of a V-cycle as one launch (rhi_mgtail.cu): up to MG_TAIL_LEVELS levels within
// MG_TAIL_SMEM bytes of shared memory per block (at most 3 values of 2048 + 512 x 16 levels).
// mg_tail_fits: a level of N cells, the next of N_next (0: none), can start it.  mg_tail_init: the
// blocks of the cluster on the current device; called for every handle.
constexpr int MG_TAIL_LEVELS = 18;
constexpr int MG_TAIL_SMEM = 128 * 1024;
template <typename T> bool mg_tail_fits(long long N, long long N_next, int blocks);
// one coarse level of the hierarchy build (rhi_linear.cu): its size and arrays (loc, wp: may be null)
template <typename T>
struct MgLevel {
    int nx, ny, nz;
    long long N;
    T *diag, *wid, *loc, *w[3], *wp[3];
};
// levels of at most this many cells (one warp per sub-partition of the cluster's SMs) are built by one
// cluster launch together
constexpr long long MG_BUILD_TAIL = 2048;
// BiCGStab's p = r + beta (p - omega v) with the scalars of scal, and rh = r after a restart (k_bicg_p)
struct BicgP {
    const double *scal = nullptr, *r = nullptr, *v = nullptr;
    double *p = nullptr, *rh = nullptr;
};
template <typename T>
struct MgTail {
    Op<T> op[MG_TAIL_LEVELS];
    int n, blocks;
    int pre, post, coarse;      // sweeps
    T omega;
    const T* b;                 // right-hand side of the first level, or in FP64 (b64), or of up
    const double* b64;
    BicgP up;
    T* x;                       // result, in T and / or FP64
    double* x64;
};
cudaError_t mg_tail_init(int* blocks32, int* blocks64);
cudaError_t mg_build_init();
// A cycle's first two sweeps of a level of N cells as one kernel, which multiplies omega / diag by b where
// the second sweep reads x: one launch and, in memory, the first sweep's x less.  Measured, FP32: 256^3
// 131 -> 99 us, 128^3 24.4 -> 22.1 us, 64^3 about 12.5 -> 7.5 us.  FP64 pays its seven
// multiplications on the FP64 pipe: 32^3 13.1 -> 7.6 us, 64^3 16.8 -> 14.2, 72^3 18.8 -> 18.1, but 80^3
// 21.3 -> 22.6 and 128^3 52.5 -> 69.6 us: the line lies at 64^3, a size below the crossing.
// Returns how many of n sweeps the first launch makes.
template <typename T>
constexpr int mg_first_sweeps(long long N, int n) {
    return n >= 2 && (sizeof(T) == 4 || N <= 1LL << 18) ? 2 : 1;
}

// device scalar slots of the Krylov iterations.  The BiCGStab and CG loops keep their control state
// on the device: S_THR (converged when r.r <= S_THR), S_MAXIT, the iteration count S_ITS, S_DONE
// (nothing left to do in this iteration), S_HALF (converged at the middle of an iteration:
// x += alpha M^-1 p only) and S_CONT (1 while another iteration follows).
// S_BEST / S_BESTIT: the smallest r.r so far and its iteration; S_STALL: the loop ended because
// r.r had not fallen below 0.81 of that best (10% in ||r||) for STALL_ITS iterations.
// Restarts: S_INNER (0: none) is a relative bound on r.r; once r.r falls below S_INNER times
// S_RR0, its value at the start or the last restart, or once the solve stagnates, the next
// iteration restarts from the current x and r with a fresh shadow vector rh = r (S_RST), at
// most MAX_RESTARTS times (S_NRST counts them).
enum { S_RZ = 0, S_PQ, S_ALPHA, S_BETA, S_RR, S_BREAK, S_TMP, S_RHO, S_OMEGA, S_SS, S_TS,
       S_TT, S_RV, S_DONE, S_ITS, S_THR, S_MAXIT, S_INNER, S_HALF, S_CONT, S_BEST, S_BESTIT,
       S_STALL, S_RR0, S_NRST, S_RST, S_NSCAL = 32 };
constexpr int STALL_ITS = 20;
constexpr int MAX_RESTARTS = 8;
// k_reduce's two forms
enum { RED_SUM = 0, RED_MAX };

// Where the last block of a kernel with a dot product takes the partials from and puts the outcome: each
// such kernel has one scalar update on scal (rhi_linear.cu), and those that decide on the loop also set the
// CUDA-graph conditional handle cond (0: none).  count null: partials only, no update.
struct Finish {
    double* partials = nullptr;
    unsigned* count = nullptr;
    double* scal = nullptr;
    unsigned long long cond = 0;
};

// number of blocks of the grid-stride streaming kernels (= number of partial sums)
int stream_blocks(long long N);

// timing / counting hook called around every launch
struct LaunchHook {
    virtual void begin(const char* name) = 0;
    virtual void end() = 0;
    virtual ~LaunchHook() {}
};

// Once per process, before the first multigrid launch: the shared-memory limit of the staged
// sweep and the address of its wait-timeout flag.
cudaError_t linear_kernels_init();
// The staged sweep's wait-timeout flag into *host (pinned), on stream st; and its reset.
cudaError_t bulk_wait_flag_read(int* host, cudaStream_t st);
cudaError_t bulk_wait_flag_clear(cudaStream_t st);

struct LinLaunch {
    cudaStream_t st;
    LaunchHook* hook;
    long long fine_N = -1;      // smoothing sweeps on a level of this size get their own name
    // device flag handed to the multigrid, conversion and BiCGStab second-half kernels: they
    // return at once while it is non-zero (null: always run)
    const double* skip = nullptr;
    LinLaunch(cudaStream_t s, LaunchHook* h);
    void begin(const char* name);
    cudaError_t end();

    cudaError_t matvec_dot(const Op<double>& A, const double* p, double* q, const Finish& F);
    cudaError_t cg_xr(long long N, const double* scal, double* x, double* r, const double* p,
                      const double* q, float* r32, const Finish& F);
    // p = z at the loop's first iteration, else z + beta p.  jacobi_dot: z = r / diag, and CG's beta
    cudaError_t cg_p(long long N, const double* scal, const double* z, double* p);
    cudaError_t jacobi_dot(long long N, const double* r, const double* diag, double* z,
                           const Finish& F);
    // CG's r.z and beta
    cudaError_t cg_beta(long long N, const double* r, const double* z, const Finish& F);
    // r32 (may be null), here and above: the FP32 copy of r
    cudaError_t cg_init(long long N, const double* b, double* r, double* x, float* r32,
                        const Finish& F);
    // sum (RED_SUM) or max (RED_MAX) of n partials into scal[slot]
    cudaError_t reduce(const double* part, int n, double* scal, int op, int slot);
    // BiCGStab (right-preconditioned) building blocks
    cudaError_t matvec_ns(const OpNS& A, const double* x, double* y, const double* w1, int two_dots,
                          const Finish& F);
    cudaError_t bicg_init(long long N, const double* b, double* r, double* rh, double* x,
                          const Finish& F);
    // p = r at the loop's first iteration and after a restart (then also rh = r), else the update;
    // p32 (may be null): its FP32 copy
    cudaError_t bicg_p(long long N, const double* scal, const double* r, const double* v,
                       double* p, double* rh, float* p32);
    cudaError_t bicg_s(long long N, const double* scal, const double* r, const double* v,
                       double* s, float* s32, const Finish& F);
    // the x / r update: converged at the middle of the iteration (S_HALF) x += alpha ph only;
    // after a breakdown nothing
    cudaError_t bicg_xr(long long N, const double* scal, double* x, const double* ph,
                        const double* sh, const double* s, const double* t, double* r, const double* rh,
                        const Finish& F);
    cudaError_t from_f32(long long N, const float* x, double* z);

    // out64 (not for the first sweep): the result goes there in FP64 instead of to xout
    template <typename T>
    cudaError_t smooth(const Op<T>& A, const T* b, const T* xin, T* xout, T omega, int first,
                       double* out64 = nullptr);
    template <typename T>
    cudaError_t mg_tail(const MgTail<T>& M);
    template <typename T>
    cudaError_t restrict_res(const Op<T>& A, const T* b, const T* x, int cnx, int cny, int cnz,
                             T* bc);
    template <typename T>
    cudaError_t prolong(int nx, int ny, int nz, int cnx, int cny, const T* xc, T* xf);
    // coarse level c of A
    template <typename TF, typename TC>
    cudaError_t build_level(const Op<TF>& A, const MgLevel<TC>& c, double omega);
    // the n coarse levels c of A, each from the one before, in one launch of `blocks` blocks; the first has
    // at most MG_BUILD_TAIL cells
    template <typename TF, typename TC>
    cudaError_t build_levels(const Op<TF>& A, const MgLevel<TC>* c, int n, double omega, int blocks);
    // finest level of a symmetric operator: wid = omega / diag (smoothers) and, if loc is not null,
    // loc = diag - (six faces) (FP64 restriction), evaluated in TF and rounded to TO
    template <typename TF, typename TO>
    cudaError_t level_prep(const Op<TF>& A, double omega, TO* wid, TO* loc);
    // FP32 copy of a symmetric FP64 operator
    cudaError_t cast_op(const Op<double>& A, float* d, float* const* w);
    cudaError_t to_f32(long long N, const double* a, float* b);
};

}  // namespace rhi
