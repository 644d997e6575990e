// Scalar Schur-system solve (Sec. 3.2.1, step (ii)): conjugate gradients on the 7-point
// matrix S, preconditioned by one geometric multigrid V-cycle (FP64, or FP32 for the mixed-
// precision form) or by Jacobi.  Reductions are deterministic: per-block partial sums are
// added in a fixed order by the last block to end.
//
// Operator of a level: (A x)_c = diag_c x_c - sum_ax (W[ax]_c x_lo + Wp[ax]_hi x_hi),
// stored per lower face (0 on zero-flux boundary faces): W couples the upper cell's row to the
// lower cell, Wp the lower cell's row to the upper cell.  Symmetric levels pass Wp = W.
#include <cooperative_groups.h>

#include <type_traits>

#include "rhi_linear.cuh"

namespace rhi {

constexpr int LIN_BLOCK = 256;
constexpr int RED_BLOCK = 1024;

// the second half of a converged BiCGStab iteration returns at once
__device__ __forceinline__ bool skipped(const double* skip) { return skip && *skip != 0.0; }

int stream_blocks(long long N) {
    const long long want = (N + LIN_BLOCK - 1) / LIN_BLOCK;
    const long long cap = 152LL * 16;                 // 16 resident blocks per SM x 152 SMs
    return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

// blocks of the kernels that end with a sum: one wave of 8 blocks per SM, since every block adds its
// own partial (a chain of FP64 additions) and takes a ticket
static int sum_blocks(long long N) {
    const long long want = (N + LIN_BLOCK - 1) / LIN_BLOCK;
    const long long cap = 152LL * 8;
    return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

template <typename T>
__device__ __forceinline__ void coords3(const Op<T>& A, long long c, int& i, int& j, int& k) {
    const unsigned cu = (unsigned)c;
    const unsigned kk = fdiv(cu, A.fd_nxy);
    const unsigned r = cu - kk * A.fd_nxy.d;
    const unsigned jj = fdiv(r, A.fd_nx);
    k = (int)kk;
    j = (int)jj;
    i = (int)(r - jj * A.fd_nx.d);
}

// coordinates of index c on an nx x ny x nz grid given the dividers of nx and nx * ny
__device__ __forceinline__ void coords_fd(long long c, const FastDiv& fx, const FastDiv& fxy,
                                          int& i, int& j, int& k) {
    const unsigned cu = (unsigned)c;
    const unsigned kk = fdiv(cu, fxy);
    const unsigned r = cu - kk * fxy.d;
    const unsigned jj = fdiv(r, fx);
    k = (int)kk;
    j = (int)jj;
    i = (int)(r - jj * fx.d);
}

// x after a cycle's first sweep, from x = 0, without that sweep's launch: omega / diag times b
template <typename T>
struct FirstSweep {
    const T* __restrict__ wid;
    const T* __restrict__ b;
    __device__ __forceinline__ T operator[](long long c) const { return wid[c] * b[c]; }
};

// sum over the six neighbours of c of W_face x_neighbour (the off-diagonal part of row c)
template <typename T, typename X>
__device__ __forceinline__ T off_row(const Op<T>& A, const X& x, long long c,
                                     int i, int j, int k) {
    const long long sx = 1, sy = A.nx, sz = (long long)A.nx * A.ny;
    const int n[3] = {A.nx, A.ny, A.nz};
    const int q[3] = {i, j, k};
    const long long s[3] = {sx, sy, sz};
    const int per[3] = {A.per[0], A.per[1], A.per[2]};
    T off = T(0);
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        long long lo, hi;
        bool has_hi = true;
        if (q[ax] > 0) lo = c - s[ax];
        else lo = c + (long long)(n[ax] - 1) * s[ax];            // W = 0 there unless periodic
        if (q[ax] < n[ax] - 1) hi = c + s[ax];
        else if (per[ax]) hi = c - (long long)(n[ax] - 1) * s[ax];
        else { hi = c; has_hi = false; }
        const T wlo = A.W[ax][c];
        off += wlo * T(x[lo]);
        if (has_hi) off += A.Wp[ax][hi] * T(x[hi]);
    }
    return off;
}

// (A x)_c with the six neighbours of c
template <typename T, typename TX>
__device__ __forceinline__ T apply_row(const Op<T>& A, const TX* __restrict__ x, long long c,
                                       int i, int j, int k, T xc) {
    return A.diag[c] * xc - off_row(A, x, c, i, j, k);
}

// one weighted-Jacobi update of cell c from the off-diagonal sum:
// x + omega (b - A x) / diag = (1 - omega) x + (omega / diag) (b + off)
template <typename T>
__device__ __forceinline__ T jacobi_update(T xc, T b, T wi, T off, T omega) {
    return (T(1) - omega) * xc + wi * (b + off);
}

// ---------------------------------------------------------------------------------------------
// Scalar updates.  A kernel with dot products ends with finish(): its last block adds all blocks'
// partials in a fixed order and applies the kernel's update, so that a Krylov iteration needs no separate
// reduction launches (about 3.6 us each inside a graph; the last block adds about 2 us).
//   RED_CG_START:   r.r of r = b: S_RR, counters cleared; done when r.r <= S_THR
//   RED_CG_BETA:    r.z: S_BETA = sum / S_RZ; S_RZ = sum
//   RED_CG_ALPHA:   p.Sp: S_PQ = sum; S_ALPHA = S_RZ / sum (breakdown flag if <= 0)
//   RED_CG_NEXT:    r.r: S_RR, S_ITS += 1; ends when converged, on a breakdown, or at S_MAXIT
//   RED_BICG_ALPHA: sum = rh.v: S_ALPHA = S_RHO / sum
//   RED_BICG_OMEGA: sums t.s and t.t: S_OMEGA
//   RED_BICG_START: r.r of r = b: S_RR = S_RHO = r.r, counters cleared; done when
//                   r.r <= S_THR (or not finite: breakdown).
//   RED_BICG_SS:    s.s: converged at the middle of the iteration when s.s <= S_THR (S_HALF,
//                   S_DONE); a breakdown flagged by the alpha reduction also sets S_DONE.
//   RED_BICG_NEXT:  r.r and rh.r: beta and rho for the next iteration, S_ITS += 1, and the
//                   loop ends when converged (or S_DONE), on a breakdown, or at S_MAXIT.
//                   When r.r has not fallen below 0.81 of its best for STALL_ITS iterations,
//                   or below S_INNER times its value at the last restart, the next iteration
//                   restarts with rh = r (up to MAX_RESTARTS times; the rounding of an FP32
//                   preconditioner slowly erodes the bi-orthogonality BiCGStab relies on); a
//                   stagnation past the last restart ends the loop, and the Newton step is
//                   then that of an inexact Newton iteration.
// The START and NEXT updates write the continue flag to S_CONT and, inside a CUDA graph, to the
// while node's conditional handle: these kernels always run to their end.
enum { RED_CG_START, RED_CG_BETA, RED_CG_ALPHA, RED_CG_NEXT, RED_BICG_START, RED_BICG_ALPHA, RED_BICG_SS,
       RED_BICG_OMEGA, RED_BICG_NEXT };
template <int op>
__device__ __forceinline__ void scalar_update(double* scal, unsigned long long cond, double s, double s2) {
    int cont = 0;
    if (op == RED_CG_START) {
        scal[S_RR] = s;
        scal[S_ITS] = 0.0;
        scal[S_BREAK] = 0.0;
        cont = s > scal[S_THR] && scal[S_MAXIT] >= 1.0;
    } else if (op == RED_CG_BETA) {
        scal[S_BETA] = s / scal[S_RZ];          // (not read in the first iteration)
        scal[S_RZ] = s;
        return;
    } else if (op == RED_CG_ALPHA) {
        scal[S_PQ] = s;
        if (!(s > 0.0)) scal[S_BREAK] = 1.0;
        scal[S_ALPHA] = (s > 0.0) ? scal[S_RZ] / s : 0.0;
        return;
    } else if (op == RED_CG_NEXT) {
        const double its = scal[S_ITS] + 1.0;
        scal[S_ITS] = its;
        scal[S_RR] = s;
        if (!isfinite(s)) scal[S_BREAK] = 1.0;
        cont = scal[S_BREAK] == 0.0 && s > scal[S_THR] && its < scal[S_MAXIT] && its < 1e6;
    } else if (op == RED_BICG_ALPHA) {
        scal[S_RST] = 0.0;                      // a restart's p and rh are in place
        scal[S_RV] = s;
        if (!(s != 0.0)) scal[S_BREAK] = 1.0;
        scal[S_ALPHA] = (s != 0.0) ? scal[S_RHO] / s : 0.0;
        return;
    } else if (op == RED_BICG_OMEGA) {          // t.s, t.t
        scal[S_TS] = s;
        scal[S_TT] = s2;
        scal[S_OMEGA] = (s2 > 0.0) ? s / s2 : 0.0;
        if (!(s2 > 0.0)) scal[S_BREAK] = 1.0;
        return;
    } else if (op == RED_BICG_SS) {
        scal[S_SS] = s;
        if (!isfinite(s)) {
            scal[S_BREAK] = 1.0;
            scal[S_DONE] = 1.0;
        } else if (scal[S_BREAK] != 0.0) {
            scal[S_DONE] = 1.0;
        } else if (!(s > scal[S_THR])) {
            scal[S_HALF] = 1.0;
            scal[S_DONE] = 1.0;
        }
        return;                                    // no loop decision here
    } else if (op == RED_BICG_START) {
        const bool fin = isfinite(s);
        scal[S_RR] = s;
        scal[S_RHO] = s;
        scal[S_ITS] = 0.0;
        scal[S_HALF] = 0.0;
        scal[S_BREAK] = fin ? 0.0 : 1.0;
        scal[S_BEST] = s;
        scal[S_BESTIT] = 0.0;
        scal[S_STALL] = 0.0;
        scal[S_RR0] = s;
        scal[S_NRST] = 0.0;
        scal[S_RST] = 0.0;
        const bool done = !(s > scal[S_THR]) || !fin || !(scal[S_MAXIT] >= 1.0);
        scal[S_DONE] = done ? 1.0 : 0.0;
        cont = !done;
    } else {                                       // RED_BICG_NEXT
        const double its = scal[S_ITS] + 1.0;
        scal[S_ITS] = its;
        if (scal[S_DONE] != 0.0) {
            cont = 0;
        } else {
            const double rho = s2;
            scal[S_RR] = s;
            scal[S_BETA] = (rho / scal[S_RHO]) * (scal[S_ALPHA] / scal[S_OMEGA]);
            scal[S_RHO] = rho;
            const bool brk = !isfinite(s) || !(rho != 0.0) || scal[S_BREAK] != 0.0;
            if (brk) scal[S_BREAK] = 1.0;
            const bool conv = !(s > scal[S_THR]);
            if (s < 0.81 * scal[S_BEST]) {
                scal[S_BEST] = s;
                scal[S_BESTIT] = its;
            }
            bool stall = its - scal[S_BESTIT] >= (double)STALL_ITS;
            const bool inner = scal[S_INNER] > 0.0 && !(s > scal[S_INNER] * scal[S_RR0]);
            if (!conv && !brk && (stall || inner) && scal[S_NRST] < (double)MAX_RESTARTS) {
                // restart from the current x and r: fresh shadow vector rh = r, rho = r.r
                scal[S_RST] = 1.0;
                scal[S_NRST] += 1.0;
                scal[S_RR0] = s;
                scal[S_RHO] = s;
                scal[S_BEST] = s;
                scal[S_BESTIT] = its;
                stall = false;
            }
            if (stall && !conv) scal[S_STALL] = 1.0;
            // (written so that a cap that is not a number also ends the loop)
            cont = !(conv || brk || stall) && its < scal[S_MAXIT] && its < 1e6;
        }
    }
    scal[S_CONT] = cont ? 1.0 : 0.0;
    if (cond) cudaGraphSetConditional((cudaGraphConditionalHandle)cond, cont ? 1u : 0u);
}

// v1 (and v2): this thread's share of the sums; called by every thread of every block.  OP: the
// update the kernel ends with, so that its code holds no other
template <bool TWO, int OP>
__device__ __forceinline__ void finish(const Finish& F, double v1, double v2) {
    __shared__ double sc[S_NSCAL];
    double s1, s2;
    // the scalars by way of shared memory, fetched by every block under its own sum (only the last
    // one, which alone writes them, after every block has its ticket, uses them)
    if (threadIdx.x < S_NSCAL && F.count) sc[threadIdx.x] = __ldcg(F.scal + threadIdx.x);
    if (!grid_sum<LIN_BLOCK, TWO>(v1, v2, F.partials, F.count, s1, s2)) return;
    if (threadIdx.x == 0) scalar_update<OP>(sc, F.cond, s1, s2);
    __syncthreads();
    if (threadIdx.x < S_NSCAL) F.scal[threadIdx.x] = sc[threadIdx.x];
}

// sum or max of partials in a fixed order by one block (where a kernel has too many blocks for its
// last one to add them, or its sum goes to a slot without an update)
__global__ void __launch_bounds__(RED_BLOCK) k_reduce(const double* __restrict__ partials, int n,
                                                      double* __restrict__ scal, int op, int slot) {
    if (op == RED_MAX) {                        // max of non-negative partials
        __shared__ double wmax[RED_BLOCK / 32];
        double m = 0.0;
        for (int q = threadIdx.x; q < n; q += RED_BLOCK) m = fmax(m, partials[q]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
        if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int q = 1; q < RED_BLOCK / 32; ++q) m = fmax(m, wmax[q]);
            scal[slot] = fmax(m, wmax[0]);
        }
        return;
    }
    double acc = 0.0;
    for (int q = threadIdx.x; q < n; q += RED_BLOCK) acc += partials[q];
    const double s = block_sum<RED_BLOCK>(acc);
    if (threadIdx.x == 0) scal[slot] = s;
}

// ---------------------------------------------------------------------------------------------
// CG building blocks (FP64)

__global__ void __launch_bounds__(LIN_BLOCK) k_matvec_dot(const Op<double> A,
                                                          const double* __restrict__ p,
                                                          double* __restrict__ q, const Finish F) {
    double acc = 0.0;
    for (long long c = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; c < A.N;
         c += (long long)gridDim.x * LIN_BLOCK) {
        int i, j, k;
        coords3(A, c, i, j, k);
        const double pc = p[c];
        const double v = apply_row(A, p, c, i, j, k, pc);
        q[c] = v;
        acc += pc * v;
    }
    finish<false, RED_CG_ALPHA>(F, acc, 0.0);
}

// x += alpha p; r -= alpha q; r.r      (alpha = scal[S_ALPHA])
__global__ void __launch_bounds__(LIN_BLOCK) k_cg_xr(long long N, const double* __restrict__ scal,
                                                     double* __restrict__ x, double* __restrict__ r,
                                                     const double* __restrict__ p,
                                                     const double* __restrict__ q,
                                                     float* __restrict__ r32, const Finish F) {
    const double alpha = scal[S_ALPHA];
    double acc = 0.0;
    for (long long c = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; c < N;
         c += (long long)gridDim.x * LIN_BLOCK) {
        x[c] += alpha * p[c];
        const double rv = r[c] - alpha * q[c];
        r[c] = rv;
        if (r32) r32[c] = (float)rv;
        acc += rv * rv;
    }
    finish<false, RED_CG_NEXT>(F, acc, 0.0);
}

// p = z + beta p    (beta = scal[S_BETA]); at the loop's first iteration p = z
__global__ void __launch_bounds__(LIN_BLOCK) k_cg_p(long long N, const double* __restrict__ scal,
                                                    const double* __restrict__ z,
                                                    double* __restrict__ p) {
    const bool first = scal[S_ITS] == 0.0;
    const double beta = first ? 0.0 : scal[S_BETA];
    for (long long c = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; c < N;
         c += (long long)gridDim.x * LIN_BLOCK)
        p[c] = first ? z[c] : z[c] + beta * p[c];
}

// z = r / diag; r.z
__global__ void __launch_bounds__(LIN_BLOCK) k_jacobi_dot(long long N, const double* __restrict__ r,
                                                          const double* __restrict__ diag,
                                                          double* __restrict__ z, const Finish F,
                                                          const double* skip) {
    if (skipped(skip)) return;
    double acc = 0.0;
    for (long long c = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; c < N;
         c += (long long)gridDim.x * LIN_BLOCK) {
        const double rv = r[c];
        const double zv = rv / diag[c];
        z[c] = zv;
        acc += rv * zv;
    }
    finish<false, RED_CG_BETA>(F, acc, 0.0);
}

// r.z
__global__ void __launch_bounds__(LIN_BLOCK) k_cg_beta(long long N, const double* __restrict__ r,
                                                       const double* __restrict__ z, const Finish F) {
    double acc = 0.0;
    for (long long c = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; c < N;
         c += (long long)gridDim.x * LIN_BLOCK)
        acc += r[c] * z[c];
    finish<false, RED_CG_BETA>(F, acc, 0.0);
}

// r = b, x = 0; r.r
__global__ void __launch_bounds__(LIN_BLOCK) k_cg_init(long long N, const double* __restrict__ b,
                                                       double* __restrict__ r,
                                                       double* __restrict__ x,
                                                       float* __restrict__ r32, const Finish F) {
    double acc = 0.0;
    for (long long c = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; c < N;
         c += (long long)gridDim.x * LIN_BLOCK) {
        const double v = b[c];
        r[c] = v;
        x[c] = 0.0;
        if (r32) r32[c] = (float)v;
        acc += v * v;
    }
    finish<false, RED_CG_START>(F, acc, 0.0);
}

// ---------------------------------------------------------------------------------------------
// BiCGStab building blocks (FP64), right preconditioning.  With the FP32 multigrid the vectors
// p and s are also written in FP32, as the cycle's right-hand side, and the cycle's last sweep writes
// its result in FP64, so no conversion passes remain.  (The product does not read an FP32 vector
// itself: a conversion takes an FP64 slot like an FMA, seven of them beside its eight; conversions
// by integer instructions with a branch for subnormals measured slower still, 449 against 321 us.)

// y = A x with the non-symmetric operator; w1.y (and y.y when TWO).  Every load of a row is issued
// before its first use; the sum is one chain of FMAs, 8 FP64 instructions a row with one dot.
// Measured at 256^3: 267 us against 321 us with the products summed apart from the diagonal.
template <bool TWO>
__global__ void __launch_bounds__(LIN_BLOCK) k_matvec_ns(const OpNS A, const double* __restrict__ x,
                                                         double* __restrict__ y,
                                                         const double* __restrict__ w1,
                                                         const Finish F) {
    if (skipped(A.skip)) return;
    double d1 = 0.0, d2 = 0.0;
    const long long sz = (long long)A.nx * A.ny;
    for (long long c = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; c < A.N;
         c += (long long)gridDim.x * LIN_BLOCK) {
        int i, j, k;
        coords_fd(c, A.fd_nx, A.fd_nxy, i, j, k);
        const int q[3] = {i, j, k};
        const int n[3] = {A.nx, A.ny, A.nz};
        const long long s[3] = {1, A.nx, sz};
        double w[6], xv[6];
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            // (the lower entry is 0 on zero-flux boundary faces, where lo is the far side)
            const long long lo = q[ax] > 0 ? c - s[ax] : c + (long long)(n[ax] - 1) * s[ax];
            const bool has = q[ax] < n[ax] - 1 || A.per[ax];
            const long long hi = q[ax] < n[ax] - 1 ? c + s[ax] : (has ? c - (long long)(n[ax] - 1) * s[ax] : c);
            xv[2 * ax] = __ldg(x + lo);
            xv[2 * ax + 1] = has ? __ldg(x + hi) : 0.0;
            w[2 * ax] = __ldg(A.Q[ax] + c);
            w[2 * ax + 1] = has ? __ldg(A.P[ax] + hi) : 0.0;
        }
        double v = __ldg(A.diag + c) * __ldg(x + c);
        const double w1c = __ldg(w1 + c);
#pragma unroll
        for (int f = 0; f < 6; ++f) v = fma(-w[f], xv[f], v);
        y[c] = v;
        d1 = fma(w1c, v, d1);
        if (TWO) d2 = fma(v, v, d2);
    }
    finish<TWO, TWO ? RED_BICG_OMEGA : RED_BICG_ALPHA>(F, d1, d2);
}

// The vector updates below take two elements per thread and turn (16-byte accesses: twice the bytes in
// flight of one; the library's vectors start on 256-byte boundaries) and the odd last one alone:
// f(i, n) works on the n elements from i on.
template <typename F>
__device__ __forceinline__ void for_pairs(long long N, F f) {
    const long long pairs = N / 2;
    for (long long q = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; q < pairs;
         q += (long long)gridDim.x * LIN_BLOCK)
        f(2 * q, std::integral_constant<int, 2>());
    if ((N & 1) && blockIdx.x == 0 && threadIdx.x == 0) f(N - 1, std::integral_constant<int, 1>());
}
template <int n>
__device__ __forceinline__ void ld_pair(const double* p, double (&v)[n]) {
    if constexpr (n == 2) {
        const double2 t = *reinterpret_cast<const double2*>(p);
        v[0] = t.x; v[1] = t.y;
    } else {
        v[0] = *p;
    }
}
template <int n>
__device__ __forceinline__ void st_pair(double* p, const double (&v)[n]) {
    if constexpr (n == 2) *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
    else *p = v[0];
}
template <int n>
__device__ __forceinline__ void st_pair(float* p, const double (&v)[n]) {
    if constexpr (n == 2) *reinterpret_cast<float2*>(p) = make_float2((float)v[0], (float)v[1]);
    else *p = (float)v[0];
}

// r = b, rh = b, x = 0; r.r
__global__ void __launch_bounds__(LIN_BLOCK) k_bicg_init(long long N, const double* __restrict__ b,
                                                         double* __restrict__ r,
                                                         double* __restrict__ rh,
                                                         double* __restrict__ x, const Finish F) {
    double acc = 0.0;
    for_pairs(N, [&](long long i, auto cnt) {
        constexpr int n = decltype(cnt)::value;
        double v[n], z[n] = {};
        ld_pair(b + i, v);
        st_pair(r + i, v);
        st_pair(rh + i, v);
        st_pair(x + i, z);
#pragma unroll
        for (int q = 0; q < n; ++q) acc = fma(v[q], v[q], acc);
    });
    finish<false, RED_BICG_START>(F, acc, 0.0);
}

// p = r + beta (p - omega v); at the loop's first iteration and after a restart p = r, and after a
// restart also the shadow vector rh = r
__global__ void __launch_bounds__(LIN_BLOCK) k_bicg_p(long long N, const double* __restrict__ scal,
                                                      const double* __restrict__ r,
                                                      const double* __restrict__ v,
                                                      double* __restrict__ p,
                                                      double* __restrict__ rh,
                                                      float* __restrict__ p32) {
    const double beta = scal[S_BETA], omega = scal[S_OMEGA];
    const bool restart = scal[S_RST] != 0.0;
    const bool first = scal[S_ITS] == 0.0 || restart;
    for_pairs(N, [&](long long i, auto cnt) {
        constexpr int n = decltype(cnt)::value;
        double rv[n], pv[n], vv[n];
        ld_pair(r + i, rv);
        if (first) {
#pragma unroll
            for (int q = 0; q < n; ++q) pv[q] = rv[q];
        } else {
            ld_pair(p + i, pv);
            ld_pair(v + i, vv);
#pragma unroll
            for (int q = 0; q < n; ++q) pv[q] = fma(beta, fma(-omega, vv[q], pv[q]), rv[q]);
        }
        st_pair(p + i, pv);
        if (p32) st_pair(p32 + i, pv);
        if (restart) st_pair(rh + i, rv);
    });
}

// s = r - alpha v; s.s
__global__ void __launch_bounds__(LIN_BLOCK) k_bicg_s(long long N, const double* __restrict__ scal,
                                                      const double* __restrict__ r,
                                                      const double* __restrict__ v,
                                                      double* __restrict__ s,
                                                      float* __restrict__ s32, const Finish F) {
    const double alpha = scal[S_ALPHA];
    double acc = 0.0;
    for_pairs(N, [&](long long i, auto cnt) {
        constexpr int n = decltype(cnt)::value;
        double rv[n], vv[n];
        ld_pair(r + i, rv);
        ld_pair(v + i, vv);
#pragma unroll
        for (int q = 0; q < n; ++q) {
            rv[q] = fma(-alpha, vv[q], rv[q]);
            acc = fma(rv[q], rv[q], acc);
        }
        st_pair(s + i, rv);
        if (s32) st_pair(s32 + i, rv);
    });
    finish<false, RED_BICG_SS>(F, acc, 0.0);
}

// Converged at the middle of the iteration (S_HALF): x += alpha ph, r untouched.  Otherwise, unless
// a breakdown ended the iteration: x += alpha ph + omega sh, r = s - omega t, r.r and rh.r (zeros when
// skipped)
__global__ void __launch_bounds__(LIN_BLOCK) k_bicg_xr(long long N, const double* __restrict__ scal,
                                                       double* __restrict__ x,
                                                       const double* __restrict__ ph,
                                                       const double* __restrict__ sh,
                                                       const double* __restrict__ s,
                                                       const double* __restrict__ t,
                                                       double* __restrict__ r,
                                                       const double* __restrict__ rh,
                                                       const Finish F) {
    const double alpha = scal[S_ALPHA], omega = scal[S_OMEGA];
    const bool half = scal[S_HALF] != 0.0;
    const bool none = !half && scal[S_DONE] != 0.0;
    double rr = 0.0, rhr = 0.0;
    if (half) {
        for_pairs(N, [&](long long i, auto cnt) {
            constexpr int n = decltype(cnt)::value;
            double xv[n], pv[n];
            ld_pair(x + i, xv);
            ld_pair(ph + i, pv);
#pragma unroll
            for (int q = 0; q < n; ++q) xv[q] = fma(alpha, pv[q], xv[q]);
            st_pair(x + i, xv);
        });
    } else if (!none) {
        for_pairs(N, [&](long long i, auto cnt) {
            constexpr int n = decltype(cnt)::value;
            double xv[n], pv[n], qv[n], sv[n], tv[n], hv[n];
            ld_pair(x + i, xv);
            ld_pair(ph + i, pv);
            ld_pair(sh + i, qv);
            ld_pair(s + i, sv);
            ld_pair(t + i, tv);
            ld_pair(rh + i, hv);
#pragma unroll
            for (int q = 0; q < n; ++q) {
                xv[q] = fma(alpha, pv[q], fma(omega, qv[q], xv[q]));
                sv[q] = fma(-omega, tv[q], sv[q]);
                rr = fma(sv[q], sv[q], rr);
                rhr = fma(hv[q], sv[q], rhr);
            }
            st_pair(x + i, xv);
            st_pair(r + i, sv);
        });
    }
    finish<true, RED_BICG_NEXT>(F, rr, rhr);
}

// ---------------------------------------------------------------------------------------------
// multigrid kernels (templated on the level precision)

// a sweep's result: in the level's precision, or in FP64 where the sweep ends the cycle (out64; the
// caller's vector, one conversion per cell under the sweep's memory time instead of a pass of its own)
template <typename T>
__device__ __forceinline__ void store_sweep(T* xout, double* out64, long long c, T v) {
    if (out64) out64[c] = (double)v;
    else xout[c] = v;
}

// weighted Jacobi with wid = omega / diag: first sweep from x = 0: x_out = wid b; else
// x_out = x_in + omega (b - A x_in) / diag, written as (1 - omega) x_in + wid (b + off).  first: 0: a
// sweep from x_in; 1: the first; 2: the first two in one pass, the first one's x made where it
// is read (the same numbers; no launch and no trip to memory for it)
template <typename T>
__global__ void __launch_bounds__(LIN_BLOCK) k_mg_smooth(const Op<T> A, const T* __restrict__ b,
                                                         const T* __restrict__ xin,
                                                         T* __restrict__ xout, T omega,
                                                         int first, double* __restrict__ out64) {
    if (skipped(A.skip)) return;
    for (long long c = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; c < A.N;
         c += (long long)gridDim.x * LIN_BLOCK) {
        const T wi = A.wid[c];
        if (first == 1) {
            xout[c] = wi * b[c];
            continue;
        }
        int i, j, k;
        coords3(A, c, i, j, k);
        if (first == 2) {
            const FirstSweep<T> x1{A.wid, b};
            xout[c] = jacobi_update(x1[c], b[c], wi, off_row(A, x1, c, i, j, k), omega);
        } else {
            store_sweep(xout, out64, c, jacobi_update(xin[c], b[c], wi, off_row(A, xin, c, i, j, k), omega));
        }
    }
}

// the first sweep of a cycle, from x = 0: x = (omega / diag) b, 16 bytes per thread (N a
// multiple of 16 / sizeof(T), 16-byte aligned arrays; the launcher checks)
template <typename T>
__global__ void __launch_bounds__(LIN_BLOCK) k_mg_smooth_first_vec(long long N,
                                                                   const T* __restrict__ wid,
                                                                   const T* __restrict__ b,
                                                                   T* __restrict__ xout,
                                                                   const double* skip) {
    if (skipped(skip)) return;
    using VT = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    const long long NV = N * (long long)sizeof(T) / 16;
    for (long long q = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; q < NV;
         q += (long long)gridDim.x * LIN_BLOCK) {
        const VT w = __ldg(reinterpret_cast<const VT*>(wid) + q);
        const VT bb = __ldg(reinterpret_cast<const VT*>(b) + q);
        VT o;
        o.x = w.x * bb.x; o.y = w.y * bb.y;
        if constexpr (sizeof(T) == 4) { o.z = w.z * bb.z; o.w = w.w * bb.w; }
        reinterpret_cast<VT*>(xout)[q] = o;
    }
}

// Weighted-Jacobi sweep marching along z: a thread owns one (i, j) column and ZM consecutive
// planes, so the x values of the planes above and below and the z-face coefficient shared by
// two planes stay in registers, and the x / y neighbour offsets are computed once.  The
// arithmetic is that of k_mg_smooth term for term (the same products summed in the same
// order), so the result is identical.  ZM = 2: every load of both planes is issued before the
// first use within 56 registers, four blocks per SM; measured at 256^3 (FP32, both couplings
// per face), 0.91 of the HBM copy bandwidth against 0.61 for ZM = 8 (whose 104 loads do not fit
// the register budget and were issued in dependent groups) and 0.78 for one cell per thread.
constexpr int ZM = 2;
template <typename T, bool TWO>
__global__ void __launch_bounds__(LIN_BLOCK) k_mg_smooth_zm(const Op<T> A, const T* __restrict__ b,
                                                            const T* __restrict__ xin,
                                                            T* __restrict__ xout, T omega,
                                                            double* __restrict__ out64) {
    if (skipped(A.skip)) return;
    const long long nxy = (long long)A.nx * A.ny;
    const long long col = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x;
    if (col >= nxy) return;
    const int k0 = blockIdx.y * ZM;
    const unsigned jj = fdiv((unsigned)col, A.fd_nx);
    const int i = (int)((unsigned)col - jj * A.fd_nx.d), j = (int)jj;
    // x and y neighbour offsets (a zero-flux lower face carries W = 0 and reads the far side)
    const long long dlo0 = i > 0 ? -1 : (long long)(A.nx - 1);
    const bool hhi0 = i < A.nx - 1 || A.per[0];
    const long long dhi0 = i < A.nx - 1 ? 1 : -(long long)(A.nx - 1);
    const long long dlo1 = j > 0 ? -(long long)A.nx : (long long)(A.ny - 1) * A.nx;
    const bool hhi1 = j < A.ny - 1 || A.per[1];
    const long long dhi1 = j < A.ny - 1 ? (long long)A.nx : -(long long)(A.ny - 1) * A.nx;
    const int nz = A.nz;
    // read-only operator arrays through non-aliasing pointers, so that the loads of later
    // planes may be issued before the stores of earlier ones
    const T* __restrict__ W0 = A.W[0];
    const T* __restrict__ W1 = A.W[1];
    const T* __restrict__ W2 = A.W[2];
    const T* __restrict__ P0 = A.Wp[0];
    const T* __restrict__ P1 = A.Wp[1];
    const T* __restrict__ P2 = A.Wp[2];
    const T* __restrict__ wd = A.wid;
    const auto X = [&](long long c) { return TWO ? __ldg(wd + c) * __ldg(b + c) : __ldg(xin + c); };
    // z: plane below k0 (the far side when k0 = 0: W = 0 there unless periodic).  All loads of
    // the ZM planes are issued first (registers), then the planes are computed in order;
    // the launcher uses this kernel only when ZM divides nz.
    const long long c0 = col + (long long)k0 * nxy;
    const long long ctop = k0 + ZM < nz ? c0 + (long long)ZM * nxy : col;   // plane above
    // wz: the lower-face coupling of each plane's row; pz: the coupling of each plane's row to
    // the plane above (Wp of the face above; the same numbers as wz[kk + 1] when symmetric)
    T xz[ZM + 2], wz[ZM], pz[ZM], w0l[ZM], w0h[ZM], w1l[ZM], w1h[ZM], x0l[ZM], x0h[ZM], x1l[ZM],
        x1h[ZM], dd[ZM], bb[ZM];
    xz[0] = X(k0 > 0 ? c0 - nxy : col + (long long)(nz - 1) * nxy);
    xz[ZM + 1] = X(ctop);
#pragma unroll
    for (int kk = 0; kk < ZM; ++kk) {
        const long long c = c0 + (long long)kk * nxy;
        const long long cu = kk + 1 < ZM ? c + nxy : ctop;
        if (!TWO) xz[kk + 1] = __ldg(xin + c);
        wz[kk] = __ldg(W2 + c);
        pz[kk] = __ldg(P2 + cu);
        w0l[kk] = __ldg(W0 + c);
        x0l[kk] = X(c + dlo0);
        w0h[kk] = hhi0 ? __ldg(P0 + c + dhi0) : T(0);
        x0h[kk] = hhi0 ? X(c + dhi0) : T(0);
        w1l[kk] = __ldg(W1 + c);
        x1l[kk] = X(c + dlo1);
        w1h[kk] = hhi1 ? __ldg(P1 + c + dhi1) : T(0);
        x1h[kk] = hhi1 ? X(c + dhi1) : T(0);
        dd[kk] = __ldg(wd + c);
        bb[kk] = __ldg(b + c);
        if (TWO) xz[kk + 1] = dd[kk] * bb[kk];
    }
#pragma unroll
    for (int kk = 0; kk < ZM; ++kk) {
        const bool hz = k0 + kk < nz - 1 || A.per[2];
        T off = T(0);
        off += w0l[kk] * x0l[kk];
        if (hhi0) off += w0h[kk] * x0h[kk];
        off += w1l[kk] * x1l[kk];
        if (hhi1) off += w1h[kk] * x1h[kk];
        off += wz[kk] * xz[kk];
        if (hz) off += pz[kk] * xz[kk + 2];
        store_sweep(xout, out64, c0 + (long long)kk * nxy, jacobi_update(xz[kk + 1], bb[kk], dd[kk], off, omega));
    }
}

// The same FP32 sweep with its rows staged in shared memory by bulk asynchronous copies.  A
// CTA owns one grid row (j) of every plane of a z-slab of ZB planes, one thread per x cell.
// For each plane it needs 12 contiguous rows of nx floats: x at (j, k), (j-1, k), (j+1, k),
// (j, k+1); b, omega / diag and the lower-face couplings W0, W1, W2 and P0 at (j, k); P1 at
// (j+1, k); P2 at (j, k+1).  For the first two sweeps in one (TWO) it is 14: b and omega / diag take
// the place of x.  One elected thread issues them as cp.async.bulk copies into a
// ring of BS stages, each completing on its stage's mbarrier; the CTA computes plane k from
// shared memory while the copies of the next planes are in flight.  Rows whose neighbour
// does not exist (zero-flux faces) are fetched from a valid row and not used, as in
// k_mg_smooth_zm, whose products and sums this kernel repeats term for term.  Requirements
// (checked by the launcher): nx a multiple of 4 and at most BULK_MAX_NX, 16-byte aligned
// arrays, nz a multiple of ZB.  Each wait on a stage is bounded: after BULK_SPIN tries the
// kernel records the plane in *err, waits (bounded) for its own copies once more, and
// returns.
constexpr int BULK_ROWS = 12, BULK_ROWS_TWO = 14;
constexpr int BULK_STAGES = 3;
constexpr int BULK_ZB = 16;
constexpr int BULK_MAX_NX = 512;
constexpr long long BULK_SPIN = 1LL << 24;

// set to 1 by a staged sweep whose wait on a stage timed out
__device__ int g_bulk_wait_error = 0;
static int* g_bulk_err_ptr = nullptr;

__device__ __forceinline__ unsigned smem_u32(const void* p) {
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes,
                                         unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}" 
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait for the phase `parity` of a stage barrier; false on timeout
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity) {
    for (long long t = 0; t < BULK_SPIN; ++t)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

template <bool TWO>
__global__ void __launch_bounds__(BULK_MAX_NX) k_mg_smooth_bulk(const Op<float> A,
                                                                const float* __restrict__ b,
                                                                const float* __restrict__ xin,
                                                                float* __restrict__ xout,
                                                                float omega, int* err,
                                                                double* __restrict__ out64) {
    if (skipped(A.skip)) return;
    constexpr int ROWS = TWO ? BULK_ROWS_TWO : BULK_ROWS;
    extern __shared__ __align__(128) float rows[];          // [BULK_STAGES][ROWS][nx]
    __shared__ __align__(8) unsigned long long bar[BULK_STAGES];
    const int nx = A.nx, ny = A.ny, nz = A.nz;
    const int i = threadIdx.x;
    const int j = blockIdx.x;
    const int k0 = blockIdx.y * BULK_ZB;
    const long long nxy = (long long)nx * ny;
    const int jm = j > 0 ? j - 1 : ny - 1;
    const int jp = j < ny - 1 ? j + 1 : 0;
    const bool hhi0 = i < nx - 1 || A.per[0];
    const bool hhi1 = j < ny - 1 || A.per[1];
    const unsigned row_bytes = (unsigned)nx * 4u;
    auto stage_row = [&](int st, int r) { return rows + ((long long)st * ROWS + r) * nx; };
    // the copies of plane k into stage st (one elected thread)
    auto issue = [&](int k, int st) {
        const int ku = k + 1 < nz ? k + 1 : 0;
        const long long c = (long long)j * nx + (long long)k * nxy;
        const long long cm = (long long)jm * nx + (long long)k * nxy;
        const long long cp = (long long)jp * nx + (long long)k * nxy;
        const long long cu = (long long)j * nx + (long long)ku * nxy;
        const float* const x = TWO ? b : xin;
        const float* src[ROWS] = {x + c, x + cm, x + cp, x + cu, A.W[0] + c, A.W[1] + c, A.W[2] + c,
                                  A.Wp[0] + c, A.Wp[1] + cp, A.Wp[2] + cu, A.wid + c};
        if constexpr (TWO) {
            src[11] = A.wid + cm;
            src[12] = A.wid + cp;
            src[13] = A.wid + cu;
        } else {
            src[11] = b + c;
        }
        mbar_expect_tx(&bar[st], row_bytes * ROWS);
#pragma unroll
        for (int r = 0; r < ROWS; ++r) bulk_g2s(stage_row(st, r), src[r], row_bytes, &bar[st]);
    };
    if (i == 0) {
#pragma unroll
        for (int st = 0; st < BULK_STAGES; ++st) mbar_init(&bar[st], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (i == 0) {
#pragma unroll
        for (int st = 0; st < BULK_STAGES; ++st)
            if (st < BULK_ZB) issue(k0 + st, st);
    }
    // x of the plane below the first one (the far side when k0 = 0: W = 0 there unless periodic)
    float xlo = 0.f;
    if (i < nx) {
        const long long c = (long long)j * nx + (long long)(k0 > 0 ? k0 - 1 : nz - 1) * nxy + i;
        xlo = TWO ? __ldg(A.wid + c) * __ldg(b + c) : __ldg(xin + c);
    }
    bool ok = true;
    for (int kk = 0; kk < BULK_ZB; ++kk) {
        const int st = kk % BULK_STAGES;
        const unsigned parity = (unsigned)((kk / BULK_STAGES) & 1);
        if (!mbar_wait(&bar[st], parity)) { ok = false; break; }
        const int k = k0 + kk;
        float xcen = 0.f;
        if (i < nx) {
            const float* XC = stage_row(st, 0);                 // (TWO: b, to be multiplied by wid)
            const float* XM = stage_row(st, 1);
            const float* XP = stage_row(st, 2);
            const float* XU = stage_row(st, 3);
            const float* R0 = stage_row(st, 4);
            const float* R1 = stage_row(st, 5);
            const float* R2 = stage_row(st, 6);
            const float* Q0 = stage_row(st, 7);
            const float* Q1 = stage_row(st, 8);
            const float* Q2 = stage_row(st, 9);
            const float* WD = stage_row(st, 10);
            const float* BB = TWO ? XC : stage_row(st, 11);
            const auto x = [&](const float* row, int w, int at) {   // w: its row of wid
                return TWO ? stage_row(st, w)[at] * row[at] : row[at];
            };
            const int il = i > 0 ? i - 1 : nx - 1;
            const int ih = i < nx - 1 ? i + 1 : 0;
            const bool hz = k < nz - 1 || A.per[2];
            xcen = x(XC, 10, i);
            float off = 0.f;
            off += R0[i] * x(XC, 10, il);
            if (hhi0) off += Q0[ih] * x(XC, 10, ih);
            off += R1[i] * x(XM, 11, i);
            if (hhi1) off += Q1[i] * x(XP, 12, i);
            off += R2[i] * xlo;
            if (hz) off += Q2[i] * x(XU, 13, i);
            store_sweep(xout, out64, (long long)j * nx + (long long)k * nxy + i,
                        jacobi_update(xcen, BB[i], WD[i], off, omega));
        }
        xlo = xcen;
        __syncthreads();                                    // stage st is free again
        if (i == 0 && kk + BULK_STAGES < BULK_ZB) issue(k0 + kk + BULK_STAGES, st);
    }
    if (!ok) {
        if (i == 0) atomicExch(err, 1);
        // the copies this CTA issued may still land: wait for them once more, bounded
        for (int st = 0; st < BULK_STAGES; ++st) mbar_wait(&bar[st], 0u);
    }
}

cudaError_t linear_kernels_init() {
    if (g_bulk_err_ptr) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_mg_smooth_bulk<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         BULK_STAGES * BULK_ROWS * BULK_MAX_NX * (int)sizeof(float));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_mg_smooth_bulk<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 BULK_STAGES * BULK_ROWS_TWO * BULK_MAX_NX * (int)sizeof(float));
    void* p = nullptr;
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&p, g_bulk_wait_error);
    if (e == cudaSuccess) g_bulk_err_ptr = static_cast<int*>(p);
    return e;
}
cudaError_t bulk_wait_flag_read(int* host, cudaStream_t st) {
    return cudaMemcpyFromSymbolAsync(host, g_bulk_wait_error, sizeof(int), 0, cudaMemcpyDeviceToHost, st);
}
cudaError_t bulk_wait_flag_clear(cudaStream_t st) {
    static const int zero = 0;
    return cudaMemcpyToSymbolAsync(g_bulk_wait_error, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, st);
}

// coarse right-hand side: (sum over the children of the fine residual b - A x) / 8, the
// transpose of the injection prolongation scaled by 1/8 (a parent with fewer than 8 children,
// at an odd extent, keeps the factor, so that the cycle stays symmetric).
//
// FP64 and symmetric: with (A x)_c = loc_c x_c + sum_faces W (x_c - x_nb), the faces
// between two children of the parent cancel in the sum, so only the faces to cells outside the
// parent are evaluated; this halves the FP64 arithmetic that bounds the FP64 instance.  (For a
// non-symmetric operator the two rows of an inner face carry W and Wp, which do not cancel.)
// Otherwise the residual of each child from its full row, which for FP32 also measured faster
// at 256^3 (16.2 against 18.8 ms per step, where the outside-face form took FP64 from 48.0 down
// to 41.9 ms).
template <typename T>
__global__ void __launch_bounds__(LIN_BLOCK) k_mg_restrict(const Op<T> A, const T* __restrict__ b,
                                                           const T* __restrict__ x, int cnx,
                                                           int cny, int cnz, FastDiv fcx,
                                                           FastDiv fcxy, T* __restrict__ bc) {
    if (skipped(A.skip)) return;
    const long long Nc = (long long)cnx * cny * cnz;
    const long long sz = (long long)A.nx * A.ny;
    const int n[3] = {A.nx, A.ny, A.nz};
    const long long s[3] = {1, A.nx, sz};
    for (long long cc = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; cc < Nc;
         cc += (long long)gridDim.x * LIN_BLOCK) {
        int I, J, K;
        coords_fd(cc, fcx, fcxy, I, J, K);
        T acc = T(0);
        const bool inner_cancel = sizeof(T) == 8 && A.loc && A.Wp[0] == A.W[0];
        if (inner_cancel) {
#pragma unroll
            for (int dk = 0; dk < 2; ++dk) {
#pragma unroll
                for (int dj = 0; dj < 2; ++dj) {
#pragma unroll
                    for (int di = 0; di < 2; ++di) {
                        const int q[3] = {2 * I + di, 2 * J + dj, 2 * K + dk};
                        if (q[0] >= n[0] || q[1] >= n[1] || q[2] >= n[2]) continue;  // odd end
                        const int d[3] = {di, dj, dk};
                        const long long c = q[0] + (long long)A.nx * (q[1] + (long long)A.ny * q[2]);
                        const T xc = x[c];
                        T fl = T(0);
#pragma unroll
                        for (int ax = 0; ax < 3; ++ax) {
                            if (d[ax] == 0) {         // lower face: the neighbour is outside
                                const long long lo = q[ax] > 0 ? c - s[ax]
                                                               : c + (long long)(n[ax] - 1) * s[ax];
                                fl += A.W[ax][c] * (xc - x[lo]);   // W = 0 on zero-flux faces
                            }
                            // upper face: outside unless it leads to the sibling d = 1
                            if (d[ax] == 1 || q[ax] + 1 >= n[ax]) {
                                long long hi = -1;
                                if (q[ax] < n[ax] - 1) hi = c + s[ax];
                                else if (A.per[ax]) hi = c - (long long)(n[ax] - 1) * s[ax];
                                if (hi >= 0) fl += A.W[ax][hi] * (xc - x[hi]);
                            }
                        }
                        acc += b[c] - A.loc[c] * xc - fl;
                    }
                }
            }
        } else {
            for (int dk = 0; dk < 2; ++dk) {
                const int k = 2 * K + dk;
                if (k >= A.nz) continue;
                for (int dj = 0; dj < 2; ++dj) {
                    const int j = 2 * J + dj;
                    if (j >= A.ny) continue;
                    for (int di = 0; di < 2; ++di) {
                        const int i = 2 * I + di;
                        if (i >= A.nx) continue;
                        const long long c = i + (long long)A.nx * (j + (long long)A.ny * k);
                        acc += b[c] - apply_row(A, x, c, i, j, k, x[c]);
                    }
                }
            }
        }
        bc[cc] = acc * T(0.125);
    }
}

// The same with eight lanes to a parent, one for each child (a warp: four parents in a row, so runs of
// eight cells along x), summed by shuffles: a child's loads do not wait for those of its siblings,
// and eight times as many threads ask for them.  On large levels the first form, with fewer
// instructions per cell, is the better one.  Measured, this form / the first, us:
//   FP32                  64^3 8.4 / 10.0   88^3 11.6 / 12.1   96^3 13.5 / 12.8   128^3 24.0 / 20.5
//   FP64, non-symmetric   64^3 12.8 / 14.0   88^3 23.2 / 24.0   96^3 29.0 / 24.7   128^3 60.0 / 49.5
//   FP64, symmetric       48^3 10.0 / 14.3   56^3 12.7 / 14.5   64^3 15.5 / 13.9   80^3 24.6 / 18.1
// (in the last one the first form leaves out the faces between children, half the arithmetic that
// bounds it).  RESTRICT_SPLIT and, for that one, RESTRICT_SPLIT_SYM: most parents of a level that
// takes this form, 80^3 and 58^3 cells, a size below the crossing.
constexpr long long RESTRICT_SPLIT = 1LL << 16, RESTRICT_SPLIT_SYM = 3LL << 13;
template <typename T>
__global__ void __launch_bounds__(LIN_BLOCK) k_mg_restrict_split(const Op<T> A, const T* __restrict__ b,
                                                                 const T* __restrict__ x, int cnx,
                                                                 int cny, int cnz, FastDiv fcx,
                                                                 FastDiv fcxy, T* __restrict__ bc) {
    if (skipped(A.skip)) return;
    const long long Nc = (long long)cnx * cny * cnz;
    const int n[3] = {A.nx, A.ny, A.nz};
    const long long s[3] = {1, A.nx, (long long)A.nx * A.ny};
    const int lane = (int)(threadIdx.x & 31u);
    const int d[3] = {lane & 1, lane >> 3 & 1, lane >> 4};
    const bool inner_cancel = sizeof(T) == 8 && A.loc && A.Wp[0] == A.W[0];
    const long long warps = (long long)gridDim.x * (LIN_BLOCK / 32);
    for (long long w = blockIdx.x * (long long)(LIN_BLOCK / 32) + threadIdx.x / 32; w * 4 < Nc; w += warps) {
        const long long cc = w * 4 + (lane >> 1 & 3);
        T acc = T(0);
        if (cc < Nc) {
            int I, J, K;
            coords_fd(cc, fcx, fcxy, I, J, K);
            const int q[3] = {2 * I + d[0], 2 * J + d[1], 2 * K + d[2]};
            if (q[0] < n[0] && q[1] < n[1] && q[2] < n[2]) {
                const long long c = q[0] + (long long)A.nx * (q[1] + (long long)A.ny * q[2]);
                const T xc = x[c];
                if (inner_cancel) {
                    T fl = T(0);
#pragma unroll
                    for (int ax = 0; ax < 3; ++ax) {
                        // the face to the outside: lower for a first child, upper for a second
                        const long long wrap = (long long)(n[ax] - 1) * s[ax];
                        const bool up = d[ax] == 1, end = q[ax] == n[ax] - 1;
                        const long long nb = up ? (end ? c - wrap : c + s[ax]) : (q[ax] > 0 ? c - s[ax] : c + wrap);
                        const T wf = up && end && !A.per[ax] ? T(0) : A.W[ax][up ? nb : c];
                        fl += wf * (xc - x[nb]);
                        // an only child has both
                        if (!up && end && A.per[ax]) fl += A.W[ax][c - wrap] * (xc - x[c - wrap]);
                    }
                    acc = b[c] - A.loc[c] * xc - fl;
                } else {
                    acc = b[c] - apply_row(A, x, c, q[0], q[1], q[2], xc);
                }
            }
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 8);
        acc += __shfl_xor_sync(0xffffffffu, acc, 16);
        if ((lane & 25) == 0 && cc < Nc) bc[cc] = acc * T(0.125);
    }
}

// x_f += x_c(parent), 16 bytes of fine cells per thread along x (4 FP32 or 2 FP64 cells, whose
// parents are 2 or 1 consecutive coarse cells); needs nx a multiple of 4 (FP32) or 2 (FP64) and
// 16-byte aligned rows, which the launcher checks.  fx, fxy divide by nx / V and nx ny / V.
template <typename T>
__global__ void __launch_bounds__(LIN_BLOCK) k_mg_prolong_vec(int nx, int ny, int nz, int cnx,
                                                              int cny, FastDiv fx, FastDiv fxy,
                                                              const T* __restrict__ xc,
                                                              T* __restrict__ xf,
                                                              const double* skip) {
    if (skipped(skip)) return;
    constexpr int V = 16 / (int)sizeof(T);
    using VT = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
    const long long NV = (long long)nx * ny * nz / V;
    for (long long q = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; q < NV;
         q += (long long)gridDim.x * LIN_BLOCK) {
        int iv, j, k;
        coords_fd(q, fx, fxy, iv, j, k);
        const T* pc = xc + (long long)(V / 2) * iv + (long long)cnx * ((j >> 1) + (long long)cny * (k >> 1));
        VT v = reinterpret_cast<VT*>(xf)[q];
        if constexpr (sizeof(T) == 4) {
            const float2 pp = *reinterpret_cast<const float2*>(pc);
            v.x += pp.x; v.y += pp.x; v.z += pp.y; v.w += pp.y;
        } else {
            const double pp = *pc;
            v.x += pp; v.y += pp;
        }
        reinterpret_cast<VT*>(xf)[q] = v;
    }
}

// x_f += x_c(parent)
template <typename T>
__global__ void __launch_bounds__(LIN_BLOCK) k_mg_prolong(int nx, int ny, int nz, int cnx, int cny,
                                                          FastDiv fx, FastDiv fxy,
                                                          const T* __restrict__ xc,
                                                          T* __restrict__ xf,
                                                          const double* skip) {
    if (skipped(skip)) return;
    const long long N = (long long)nx * ny * nz;
    for (long long c = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; c < N;
         c += (long long)gridDim.x * LIN_BLOCK) {
        int i, j, k;
        coords_fd(c, fx, fxy, i, j, k);
        xf[c] += xc[(i >> 1) + (long long)cnx * ((j >> 1) + (long long)cny * (k >> 1))];
    }
}

// One coarse cell of the hierarchy: the operator by re-discretisation, and the smoother's omega /
// diagonal.  Local diagonal = mean of the children's local diagonals (diag - the six couplings of their
// rows); each face array of the coarse cell's lower face = (mean of that array over the existing fine
// lower faces of its first-layer children) / 4, W from W and, for a non-symmetric operator, Wp from Wp;
// diagonal = local diagonal + the row's six couplings, of which the upper ones are the Wp of the faces
// above, formed here from the same fine entries as the cells above form them.  (Counts of children are
// powers of two, so the means are exact products.)
//
// Sums of couplings are shared between the faces and the local diagonal: 8.5 loads and about 8 FP64
// additions per fine cell.  Measured for all five coarse levels of a 256^3 FP32 hierarchy, both
// couplings per face: 0.63 ms in 5 launches, against 1.04 ms in 15 for separate passes (operator, diagonal,
// omega / diagonal) with a 64-bit division and dependent loads per child.
template <typename TF, typename TC>
__device__ __forceinline__ void build_cell(const Op<TF>& A, const MgLevel<TC>& c, int I, int J, int K,
                                           long long cc, double omega) {
    const long long s[3] = {1, A.nx, (long long)A.nx * A.ny};
    const int n[3] = {A.nx, A.ny, A.nz}, q0[3] = {2 * I, 2 * J, 2 * K};
    const long long c0 = q0[0] + s[1] * q0[1] + s[2] * q0[2];
    // per axis: a second child, and the fine face above the parent (its offset from the last layer)
    bool two[3], up[3];
    long long above[3];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        two[ax] = q0[ax] + 1 < n[ax];
        const int last = q0[ax] + (two[ax] ? 1 : 0);
        up[ax] = last < n[ax] - 1 || A.per[ax];
        above[ax] = last < n[ax] - 1 ? s[ax] : -(long long)(n[ax] - 1) * s[ax];
    }
    double dl = 0.0, tot = 0.0, wl[3] = {0.0, 0.0, 0.0}, wp[3] = {0.0, 0.0, 0.0}, wu[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int dk = 0; dk < 2; ++dk)
#pragma unroll
        for (int dj = 0; dj < 2; ++dj)
#pragma unroll
            for (int di = 0; di < 2; ++di) {
                const int d[3] = {di, dj, dk};
                if ((di && !two[0]) || (dj && !two[1]) || (dk && !two[2])) continue;
                const long long f = c0 + di + dj * s[1] + dk * s[2];
                dl += widen(A.diag[f]);
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) {
                    const double w = widen(A.W[ax][f]), v = widen(A.Wp[ax][f]);
                    if (d[ax] == 0) { wl[ax] += w; wp[ax] += v; }      // the parent's lower face
                    else tot += w + v;                                 // a face between children
                    if ((d[ax] == 1 || !two[ax]) && up[ax])            // the parent's upper face
                        wu[ax] += widen(A.Wp[ax][f + above[ax]]);
                }
            }
    double diag = 0.0;
    const double half[3] = {two[0] ? 0.5 : 1.0, two[1] ? 0.5 : 1.0, two[2] ? 0.5 : 1.0};
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        tot += wl[ax] + wu[ax];
        const double mean = 0.25 * half[(ax + 1) % 3] * half[(ax + 2) % 3];
        const double wlc = mean * wl[ax];
        diag += wlc + mean * wu[ax];
        c.w[ax][cc] = (TC)wlc;
        if (c.wp[0]) c.wp[ax][cc] = (TC)(mean * wp[ax]);
    }
    const double local = (dl - tot) * (half[0] * half[1] * half[2]);
    diag += local;
    c.diag[cc] = (TC)diag;
    if (c.loc) c.loc[cc] = (TC)local;
    c.wid[cc] = (TC)omega / (TC)diag;
}

template <typename TF, typename TC>
__global__ void __launch_bounds__(LIN_BLOCK) k_mg_build(const Op<TF> A, const MgLevel<TC> c, FastDiv fcx,
                                                        FastDiv fcxy, double omega) {
    const long long cc = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (cc >= c.N) return;
    int I, J, K;
    coords_fd(cc, fcx, fcxy, I, J, K);
    build_cell<TF, TC>(A, c, I, J, K, cc, omega);
}

// Small levels, each from the one before, by one cluster with its barrier between them.  The levels are
// read and written in global memory (plain loads: the barrier orders them).
template <typename TC>
struct BuildArgs {
    MgLevel<TC> c[MG_TAIL_LEVELS];
    int n;
    double omega;
};
template <typename TF, typename TC>
__global__ void __launch_bounds__(LIN_BLOCK) k_mg_build_tail(const __grid_constant__ Op<TF> A,
                                                             const __grid_constant__ BuildArgs<TC> B) {
    const int me = (int)(blockIdx.x * LIN_BLOCK + threadIdx.x), all = (int)(gridDim.x * LIN_BLOCK);
    for (int l = 0; l < B.n; ++l) {
        const MgLevel<TC> c = B.c[l];
        const int nxy = c.nx * c.ny;
        for (int cc = me; cc < (int)c.N; cc += all) {
            const int K = cc / nxy, J = (cc - K * nxy) / c.nx, I = cc - K * nxy - J * c.nx;
            if (l == 0) {
                build_cell<TF, TC>(A, c, I, J, K, cc, B.omega);
            } else {
                const MgLevel<TC>& f = B.c[l - 1];
                Op<TC> o{};
                o.nx = f.nx; o.ny = f.ny; o.nz = f.nz;
                o.diag = f.diag;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    o.per[a] = A.per[a];
                    o.W[a] = f.w[a];
                    o.Wp[a] = f.wp[0] ? f.wp[a] : f.w[a];
                }
                build_cell<TC, TC>(o, c, I, J, K, cc, B.omega);
            }
        }
        if (l + 1 < B.n) cooperative_groups::this_cluster().sync();
    }
}

// FP32 copy of a symmetric finest operator
__global__ void __launch_bounds__(LIN_BLOCK) k_cast_op(const Op<double> A, float* __restrict__ d,
                                                       float* __restrict__ wx,
                                                       float* __restrict__ wy,
                                                       float* __restrict__ wz) {
    for (long long c = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; c < A.N;
         c += (long long)gridDim.x * LIN_BLOCK) {
        d[c] = (float)A.diag[c];
        wx[c] = (float)A.W[0][c];
        wy[c] = (float)A.W[1][c];
        wz[c] = (float)A.W[2][c];
    }
}

// wid = omega / diag and, where loc is given, loc = diag - (sum of the six couplings of
// the row), in TF
template <typename TF, typename TO>
__global__ void __launch_bounds__(LIN_BLOCK) k_mg_level_prep(const Op<TF> A, double omega,
                                                             TO* __restrict__ wid,
                                                             TO* __restrict__ loc) {
    const long long sz = (long long)A.nx * A.ny;
    for (long long c = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; c < A.N;
         c += (long long)gridDim.x * LIN_BLOCK) {
        const TF d = A.diag[c];
        wid[c] = (TO)((TF)omega / d);
        if (loc) {
            int i, j, k;
            coords3(A, c, i, j, k);
            const int q[3] = {i, j, k};
            const int n[3] = {A.nx, A.ny, A.nz};
            const long long s[3] = {1, A.nx, sz};
            TF f = TF(0);
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) {
                f += A.W[ax][c];
                if (q[ax] < n[ax] - 1) f += A.Wp[ax][c + s[ax]];
                else if (A.per[ax]) f += A.Wp[ax][c - (long long)(n[ax] - 1) * s[ax]];
            }
            loc[c] = (TO)(d - f);
        }
    }
}

template <bool VEC>
__global__ void __launch_bounds__(LIN_BLOCK) k_to_f32(long long N, const double* __restrict__ a,
                                                      float* __restrict__ b, const double* skip) {
    if (skipped(skip)) return;
    long long done = 0;
    if (VEC) {
        const long long N4 = N / 4;
        for (long long q = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; q < N4;
             q += (long long)gridDim.x * LIN_BLOCK) {
            const double2 u = reinterpret_cast<const double2*>(a)[2 * q];
            const double2 v = reinterpret_cast<const double2*>(a)[2 * q + 1];
            reinterpret_cast<float4*>(b)[q] = make_float4((float)u.x, (float)u.y, (float)v.x, (float)v.y);
        }
        done = 4 * N4;
    }
    for (long long c = done + blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; c < N;
         c += (long long)gridDim.x * LIN_BLOCK)
        b[c] = (float)a[c];
}

// z = x widened to FP64 (a cycle without post-sweeps, whose last sweep would have done it)
__global__ void __launch_bounds__(LIN_BLOCK) k_from_f32(long long N, const float* __restrict__ x,
                                                        double* __restrict__ z,
                                                        const double* skip) {
    if (skipped(skip)) return;
    for (long long c = blockIdx.x * (long long)LIN_BLOCK + threadIdx.x; c < N;
         c += (long long)gridDim.x * LIN_BLOCK)
        z[c] = (double)x[c];
}

// ---------------------------------------------------------------------------------------------
// host-side launchers

LinLaunch::LinLaunch(cudaStream_t s, LaunchHook* h) : st(s), hook(h) {}

void LinLaunch::begin(const char* name) { if (hook) hook->begin(name); }
cudaError_t LinLaunch::end() {
    cudaError_t e = cudaGetLastError();
    if (hook) hook->end();
    return e;
}

cudaError_t LinLaunch::matvec_dot(const Op<double>& A, const double* p, double* q, const Finish& F) {
    begin("cg_matvec_dot");
    k_matvec_dot<<<sum_blocks(A.N), LIN_BLOCK, 0, st>>>(A, p, q, F);
    return end();
}
cudaError_t LinLaunch::cg_xr(long long N, const double* scal, double* x, double* r,
                             const double* p, const double* q, float* r32, const Finish& F) {
    begin("cg_update_xr");
    k_cg_xr<<<sum_blocks(N), LIN_BLOCK, 0, st>>>(N, scal, x, r, p, q, r32, F);
    return end();
}
cudaError_t LinLaunch::cg_p(long long N, const double* scal, const double* z, double* p) {
    begin("cg_update_p");
    k_cg_p<<<stream_blocks(N), LIN_BLOCK, 0, st>>>(N, scal, z, p);
    return end();
}
cudaError_t LinLaunch::jacobi_dot(long long N, const double* r, const double* diag, double* z,
                                  const Finish& F) {
    begin("precond_jacobi");
    k_jacobi_dot<<<sum_blocks(N), LIN_BLOCK, 0, st>>>(N, r, diag, z, F, skip);
    return end();
}
cudaError_t LinLaunch::cg_beta(long long N, const double* r, const double* z, const Finish& F) {
    begin("dot");
    k_cg_beta<<<sum_blocks(N), LIN_BLOCK, 0, st>>>(N, r, z, F);
    return end();
}
cudaError_t LinLaunch::cg_init(long long N, const double* b, double* r, double* x, float* r32,
                               const Finish& F) {
    begin("cg_init");
    k_cg_init<<<sum_blocks(N), LIN_BLOCK, 0, st>>>(N, b, r, x, r32, F);
    return end();
}
cudaError_t LinLaunch::reduce(const double* part, int n, double* scal, int op, int slot) {
    begin("reduce");
    k_reduce<<<1, RED_BLOCK, 0, st>>>(part, n, scal, op, slot);
    return end();
}

cudaError_t LinLaunch::matvec_ns(const OpNS& A, const double* x, double* y, const double* w1,
                                 int two_dots, const Finish& F) {
    begin("bicg_matvec");
    OpNS B = A;
    B.skip = skip;
    const int nb = sum_blocks(A.N);
    if (two_dots) k_matvec_ns<true><<<nb, LIN_BLOCK, 0, st>>>(B, x, y, w1, F);
    else k_matvec_ns<false><<<nb, LIN_BLOCK, 0, st>>>(B, x, y, w1, F);
    return end();
}
cudaError_t LinLaunch::bicg_init(long long N, const double* b, double* r, double* rh, double* x,
                                 const Finish& F) {
    begin("bicg_init");
    k_bicg_init<<<sum_blocks(N), LIN_BLOCK, 0, st>>>(N, b, r, rh, x, F);
    return end();
}
cudaError_t LinLaunch::bicg_p(long long N, const double* scal, const double* r, const double* v,
                              double* p, double* rh, float* p32) {
    begin(p32 ? "bicg_update_p_f32" : "bicg_update_p");
    k_bicg_p<<<stream_blocks(N), LIN_BLOCK, 0, st>>>(N, scal, r, v, p, rh, p32);
    return end();
}
cudaError_t LinLaunch::bicg_s(long long N, const double* scal, const double* r, const double* v,
                              double* s, float* s32, const Finish& F) {
    begin(s32 ? "bicg_update_s_f32" : "bicg_update_s");
    k_bicg_s<<<sum_blocks(N), LIN_BLOCK, 0, st>>>(N, scal, r, v, s, s32, F);
    return end();
}
cudaError_t LinLaunch::bicg_xr(long long N, const double* scal, double* x, const double* ph,
                               const double* sh, const double* s, const double* t, double* r,
                               const double* rh, const Finish& F) {
    begin("bicg_update_xr");
    k_bicg_xr<<<sum_blocks(N), LIN_BLOCK, 0, st>>>(N, scal, x, ph, sh, s, t, r, rh, F);
    return end();
}
cudaError_t LinLaunch::from_f32(long long N, const float* x, double* z) {
    begin("mg_from_f32");
    k_from_f32<<<stream_blocks(N), LIN_BLOCK, 0, st>>>(N, x, z, skip);
    return end();
}

template <typename T>
cudaError_t LinLaunch::smooth(const Op<T>& A, const T* b, const T* xin, T* xout, T omega,
                              int first, double* out64) {
    // the finest level's sweeps get their own names (the first sweep of a cycle, from x = 0,
    // reads only b and omega / diag)
    if (A.N == fine_N && first == 2) begin(sizeof(T) == 4 ? "mg_smooth_f32_fine_two" : "mg_smooth_f64_fine_two");
    else if (A.N == fine_N && first) begin(sizeof(T) == 4 ? "mg_smooth_f32_fine_first" : "mg_smooth_f64_fine_first");
    else if (A.N == fine_N) begin(sizeof(T) == 4 ? "mg_smooth_f32_fine" : "mg_smooth_f64_fine");
    else begin(sizeof(T) == 4 ? "mg_smooth_f32" : "mg_smooth_f64");
    const long long nxy = (long long)A.nx * A.ny;
    Op<T> B = A;
    B.skip = skip;
    // (FP32 only: the FP64 sweep is bound by its FP64 arithmetic, not by load latency, and
    // its z-marching form measured slower)
    const auto al16 = [](const void* p) { return ((unsigned long long)p & 15ull) == 0; };
    // the staged sweep on large rows (measured 0.966 of HBM against 0.909 for the z-march at
    // 256^3, even at 192^3, and slower on rows of 128 whose level fits in L2)
    bool bulk_ok = false;
    if constexpr (sizeof(T) == 4) {
        bulk_ok = first != 1 && xin != xout && g_bulk_err_ptr && A.nx % 4 == 0 && A.nx >= 256 &&
                  A.nx <= BULK_MAX_NX && A.nz % BULK_ZB == 0 && (first || al16(xin)) && al16(b) &&
                  al16(A.wid) && al16(A.W[0]) && al16(A.W[1]) && al16(A.W[2]) &&
                  al16(A.Wp[0]) && al16(A.Wp[1]) && al16(A.Wp[2]);
    }
    const bool zm_ok = sizeof(T) == 4 && first != 1 && A.nz % ZM == 0 && nxy >= 4 * LIN_BLOCK && xin != xout;
    if (first == 1 && (A.N * (long long)sizeof(T)) % 16 == 0 && al16(A.wid) && al16(b) && al16(xout)) {
        k_mg_smooth_first_vec<T><<<stream_blocks(A.N * (long long)sizeof(T) / 16), LIN_BLOCK, 0, st>>>(
            A.N, A.wid, b, xout, skip);
    } else if (bulk_ok) {
        if constexpr (sizeof(T) == 4) {
            const size_t smem = (size_t)BULK_STAGES * (first ? BULK_ROWS_TWO : BULK_ROWS) * A.nx * sizeof(float);
            const dim3 g((unsigned)A.ny, (unsigned)(A.nz / BULK_ZB));
            const unsigned nt = (unsigned)((A.nx + 31) / 32 * 32);
            if (first) k_mg_smooth_bulk<true><<<g, nt, smem, st>>>(B, b, xin, xout, omega, g_bulk_err_ptr, out64);
            else k_mg_smooth_bulk<false><<<g, nt, smem, st>>>(B, b, xin, xout, omega, g_bulk_err_ptr, out64);
        }
    } else if (zm_ok) {
        if constexpr (sizeof(T) == 4) {
            const dim3 g((unsigned)((nxy + LIN_BLOCK - 1) / LIN_BLOCK), (unsigned)(A.nz / ZM));
            if (first) k_mg_smooth_zm<T, true><<<g, LIN_BLOCK, 0, st>>>(B, b, xin, xout, omega, out64);
            else k_mg_smooth_zm<T, false><<<g, LIN_BLOCK, 0, st>>>(B, b, xin, xout, omega, out64);
        }
    } else {
        k_mg_smooth<T><<<stream_blocks(A.N), LIN_BLOCK, 0, st>>>(B, b, xin, xout, omega, first, out64);
    }
    return end();
}
template <typename T>
cudaError_t LinLaunch::restrict_res(const Op<T>& A, const T* b, const T* x, int cnx, int cny,
                                    int cnz, T* bc) {
    if (A.N == fine_N) begin(sizeof(T) == 4 ? "mg_restrict_f32_fine" : "mg_restrict_f64_fine");
    else begin(sizeof(T) == 4 ? "mg_restrict_f32" : "mg_restrict_f64");
    Op<T> B = A;
    B.skip = skip;
    const long long Nc = (long long)cnx * cny * cnz;
    const FastDiv fx = make_fastdiv((unsigned)cnx), fxy = make_fastdiv((unsigned)cnx * cny);
    const bool sym64 = sizeof(T) == 8 && A.loc && A.Wp[0] == A.W[0];
    if (Nc <= (sym64 ? RESTRICT_SPLIT_SYM : RESTRICT_SPLIT))
        k_mg_restrict_split<T><<<stream_blocks(Nc * 8), LIN_BLOCK, 0, st>>>(B, b, x, cnx, cny, cnz, fx, fxy, bc);
    else
        k_mg_restrict<T><<<stream_blocks(Nc), LIN_BLOCK, 0, st>>>(B, b, x, cnx, cny, cnz, fx, fxy, bc);
    return end();
}
template <typename T>
cudaError_t LinLaunch::prolong(int nx, int ny, int nz, int cnx, int cny, const T* xc, T* xf) {
    if ((long long)nx * ny * nz == fine_N) begin(sizeof(T) == 4 ? "mg_prolong_f32_fine" : "mg_prolong_f64_fine");
    else begin(sizeof(T) == 4 ? "mg_prolong_f32" : "mg_prolong_f64");
    constexpr int V = 16 / (int)sizeof(T);
    const long long NV = (long long)nx * ny * nz / V;
    // the vector form: whole 16-byte groups of fine cells along x, their parents at an offset
    // of V / 2 per group (cnx = nx / 2 is then a multiple of V / 2), aligned rows
    if (nx % V == 0 && cnx * 2 == nx && ((unsigned long long)xf & 15ull) == 0 &&
        ((unsigned long long)xc & (sizeof(T) * V / 2 - 1)) == 0) {
        k_mg_prolong_vec<T><<<stream_blocks(NV), LIN_BLOCK, 0, st>>>(
            nx, ny, nz, cnx, cny, make_fastdiv((unsigned)(nx / V)), make_fastdiv((unsigned)(nx / V) * ny),
            xc, xf, skip);
    } else {
        k_mg_prolong<T><<<stream_blocks((long long)nx * ny * nz), LIN_BLOCK, 0, st>>>(
            nx, ny, nz, cnx, cny, make_fastdiv((unsigned)nx), make_fastdiv((unsigned)nx * ny), xc,
            xf, skip);
    }
    return end();
}
template <typename TF, typename TC>
cudaError_t LinLaunch::build_level(const Op<TF>& A, const MgLevel<TC>& c, double omega) {
    begin("mg_build");
    // a cell's chain of FP64 additions (64 cycles each) is the time of a small level: small blocks spread its
    // warps over all SMs
    const int block = c.N < 152LL * LIN_BLOCK ? 64 : LIN_BLOCK;
    k_mg_build<TF, TC><<<(unsigned)((c.N + block - 1) / block), block, 0, st>>>(
        A, c, make_fastdiv((unsigned)c.nx), make_fastdiv((unsigned)c.nx * c.ny), omega);
    return end();
}
template <typename TF, typename TC>
cudaError_t LinLaunch::build_levels(const Op<TF>& A, const MgLevel<TC>* c, int n, double omega,
                                    int blocks) {
    begin("mg_build_tail");
    BuildArgs<TC> B{};
    B.n = n;
    B.omega = omega;
    for (int l = 0; l < n; ++l) B.c[l] = c[l];
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = blocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(LIN_BLOCK);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_mg_build_tail<TF, TC>, A, B);
    const cudaError_t e2 = end();
    return e != cudaSuccess ? e : e2;
}
// the cluster of the coarse-end kernel (16 blocks, a non-portable size) for the build too; called for
// every handle
cudaError_t mg_build_init() {
    cudaError_t e = cudaFuncSetAttribute(k_mg_build_tail<double, double>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mg_build_tail<double, float>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_mg_build_tail<float, float>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}
template <typename TF, typename TO>
cudaError_t LinLaunch::level_prep(const Op<TF>& A, double omega, TO* wid, TO* loc) {
    begin("mg_level_prep");
    k_mg_level_prep<TF, TO><<<stream_blocks(A.N), LIN_BLOCK, 0, st>>>(A, omega, wid, loc);
    return end();
}
cudaError_t LinLaunch::cast_op(const Op<double>& A, float* d, float* const* w) {
    begin("mg_cast_op");
    k_cast_op<<<stream_blocks(A.N), LIN_BLOCK, 0, st>>>(A, d, w[0], w[1], w[2]);
    return end();
}
cudaError_t LinLaunch::to_f32(long long N, const double* a, float* b) {
    begin("mg_to_f32");
    if ((((unsigned long long)a | (unsigned long long)b) & 15ull) == 0)
        k_to_f32<true><<<stream_blocks((N + 3) / 4), LIN_BLOCK, 0, st>>>(N, a, b, skip);
    else
        k_to_f32<false><<<stream_blocks(N), LIN_BLOCK, 0, st>>>(N, a, b, skip);
    return end();
}
template cudaError_t LinLaunch::smooth<double>(const Op<double>&, const double*, const double*,
                                               double*, double, int, double*);
template cudaError_t LinLaunch::smooth<float>(const Op<float>&, const float*, const float*,
                                              float*, float, int, double*);
template cudaError_t LinLaunch::restrict_res<double>(const Op<double>&, const double*,
                                                     const double*, int, int, int, double*);
template cudaError_t LinLaunch::restrict_res<float>(const Op<float>&, const float*, const float*,
                                                    int, int, int, float*);
template cudaError_t LinLaunch::prolong<double>(int, int, int, int, int, const double*, double*);
template cudaError_t LinLaunch::prolong<float>(int, int, int, int, int, const float*, float*);
template cudaError_t LinLaunch::build_level<double, double>(const Op<double>&, const MgLevel<double>&, double);
template cudaError_t LinLaunch::build_level<double, float>(const Op<double>&, const MgLevel<float>&, double);
template cudaError_t LinLaunch::build_level<float, float>(const Op<float>&, const MgLevel<float>&, double);
template cudaError_t LinLaunch::build_levels<double, double>(const Op<double>&, const MgLevel<double>*, int, double, int);
template cudaError_t LinLaunch::build_levels<double, float>(const Op<double>&, const MgLevel<float>*, int, double, int);
template cudaError_t LinLaunch::build_levels<float, float>(const Op<float>&, const MgLevel<float>*, int, double, int);
template cudaError_t LinLaunch::level_prep<double, double>(const Op<double>&, double, double*,
                                                           double*);
template cudaError_t LinLaunch::level_prep<double, float>(const Op<double>&, double, float*, float*);

}  // namespace rhi
