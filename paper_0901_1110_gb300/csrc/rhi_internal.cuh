// Internal declarations shared by the CUDA translation units of librhi.
#pragma once

#include <cfloat>
#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "rhi.h"
#include "rhi_fastdiv.h"

namespace rhi {

// ---------------------------------------------------------------------------------------------
// physical constants (CGS)
constexpr double C_LIGHT = 2.99792458e10;
constexpr double K_BOLTZ = 1.380649e-16;
constexpr double M_H = 1.67262192e-24;    // proton mass
constexpr double EV = 1.602176634e-12;
constexpr double GAMMA = 5.0 / 3.0;
constexpr double SIGMA_SB = 5.670374419e-5;   // erg cm^-2 s^-1 K^-4

// rate table: 2^TABLE_BITS bins per octave of T over [2^0, 2^TABLE_OCTAVES) K
constexpr int TABLE_BITS = 6;
constexpr int TABLE_OCTAVES = 30;
constexpr int NBINS = TABLE_OCTAVES << TABLE_BITS;
constexpr int NRATES = 11;
// largest double below 2^30
constexpr double T_TABLE_MAX = 1073741823.9999998807907104;

// rate columns
enum { R_ALPHA_HII = 0, R_BETA_HI, R_ALPHA_HEII, R_BETA_HEI, R_ALPHA_HEIII, R_BETA_HEII,
       R_COOL_HI, R_COOL_HII, R_COOL_HEI, R_COOL_HEII, R_COOL_HEIII };

// Host: node values and in-bin slopes of every coefficient, layout [bin][rate] of
// (value at the bin's lower node, slope); NBINS * NRATES entries.
std::vector<double2> build_rate_table();

// ---------------------------------------------------------------------------------------------
// per-step constants handed to kernels by value
struct StepParams {
    int nx, ny, nz;
    long long N;
    FastDiv fd_nx, fd_nxy;            // division by nx and nx * ny
    int per_x, per_y, per_z;          // periodic axes
    int dir_mask;                     // bit d: face d (x-, x+, y-, y+, z-, z+) is Dirichlet
    double Eb[6];                     // E on the Dirichlet faces
    double ia3, adot_a;               // 1/a^3, adot / a
    double dth;                       // dt theta
    double half_adx;                  // a dx / 2
    double R_min;                     // limiter floor 1 / (a L)
    // face formulas, whose results come multiplied by dt theta: a dx / 4, 2 R_min, and with
    // d = c dth / (a dx)^2: 2 d, -1 / (2 d), d a dx / 2, d (a dx)^2 / 3 (no limiter) over (a dx)^2
    double quart_adx, R_min2, cF, cK, cV, cD;
    double kappa_floor;
    int isothermal, limiter;
    int limiter_newton;               // 1: keep dD/dE in the Newton matrix (non-symmetric S)
    double y_he;
    double u_e, u_n, u_E, iu_e, iu_n, iu_E;
    // constants of the local model: rho = cR n_H, n_tot = cN n_H + n_e, dT/de = cT n_H / n_tot,
    // cTR = cT / cR; with dt theta folded in: i3 = dth / a^3, cE3 = c dth / a^3, cdth = c dth,
    // madot_dth = m adot/a dth, adot2_dth = 2 adot/a dth, one_adot2 = 1 + adot2_dth; and with
    // the ratios of scalings: r_ne = u_n / u_e, r_en = u_e / u_n, the U column's cz0 (times heating
    // / rho) and cz[X] (times n_X), ksk[X] = d kappa / d n_X in scaled unknowns
    double cR, cN, cT, cTR, i3, cE3, cdth, madot_dth, adot2_dth, one_adot2, r_ne, r_en, cz0;
    double cz[3], ksk[3];
    double dtm1_dth, dt_dth;          // (theta - 1) / theta, 1 / theta
    double sk[3], pg[3], ph[3];
    double tau, tau_tiny;             // positivity cap: tau, 1e-13 tau
    // LTE coupling (eq. LTE_coupling; no species): constant opacities, T = lte_cT e
    int lte;
    double kappa_total, kappa_planck, lte_cT;
    const double2* __restrict__ table;
};

// ---------------------------------------------------------------------------------------------
// arithmetic

// Reciprocal to within one unit in the last place: the hardware's reciprocal seed (PTX
// rcp.approx.ftz.f64, about 20 bits) and one third-order Householder step r (1 + e + e^2) with
// e = 1 - d r, whose error is e^3 < 2^-55: three FP64 instructions where the IEEE division takes
// about ten.  For normal d below 2^1021 in size (a seed under 2^-1022 is flushed to 0); NaN for d = 0 or
// subnormal.
__device__ __forceinline__ double fast_rcp(double d) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    const double e = fma(-d, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// FP32 to FP64 on the integer pipe, exact for every value: a conversion instruction takes the FP64 pipe
// as long as an FMA (64 cycles a warp), which is most of a small level's build.  No branch; subnormals
// are scaled up in FP32 first.
__device__ __forceinline__ double widen(float f) {
    const bool small = (__float_as_uint(f) & 0x7fffffffu) < 0x00800000u;
    const unsigned u = __float_as_uint(small ? f * 18446744073709551616.0f : f), m = u & 0x7fffffffu;
    unsigned hi = (m >> 3) + (small ? (896u - 64u) << 20 : 896u << 20);
    hi = m == 0u ? 0u : hi;
    hi = m >= 0x7f800000u ? 0x7ff00000u | (m >> 3 & 0xfffffu) : hi;
    return __hiloint2double((int)((u & 0x80000000u) | hi), (int)(u << 29));
}
__device__ __forceinline__ double widen(double f) { return f; }

// z / (1 + exp(-z)).  Two special-function results each (192 a row bound the forward pass); FAST: the
// quotient from the reciprocal approximation and one residual correction, q + (z - q d) r, which rounds as
// the IEEE division does but for a last bit now and then, in 6 instructions instead of a division's 15
// or so.  The residual is not a number where exp(-z) overflows (r = 0, q = -0) and at z = inf: fmaxf then
// gives its other operand, and the results are the division's -0 and inf.  (A bound on d, from which r
// came too, left z / 3e38 and NaN there; bounds on q and d cost 304 against 288 us for 128^3 rows.)
// The guess keeps the division: its FP64 results are held to the bit, and its time is its FP64
// logarithms'.
template <bool FAST>
__device__ __forceinline__ float silu_f(float z) {
    if constexpr (!FAST) return z / (1.0f + __expf(-z));
    const float d = 1.0f + __expf(-z);
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(d));
    const float q = z * r;
    return fmaf(fmaxf(fmaf(-q, d, z), -FLT_MAX), r, q);
}

// A value the compiler cannot see through.  `for (int go = rare; go; go = opaque(0)) {...}` is an `if`
// that stays a branch: as predicated instructions, FP64 work of a rare case would take its time on
// the FP64 pipe in every case.
__device__ __forceinline__ int opaque(int v) {
    asm volatile("" : "+r"(v));
    return v;
}

// ---------------------------------------------------------------------------------------------
// grid helpers

struct Nbr {
    long long lo[3], hi[3];           // neighbour indices (valid only where the face exists)
    bool has_lo[3], has_hi[3];        // face carries flux
};

__device__ __forceinline__ void cell_coords(const StepParams& P, long long c, int& i, int& j,
                                            int& k) {
    const unsigned cu = (unsigned)c;
    const unsigned kk = fdiv(cu, P.fd_nxy);
    const unsigned r = cu - kk * P.fd_nxy.d;
    const unsigned jj = fdiv(r, P.fd_nx);
    k = (int)kk;
    j = (int)jj;
    i = (int)(r - jj * P.fd_nx.d);
}

__device__ __forceinline__ Nbr neighbours(const StepParams& P, long long c, int i, int j, int k) {
    Nbr b;
    const long long sx = 1, sy = P.nx, sz = (long long)P.nx * P.ny;
    const int n[3] = {P.nx, P.ny, P.nz};
    const int q[3] = {i, j, k};
    const long long s[3] = {sx, sy, sz};
    const int per[3] = {P.per_x, P.per_y, P.per_z};
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        if (q[ax] > 0) { b.lo[ax] = c - s[ax]; b.has_lo[ax] = true; }
        else if (per[ax]) { b.lo[ax] = c + (long long)(n[ax] - 1) * s[ax]; b.has_lo[ax] = true; }
        else { b.lo[ax] = c; b.has_lo[ax] = false; }
        if (q[ax] < n[ax] - 1) { b.hi[ax] = c + s[ax]; b.has_hi[ax] = true; }
        else if (per[ax]) { b.hi[ax] = c - (long long)(n[ax] - 1) * s[ax]; b.has_hi[ax] = true; }
        else { b.hi[ax] = c; b.has_hi[ax] = false; }
    }
    return b;
}

// ---------------------------------------------------------------------------------------------
// Deterministic block reduction of a double; result valid in thread 0.  One warp adds everything: a
// warp's FP64 instruction takes its sub-partition's pipe for 64 cycles whatever its lanes hold, so
// 12 instructions of one warp cost less than 5 of each of eight warps.
template <int BLOCK>
__device__ __forceinline__ double block_sum(double v) {
    __shared__ double part[BLOCK];
    part[threadIdx.x] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < 32) {
        s = part[threadIdx.x];
#pragma unroll
        for (int q = 1; q < BLOCK / 32; ++q) s += part[threadIdx.x + 32 * q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    }
    __syncthreads();
    return s;
}

// two sums at once, by two warps; valid in thread 0
template <int BLOCK>
__device__ __forceinline__ void block_sum2(double& v1, double& v2) {
    static_assert(BLOCK >= 64, "two warps");
    __shared__ double part[2][BLOCK];
    part[0][threadIdx.x] = v1;
    part[1][threadIdx.x] = v2;
    __syncthreads();
    if (threadIdx.x < 64) {
        const double* p = part[threadIdx.x >> 5] + (threadIdx.x & 31);
        double s = p[0];
#pragma unroll
        for (int q = 1; q < BLOCK / 32; ++q) s += p[32 * q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        v1 = s;
        if (threadIdx.x == 32) part[1][0] = s;
    }
    __syncthreads();
    v2 = part[1][0];
    __syncthreads();
}

// Grid-wide sum without a second launch: every block writes its partial and takes a ticket; the
// block with the last one (true) adds the partials in a fixed order, so the result does not depend on
// the order the blocks ended in.  Returns true in all threads of that block; the sums are valid in
// its thread 0.  The counter wraps to 0 by itself; launches that share it run one after another.
template <int BLOCK, bool TWO>
__device__ __forceinline__ bool grid_sum(double v1, double v2, double* partials, unsigned* count,
                                         double& s1, double& s2) {
    __shared__ bool last_block;
    const int n = (int)gridDim.x;
    s1 = v1;
    s2 = v2;
    if constexpr (TWO) block_sum2<BLOCK>(s1, s2);
    else s1 = block_sum<BLOCK>(v1);
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = s1;
        if (TWO) partials[n + blockIdx.x] = s2;
        last_block = false;
        if (count) {
            // the ticket releases this thread's partials and, with the last one, acquires all others'
            // (for the block by way of its barrier)
            unsigned t;
            asm volatile("atom.acq_rel.gpu.global.inc.u32 %0, [%1], %2;"
                         : "=r"(t) : "l"(count), "r"((unsigned)n - 1u) : "memory");
            last_block = t == (unsigned)n - 1u;
        }
    }
    __syncthreads();
    if (!last_block) return false;
    double a1 = 0.0, a2 = 0.0;
    for (int q = (int)threadIdx.x; q < n; q += BLOCK) {
        a1 += __ldcg(partials + q);
        if (TWO) a2 += __ldcg(partials + n + q);
    }
    s1 = a1;
    s2 = a2;
    if constexpr (TWO) block_sum2<BLOCK>(s1, s2);
    else s1 = block_sum<BLOCK>(a1);
    return true;
}

// ---------------------------------------------------------------------------------------------
// kernel launch wrappers (defined in the .cu files); all return cudaGetLastError()

struct PhysBuffers {
    // state U^n
    const double* E_n;
    const double* n_n;      // ns * N
    const double* eh;       // e^n (specific energy before the step)
    const double* nH;
    const double* src;
    const double* Tiso;
    // iterate U (e_c, n, E) and its opacity
    const double* ec;       // may be null: e_c = 0
    const double* n;
    const double* E;
    const double* kap;
    // per lower face, times dt theta (3 * N): the coefficients W (limiter_jacobian 0), or with
    // `flux` the fluxes W (E_c - E_lower), all the residual needs
    const double* W;
    int flux;
    double* g;              // (ns + 2) * N
    // outputs of the cell kernel
    // Schur diagonal (scaled): complete (D lagged), or with `flux` its local part, which
    // launch_schur_assemble completes
    double* diag;
    double* rhs;            // Schur right-hand side (scaled), without the faces' opacity terms
    // exact matrix: the cell's opacity response to its E and to its residual,
    // (d kappa / d n) M^-1 U and (d kappa / d n) M^-1 f_M (scaled; null: not needed)
    double* rho;
    double* phi;
    double* fMt;            // (ns + 1) * N   M^-1 f_M (scaled)
    double* MiU;            // (ns + 1) * N   M^-1 U  (scaled)
    double* f_out;          // optional (ns + 2) * N scaled residual
    double* partials;       // per-block sums of the squared scaled residual
    unsigned* count;        // with it, their sum goes to *norm_sq (null: partials only)
    double* norm_sq;
    double* U0;             // optional predictor output (ns + 2) * N
};

enum CellMode { MODE_PREP = 0, MODE_ITER = 1, MODE_PREP_PREDICT = 2, MODE_RESID = 3 };

cudaError_t launch_kappa(const StepParams& P, int ns, const double* n, double* kap,
                         cudaStream_t st);
// Face arrays, times dt theta.  jm (limiter_jacobian) 0: the coefficients W.  1, 2: the fluxes
// W (E_c - E_lower) into W, the Newton-matrix entries P and Q into PQ (6 N) and, for 2, the opacity
// terms K.  resid_only: W (fluxes) alone, with the same arithmetic.
cudaError_t launch_faces(const StepParams& P, int jm, int resid_only, const double* E,
                         const double* kap, double* W, double* PQ, double* K, cudaStream_t st);
// The Newton matrix in E of limiter_jacobian 1 or 2 from an evaluated iterate: entries PQ (P then
// Q per lower face, times dt theta), diagonal and right-hand side, and the finest level of the
// multigrid hierarchy built from it (f32: the FP32 operator; wid64: omega / diagonal; or neither).
struct SchurIn {
    const double *PQ, *K, *dloc, *rhs, *rho, *phi;   // K, rho, phi null: limiter_jacobian 1
};
struct SchurOut {
    double *PQ, *diag, *rhs;
    float *d32, *wid32, *W32[3], *Wp32[3];
    double* wid64;
    double omega;
};
cudaError_t launch_schur_assemble(const StepParams& P, const SchurIn& I, const SchurOut& O,
                                  cudaStream_t st);
// Schur diagonal of the lagged-D matrix (coefficients W) from the local part dloc of the Newton
// matrix's
cudaError_t launch_lagged_diag(const StepParams& P, const double* W, const double* dloc,
                               const double* E, const double* kap, double* diag, cudaStream_t st);
cudaError_t launch_export_faces(const StepParams& P, const double* Q, const double* Pf,
                                double* S_lo, double* S_hi, cudaStream_t st);
cudaError_t launch_cell(const StepParams& P, int ns, int mode, const PhysBuffers& B,
                        int nblocks, cudaStream_t st);
int cell_block_size();
cudaError_t launch_update(const StepParams& P, int ns, double lam, const double* ec0,
                          const double* n0, const double* E0, const double* eh,
                          const double* nH, const double* sE, const double* fMt,
                          const double* MiU, double* ec1, double* n1, double* E1,
                          double* kap1, cudaStream_t st);
cudaError_t launch_finalize(const StepParams& P, int ns, const double* ec, double* eh,
                            cudaStream_t st);
cudaError_t launch_temperature(const StepParams& P, int ns, const double* e, const double* n,
                               const double* nH, double* T, cudaStream_t st);
cudaError_t launch_check_state(const StepParams& P, int ns, const double* E, const double* e,
                               const double* n, const double* nH, int* bad, cudaStream_t st);
// emissivity of up to SOURCE_BATCH point sources added to src, in their order
constexpr int SOURCE_BATCH = 128;
struct SourceBatch {
    int n;
    long long cell[SOURCE_BATCH];
    double value[SOURCE_BATCH];
};
cudaError_t launch_deposit(const SourceBatch& S, double* src, cudaStream_t st);
// block partials (nblocks of 256 threads) of the step's error estimate against the predictor
// Up: sum of q^pn, or max q when pn < 0
cudaError_t launch_time_error(const StepParams& P, int ns, const double* ec, const double* n,
                              const double* E, const double* Up, double pn, double* partials,
                              int nblocks, cudaStream_t st);

}  // namespace rhi
