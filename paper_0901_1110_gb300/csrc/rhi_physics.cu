// Cell-local physics of the implicit step: opacity, limiter face coefficients, the fused
// residual / Jacobian / Schur-elimination kernel, the Newton update with positivity cap, and
// small state kernels.  All FP64.
//
// Reference passages: Sec. 3.2 (theta scheme, eqs. energy/chemistry/radiation_simplified,
// operators mDE, mLe, mLn, mLE, residual eq. nonlinear_residual, RMS norm eq. rmsnorm),
// Sec. 3.2.1 (Newton matrix eqs. jacobian_matrix / jacobian_submatrices, Schur steps (i)-(iii),
// eqs. newton_system2, schur_components, step_ia), Sec. 3.2.2 (scalings eq. scalings),
// Sec. 2.2 (limiter eq. limiter).
#include "rhi_internal.cuh"

namespace rhi {

constexpr int CELL_BLOCK = 128;
int cell_block_size() { return CELL_BLOCK; }

// ---------------------------------------------------------------------------------------------
// opacity kappa = sum_X sk_X n_X / a^3

__global__ void k_kappa(const StepParams P, int ns, const double* __restrict__ n,
                        double* __restrict__ kap) {
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c >= P.N) return;
    if (ns == 0) { kap[c] = P.kappa_total; return; }          // LTE: constant opacity
    double s = P.sk[0] * n[c];
    if (ns == 3) s += P.sk[1] * n[P.N + c] + P.sk[2] * n[2 * P.N + c];
    kap[c] = P.ia3 * s;
}

cudaError_t launch_kappa(const StepParams& P, int ns, const double* n, double* kap,
                         cudaStream_t st) {
    const int b = 256;
    k_kappa<<<(unsigned)((P.N + b - 1) / b), b, 0, st>>>(P, ns, n, kap);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// face coefficients D / (a dx)^2 of each cell's three lower faces (eq. limiter)
//
// R = |E_b - E_a| / (a dx Ebar) floored at R_min; with q = max(|dE|, R_min a dx Ebar) and
// s = a dx Ebar, D = c s (2 kappa s + q) / (6 kappa^2 s^2 + 3 kappa q s + q^2): one division.
//
// With dD/dE kept in the Newton matrix (Sec. 3.2.1 lags only the opacity), the face between
// lower cell a and upper cell b (dE = E_b - E_a) contributes dt theta P to b's diagonal and
// -dt theta Q to (b, a), dt theta Q to a's diagonal and -dt theta P to (a, b), where
// P = W + (dW/dE_b) dE and Q = W - (dW/dE_a) dE.  With R dD/dR = -c q^2 (4 kappa s + q) s / den^2
// and t = dE / (E_a + E_b): P = W + R dD/dR (1 - t) / (a dx)^2, Q = W + R dD/dR (1 + t) / (a dx)^2
// (both = W where R sits at its floor).
//
// The exact Newton matrix also keeps D's opacity dependence: K = (1/2) (dW/dkappa) dE per face,
// with dD/dkappa = -c s^2 (12 kappa^2 s^2 + 12 kappa s q + q^2) / den^2 (the quotient rule on
// eq. limiter; each cell's kappa enters the face mean with weight 1/2).

struct FaceCoef { double W, P, Q, K; };

// JM: 0 W only; 1 W, P, Q (dD/dE kept); 2 W, P, Q, K (exact)
// The limiter's face coefficients depend on (s, dE) = (a dx Ebar, E_b - E_a) only through
// their ratio: W, P and Q, and K apart from its factor dE, are homogeneous of degree 0.  Their
// squares and the 1 / den^2 of the derivatives leave the FP64 range once Ebar falls below about
// 1e-90 (deep neutral gas after many absorbing steps), and the result turns into 0 / 0 or
// x * inf.  A faint face is therefore brought to s in [1, 2) by a power of two, which is exact;
// the test runs on the bit pattern (integer pipe), s > 0 and below 2^-64.
__device__ __forceinline__ void faint_rescale(double& s, double& dE) {
    const long long sb = __double_as_longlong(s);
    if (sb > 0 && sb < 0x3BF0000000000000LL) {
        const int e = ilogb(s);
        s = scalbn(s, -e);
        dE = scalbn(dE, -e);
    }
}

// FP64 instructions bound the face kernel, so with h = s / 2 and k = kappa s = (ka + kb) h the
// formulas share their parts: m = 2 k + q gives den = 3 k m + q^2; B = 2 c h / (den (a dx)^2)
// gives W = B m and K = -B^2 (12 k (k + q) + q^2) dE (a dx)^2 / (2 c); and
// G = q^2 (4 k + q) / den^2 gives the derivative terms, R dD/dR / (a dx)^2 = -2 c h G / (a dx)^2.
// The floor of q compares bit patterns (integer pipe).  Measured at 256^3, exact matrix: 2.99 ms per
// launch against 4.24 ms for the separate formulas with an IEEE division (W alone: 1.59, 2.14 ms).
template <int JM, bool WONLY = false>
__device__ __forceinline__ FaceCoef face_coef(const StepParams& P, double Ea, double Eb,
                                              double ka, double kb) {
    FaceCoef r;
    r.K = 0.0;
    if (P.limiter) {
        double h = (Ea + Eb) * P.quart_adx;                     // a dx Ebar / 2
        const double dE = Eb - Ea;
        double dEs = dE;                                        // dE on the scale of h
        faint_rescale(h, dEs);
        const double qraw = fabs(dEs), qmin = P.R_min2 * h;
        const bool free_R = __double_as_longlong(qraw) > __double_as_longlong(qmin);
        const double q = free_R ? qraw : qmin;
        const double k = (ka + kb) * h;
        const double m = fma(2.0, k, q), k3 = 3.0 * k, q2 = q * q;
        const double iden = fast_rcp(fma(k3, m, q2));
        const double A = P.cF * h;
        const double Bf = A * iden;
        r.W = Bf * m;
        if (JM == 0 || WONLY) {
            r.P = r.Q = r.W;
            return r;
        }
        if (JM == 2) r.K = (Bf * Bf) * (fma(4.0 * k3, k + q, q2) * (P.cK * dE));
        const double G = free_R ? q2 * fma(4.0, k, q) * (iden * iden) : 0.0;
        const double u = fma(-A, G, r.W), v = P.cV * dEs;
        r.P = fma(v, G, u);
        r.Q = fma(-v, G, u);
        return r;
    }
    r.W = P.cD / fmax(0.5 * (ka + kb), P.kappa_floor);
    r.P = r.Q = r.W;
    if (JM == 2 && 0.5 * (ka + kb) > P.kappa_floor) r.K = -0.5 * r.W / (0.5 * (ka + kb)) * (Eb - Ea);
    return r;
}

// A Dirichlet face: the boundary value E_b sits on the face, half a cell from the centre, and
// the face's opacity is the cell's.  The coefficient is D / (a^2 dx dx/2) with R over that
// half-cell distance (s = a (dx/2) Ebar); Qd is the cell's Newton-diagonal entry
// W - dW/dE_c (E_b - E_c) and dWdk = dW/dkappa (exact matrix).
struct BoundaryFace { double W, Qd, dWdk; };         // times dt theta

__device__ __forceinline__ BoundaryFace boundary_face(const StepParams& P, double E, double Eb,
                                                      double kap) {
    BoundaryFace r;
    if (P.limiter) {
        const double Esum = E + Eb;
        double s = 0.5 * Esum * P.half_adx;
        double dE = Eb - E;
        faint_rescale(s, dE);
        const double qraw = fabs(dE);
        const double q = fmax(qraw, P.R_min * s);
        const double ks = kap * s;
        const double den = 6.0 * ks * ks + 3.0 * ks * q + q * q;
        const double iden = 1.0 / den;
        r.W = s * (2.0 * ks + q) * iden * P.cF;
        r.Qd = r.W;
        if (P.limiter_newton >= 1 && qraw > P.R_min * s) {
            const double X = -q * q * (4.0 * ks + q) * iden * iden * P.cF;
            r.Qd = r.W + X * s + X * dE * 0.5 * P.half_adx;
        }
        r.dWdk = -s * s * (12.0 * ks * ks + 12.0 * ks * q + q * q) * iden * iden * P.cF;
        return r;
    }
    r.W = 2.0 * P.cD / fmax(kap, P.kappa_floor);
    r.Qd = r.W;
    r.dWdk = kap > P.kappa_floor ? -r.W / kap : 0.0;
    return r;
}

// JM 0: the coefficients W.  JM 1, 2: the fluxes W (E_c - E_lower), which are all the residual
// needs (each computed once per face instead of by both cells of it), P, Q and K; WONLY: the fluxes
// alone (a trial iterate evaluated for its residual), by the same arithmetic.
template <int JM, bool WONLY = false>
__global__ void __launch_bounds__(256) k_faces(const StepParams P, const double* __restrict__ E,
                                               const double* __restrict__ kap,
                                               double* __restrict__ W, double* __restrict__ PQv,
                                               double* __restrict__ Kv) {
    constexpr bool PQ = JM >= 1 && !WONLY;
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c >= P.N) return;
    int i, j, k;
    cell_coords(P, c, i, j, k);
    const Nbr b = neighbours(P, c, i, j, k);
    const double Ec = E[c], kc = kap[c];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        FaceCoef f{0.0, 0.0, 0.0, 0.0};
        const double El = E[b.lo[ax]];
        if (b.has_lo[ax]) f = face_coef<JM, WONLY>(P, El, Ec, kap[b.lo[ax]], kc);
        W[ax * P.N + c] = JM == 0 ? f.W : f.W * (Ec - El);
        if (PQ) {
            PQv[ax * P.N + c] = f.P;
            PQv[(3 + ax) * P.N + c] = f.Q;
        }
        if (JM == 2 && !WONLY) Kv[ax * P.N + c] = f.K;
    }
}

cudaError_t launch_faces(const StepParams& P, int jm, int resid_only, const double* E,
                         const double* kap, double* W, double* PQ, double* K, cudaStream_t st) {
    const int b = 256;
    const unsigned g = (unsigned)((P.N + b - 1) / b);
    if (jm == 2 && !resid_only && !K) jm = 1;          // constant opacity: no opacity terms
    if (jm == 0) k_faces<0><<<g, b, 0, st>>>(P, E, kap, W, nullptr, nullptr);
    else if (jm == 1 && resid_only) k_faces<1, true><<<g, b, 0, st>>>(P, E, kap, W, nullptr, nullptr);
    else if (jm == 1) k_faces<1><<<g, b, 0, st>>>(P, E, kap, W, PQ, nullptr);
    else if (resid_only) k_faces<2, true><<<g, b, 0, st>>>(P, E, kap, W, nullptr, nullptr);
    else k_faces<2><<<g, b, 0, st>>>(P, E, kap, W, PQ, K);
    return cudaGetLastError();
}

// Newton matrix in E.  The diagonal is the local part plus the row's own face entries, P of its
// lower faces and Q of its upper ones.  In the exact matrix the E row of a cell also couples to the
// species of the cell and of its face neighbours through D's opacity: after the cell-local
// elimination dn_j = -M_j^-1 f_M,j - M_j^-1 U_j dE_j, face f (lower cell l, upper cell u, stored at
// u) adds, with rho_j = sum_X (dkappa/dn_X) (M^-1 U)_j,X and phi_j likewise with M^-1 f_M (scaled),
//   P_f -= K_f rho_u,  Q_f += K_f rho_l,
//   rhs_u += K_f (phi_l + phi_u),  rhs_l -= K_f (phi_l + phi_u),
// and the diagonal follows from the changed P and Q.  The cell kernel hands over rho and phi, so a
// face costs four FMAs here.  Each thread writes its cell's three lower faces, out of place: the
// cell below reads this cell's original Q and K.  The finest multigrid level, copied from the same
// entries, is written in the same pass.
//
// Bound by the FP64 pipe, with HBM close behind (200 B per cell with the FP32 level).  Measured at
// 256^3, H + He: 1.21 ms, against 2.68 ms for the in-place opacity coupling that formed rho and phi of
// every neighbour, the FP32 copy and the omega / diagonal pass that this replaces; the cell
// kernel without the diagonal's face sums and with one flux per face 7.39 against 8.09 ms.
template <bool KAPPA, int PC>
__global__ void __launch_bounds__(256) k_schur_assemble(const StepParams P, const SchurIn I,
                                                        const SchurOut O) {
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long N = P.N;
    if (c >= N) return;
    int i, j, k;
    cell_coords(P, c, i, j, k);
    const Nbr b = neighbours(P, c, i, j, k);
    double rc = 0.0, pc = 0.0;
    if (KAPPA) { rc = __ldg(I.rho + c); pc = __ldg(I.phi + c); }
    double diag = __ldg(I.dloc + c), dr = 0.0;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        double p = 0.0, q = 0.0;
        if (b.has_lo[ax]) {
            const long long l = b.lo[ax];
            p = __ldg(I.PQ + ax * N + c);
            q = __ldg(I.PQ + (3 + ax) * N + c);
            if (KAPPA) {
                const double K = __ldg(I.K + ax * N + c);
                p = fma(-K, rc, p);
                q = fma(K, __ldg(I.rho + l), q);
                dr = fma(K, __ldg(I.phi + l) + pc, dr);
            }
            diag += p;
        }
        if (b.has_hi[ax]) {
            const long long h = b.hi[ax];
            double qh = __ldg(I.PQ + (3 + ax) * N + h);
            if (KAPPA) {
                const double K = __ldg(I.K + ax * N + h);
                qh = fma(K, rc, qh);
                dr = fma(-K, pc + __ldg(I.phi + h), dr);
            }
            diag += qh;
        }
        O.PQ[ax * N + c] = p;
        O.PQ[(3 + ax) * N + c] = q;
        if (PC == 1) {
            O.W32[ax][c] = (float)(q);
            O.Wp32[ax][c] = (float)(p);
        }
    }
    O.diag[c] = diag;
    O.rhs[c] = __ldg(I.rhs + c) + dr;
    if (PC == 1) {
        O.d32[c] = (float)(diag);
        O.wid32[c] = (float)(O.omega * fast_rcp(diag));
    }
    if (PC == 2) O.wid64[c] = O.omega * fast_rcp(diag);
}

cudaError_t launch_schur_assemble(const StepParams& P, const SchurIn& I, const SchurOut& O,
                                  cudaStream_t st) {
    const int b = 256;
    const unsigned g = (unsigned)((P.N + b - 1) / b);
    const int pc = O.d32 ? 1 : (O.wid64 ? 2 : 0);
    if (I.K) {
        if (pc == 1) k_schur_assemble<true, 1><<<g, b, 0, st>>>(P, I, O);
        else if (pc == 2) k_schur_assemble<true, 2><<<g, b, 0, st>>>(P, I, O);
        else k_schur_assemble<true, 0><<<g, b, 0, st>>>(P, I, O);
    } else {
        if (pc == 1) k_schur_assemble<false, 1><<<g, b, 0, st>>>(P, I, O);
        else if (pc == 2) k_schur_assemble<false, 2><<<g, b, 0, st>>>(P, I, O);
        else k_schur_assemble<false, 0><<<g, b, 0, st>>>(P, I, O);
    }
    return cudaGetLastError();
}

// Diagonal of the lagged-D matrix (the breakdown fallback, the mg_matrix = 0 hierarchy and the
// Jacobi preconditioner of a solver that keeps dD/dE): the local part, whose Dirichlet faces carry
// the Newton entry, plus the coefficients W of the six faces.
__global__ void k_lagged_diag(const StepParams P, const double* __restrict__ W,
                              const double* __restrict__ dloc, const double* __restrict__ E,
                              const double* __restrict__ kap, double* __restrict__ diag) {
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c >= P.N) return;
    int i, j, k;
    cell_coords(P, c, i, j, k);
    const Nbr b = neighbours(P, c, i, j, k);
    double d = dloc[c];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        d += W[ax * P.N + c];
        if (b.has_hi[ax]) d += W[ax * P.N + b.hi[ax]];
    }
    if (P.dir_mask) {
        const int q[3] = {i, j, k};
        const int ext[3] = {P.nx, P.ny, P.nz};
        for (int f = 0; f < 6; ++f) {
            const int ax = f >> 1;
            if ((P.dir_mask >> f & 1) && q[ax] == ((f & 1) ? ext[ax] - 1 : 0)) {
                const BoundaryFace bf = boundary_face(P, E[c], P.Eb[f], kap[c]);
                d += bf.W - bf.Qd;
            }
        }
    }
    diag[c] = d;
}

cudaError_t launch_lagged_diag(const StepParams& P, const double* W, const double* dloc,
                               const double* E, const double* kap, double* diag, cudaStream_t st) {
    const int b = 256;
    k_lagged_diag<<<(unsigned)((P.N + b - 1) / b), b, 0, st>>>(P, W, dloc, E, kap, diag);
    return cudaGetLastError();
}

// Newton-matrix face entries of each cell for inspection: S_lo[ax] couples a cell to its
// lower neighbour, S_hi[ax] to its upper neighbour (positive numbers; the matrix entries are
// their negatives; 0 where the face carries no flux).
__global__ void k_export_faces(const StepParams P, const double* __restrict__ Q,
                               const double* __restrict__ Pf, double* __restrict__ lo,
                               double* __restrict__ hi) {
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c >= P.N) return;
    int i, j, k;
    cell_coords(P, c, i, j, k);
    const Nbr b = neighbours(P, c, i, j, k);
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        if (lo) lo[ax * P.N + c] = Q[ax * P.N + c];
        if (hi) hi[ax * P.N + c] = b.has_hi[ax] ? Pf[ax * P.N + b.hi[ax]] : 0.0;
    }
}

// Q, Pf: the rows' couplings to the lower and from the lower cell per lower face (equal for the
// lagged-D matrix); S_lo or S_hi may be null
cudaError_t launch_export_faces(const StepParams& P, const double* Q, const double* Pf,
                                double* S_lo, double* S_hi, cudaStream_t st) {
    const int b = 256;
    k_export_faces<<<(unsigned)((P.N + b - 1) / b), b, 0, st>>>(P, Q, Pf, S_lo, S_hi);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// local reaction operators and their derivatives (eqs. mLe, mLn, mLE, jacobian_submatrices)

// What the cell kernel takes from the local operators, scaled at the source: every operator comes
// multiplied by dt theta and the Jacobian already as the block M = I + dt theta dL/dx of
// eq. schur_components in scaled unknowns.
//
// FP64 instructions bound the cell kernel (2 per clock per SM), so the formulas are arranged to
// need few of them.  The species and the energy depend on n_e and T through the same two numbers, so
// the Jacobian is a sparse part plus a rank-one part: d n_e / d n = (-1, -2, -1) times
// q_r = dt theta / a^3 (B_r + n_e dB_r/dT dT/dn_e) for row r.  B2 = b2 n_HeII - B1 - a2 n_HeIII
// reuses B1; dt theta and the ratios of scalings sit in per-step constants.
// Measured at 256^3, H + He, exact matrix: 8.09 ms per launch against 11.33 ms for the term by term
// form with IEEE divisions and FP64 comparisons (f alone: 3.27 against 3.98 ms).
template <int NS>
struct Local {
    double L[NS + 1];          // dt theta L_e, dt theta L_n1 ..
    double LE;                 // dt theta times the local part of the E operator
    double M[NS + 1][NS + 1];  // scaled block M
    double zU[NS + 1];         // scaled column U
    double dLEE;               // dt theta dL_E/dE
    double LrE;                // NS = 0: scaled entry of the row L
};

template <int NS, bool JAC>
__device__ __forceinline__ void local_model(const StepParams& P, double ec,
                                            const double (&n)[NS > 0 ? NS : 1],
                                            double E, double eh, double nH, double src,
                                            double Tfix, Local<NS>& o) {
    if constexpr (NS == 0) {
        // LTE coupling (eq. LTE_coupling): emission 4 pi eta = 4 kappa_P sigma T^4, heating
        // c kappa E / rho, cooling 4 pi eta / rho; T = lte_cT e
        const double irho = fast_rcp(P.cR * nH);
        const double e = eh + ec;
        const double T = P.isothermal ? Tfix : P.lte_cT * e;
        const double T2 = T * T;
        const double emis = P.dth * 4.0 * P.kappa_planck * SIGMA_SB * T2 * T2;
        const double ck = P.dth * C_LIGHT * P.kappa_total;
        const double ckE = ck * E;
        o.L[0] = P.isothermal ? 0.0 : fma(P.dth * 2.0 * P.adot_a, ec, (emis - ckE) * irho);
        o.LE = fma(P.madot_dth, E, -P.dth * src) + (ckE - emis);
        if constexpr (!JAC) return;
        const double demis = P.isothermal ? 0.0 : P.dth * 16.0 * P.kappa_planck * SIGMA_SB * T2 * T * P.lte_cT;
        o.M[0][0] = P.isothermal ? 1.0 : 1.0 + P.dth * 2.0 * P.adot_a + demis * irho;
        o.zU[0] = P.isothermal ? 0.0 : -ck * irho * (P.u_E * P.iu_e);
        o.LrE = -demis * (P.u_e * P.iu_E);
        o.dLEE = P.madot_dth + ck;
        return;
    } else {
    const double nHI = n[0];
    double nHeI = 0.0, nHeII = 0.0, nHeIII = 0.0;
    const double nHII = nH - nHI;
    double ne = nHII;
    if constexpr (NS == 3) {
        nHeI = n[1];
        nHeII = n[2];
        nHeIII = P.y_he * nH - nHeI - nHeII;
        ne = fma(2.0, nHeIII, nHII + nHeII);
    }
    const double irho = fast_rcp(P.cR * nH);
    const double intot = fast_rcp(fma(P.cN, nH, ne));
    const double e = eh + ec;
    double T, dT_dec, dT_dne;
    if (P.isothermal) {
        T = Tfix;
        dT_dec = 0.0;
        dT_dne = 0.0;
    } else {
        dT_dec = P.cT * nH * intot;                         // T is proportional to e
        T = dT_dec * e;
        dT_dne = -T * intot;                                // d n_tot = d n_e
    }

    // tabulated coefficients: bin = binary exponent and top mantissa bits of clamped T.  T >= 1
    // and T <= T_TABLE_MAX are tested on the bit pattern (integer pipe); a negative T is below 1
    const long long tb = __double_as_longlong(T);
    constexpr long long ONE = 0x3FF0000000000000LL, TMAX = 0x41CFFFFFFFFFFFFFLL;
    const bool below = tb < ONE, above = tb > TMAX;
    const unsigned long long bits = (unsigned long long)(below ? ONE : (above ? TMAX : tb));
    const double Tc = __longlong_as_double((long long)bits);
    const int bin = (int)((bits >> (52 - TABLE_BITS)) - (1023ull << TABLE_BITS));
    const double Ti = __longlong_as_double((long long)(bits & ~((1ull << (52 - TABLE_BITS)) - 1ull)));
    const double dTi = Tc - Ti;
    const double2* row = P.table + (long long)bin * NRATES;
    double k[NRATES], dk[NRATES];
#pragma unroll
    for (int r = 0; r < NRATES; ++r) {
        const bool need = (NS == 3) || r == R_ALPHA_HII || r == R_BETA_HI || r == R_COOL_HI ||
                          r == R_COOL_HII;
        if (need) {
            const double2 v = __ldg(row + r);
            k[r] = fma(v.y, dTi, v.x);
            dk[r] = (below || above) ? 0.0 : v.y;
        } else {
            k[r] = 0.0;
            dk[r] = 0.0;
        }
    }
    double C = fma(k[R_COOL_HI], nHI, k[R_COOL_HII] * nHII);
    const double B0 = fma(k[R_BETA_HI], nHI, -(k[R_ALPHA_HII] * nHII));
    const double Ed = P.cE3 * E;                            // dt theta c E / a^3
    const double ne3 = P.i3 * ne;                           // dt theta n_e / a^3
    const double GHI = P.pg[0] * Ed;
    double heat = P.ph[0] * nHI, skn = P.sk[0] * nHI;
    o.L[1] = fma(GHI, nHI, ne3 * B0);
    double B1 = 0.0, B2 = 0.0, GHeI = 0.0, GHeII = 0.0;
    if constexpr (NS == 3) {
        C = fma(k[R_COOL_HEI], nHeI, C);
        C = fma(k[R_COOL_HEII], nHeII, C);
        C = fma(k[R_COOL_HEIII], nHeIII, C);
        B1 = fma(k[R_BETA_HEI], nHeI, -(k[R_ALPHA_HEII] * nHeII));
        B2 = fma(-k[R_ALPHA_HEIII], nHeIII, fma(k[R_BETA_HEII], nHeII, -B1));
        GHeI = P.pg[1] * Ed;
        GHeII = P.pg[2] * Ed;
        const double g1 = GHeI * nHeI;
        o.L[2] = fma(ne3, B1, g1);
        o.L[3] = fma(GHeII, nHeII, fma(ne3, B2, -g1));
        heat = fma(P.ph[1], nHeI, fma(P.ph[2], nHeII, heat));
        skn = fma(P.sk[1], nHeI, fma(P.sk[2], nHeII, skn));
    }
    o.L[0] = P.isothermal ? 0.0 : fma(P.adot2_dth, ec, irho * fma(ne3, C, -(Ed * heat)));
    o.dLEE = fma(P.cE3, skn, P.madot_dth);
    o.LE = fma(o.dLEE, E, -P.dth * src);
    if constexpr (!JAC) return;

    // energy row; column e of the species rows
    double dCdT = fma(dk[R_COOL_HI], nHI, dk[R_COOL_HII] * nHII);
    if constexpr (NS == 3) {
        dCdT = fma(dk[R_COOL_HEI], nHeI, dCdT);
        dCdT = fma(dk[R_COOL_HEII], nHeII, dCdT);
        dCdT = fma(dk[R_COOL_HEIII], nHeIII, dCdT);
    }
    if (P.isothermal) {
#pragma unroll
        for (int s = 0; s <= NS; ++s) o.M[0][s] = s == 0 ? 1.0 : 0.0;
        o.zU[0] = 0.0;
    } else {
        const double x0 = ne3 * dCdT;
        const double ir = irho * P.r_ne;
        const double q0 = ir * fma(x0, dT_dne, P.i3 * C), en = -(ir * Ed), ni = ir * ne3;
        o.M[0][0] = fma(x0, P.cTR * intot, P.one_adot2);    // cTR intot = dT_dec / rho
        o.M[0][1] = fma(ni, k[R_COOL_HI] - k[R_COOL_HII], fma(en, P.ph[0], -q0));
        if constexpr (NS == 3) {
            o.M[0][2] = fma(ni, k[R_COOL_HEI] - k[R_COOL_HEIII], fma(en, P.ph[1], -2.0 * q0));
            o.M[0][3] = fma(ni, k[R_COOL_HEII] - k[R_COOL_HEIII], fma(en, P.ph[2], -q0));
        }
        o.zU[0] = P.cz0 * heat * irho;
    }
    const double dTs = dT_dec * P.r_en;
    const double t0 = ne3 * fma(dk[R_BETA_HI], nHI, -(dk[R_ALPHA_HII] * nHII));
    const double q1 = fma(t0, dT_dne, P.i3 * B0);
    o.M[1][0] = t0 * dTs;
    o.M[1][1] = fma(ne3, k[R_BETA_HI] + k[R_ALPHA_HII], 1.0 + GHI) - q1;
    o.zU[1] = P.cz[0] * nHI;
    if constexpr (NS == 3) {
        const double dB1 = fma(dk[R_BETA_HEI], nHeI, -(dk[R_ALPHA_HEII] * nHeII));
        const double t1 = ne3 * dB1;
        const double t2 = ne3 * fma(-dk[R_ALPHA_HEIII], nHeIII, fma(dk[R_BETA_HEII], nHeII, -dB1));
        const double q2 = fma(t1, dT_dne, P.i3 * B1), q3 = fma(t2, dT_dne, P.i3 * B2);
        o.M[1][2] = -2.0 * q1;
        o.M[1][3] = -q1;
        o.M[2][0] = t1 * dTs;
        o.M[2][1] = -q2;
        o.M[2][2] = fma(-2.0, q2, fma(ne3, k[R_BETA_HEI], 1.0 + GHeI));
        o.M[2][3] = fma(-ne3, k[R_ALPHA_HEII], -q2);
        o.M[3][0] = t2 * dTs;
        o.M[3][1] = -q3;
        o.M[3][2] = fma(-2.0, q3, fma(ne3, k[R_ALPHA_HEIII] - k[R_BETA_HEI], -GHeI));
        o.M[3][3] = fma(ne3, k[R_BETA_HEII] + k[R_ALPHA_HEII] + k[R_ALPHA_HEIII], 1.0 + GHeII) - q3;
        o.zU[2] = P.cz[1] * nHeI;
        o.zU[3] = fma(P.cz[2], nHeII, -o.zU[2]);
    }
    }
}

// Gaussian elimination with partial pivoting for two right-hand sides (step (i), eq. step_ia).
// Pivots are compared by the magnitude's upper 32 bits on the integer pipe.
template <int NM>
__device__ __forceinline__ void lu_solve2(double (&A)[NM][NM], double (&y)[NM], double (&z)[NM]) {
    double inv[NM];
    auto mag = [](double v) { return __double2hiint(v) & 0x7fffffff; };
#pragma unroll
    for (int k = 0; k < NM; ++k) {
        int p = k;
        int best = mag(A[k][k]);
#pragma unroll
        for (int r = k + 1; r < NM; ++r) {
            const int v = mag(A[r][k]);
            if (v > best) { best = v; p = r; }
        }
#pragma unroll
        for (int r = k + 1; r < NM; ++r) {
            if (r == p) {
#pragma unroll
                for (int c = k; c < NM; ++c) { const double t = A[k][c]; A[k][c] = A[r][c]; A[r][c] = t; }
                double t = y[k]; y[k] = y[r]; y[r] = t;
                t = z[k]; z[k] = z[r]; z[r] = t;
            }
        }
        inv[k] = fast_rcp(A[k][k]);
#pragma unroll
        for (int r = k + 1; r < NM; ++r) {
            const double m = A[r][k] * inv[k];
#pragma unroll
            for (int c = k + 1; c < NM; ++c) A[r][c] -= m * A[k][c];
            y[r] -= m * y[k];
            z[r] -= m * z[k];
        }
    }
#pragma unroll
    for (int k = NM - 1; k >= 0; --k) {
        double sy = y[k], sz = z[k];
#pragma unroll
        for (int c = k + 1; c < NM; ++c) { sy -= A[k][c] * y[c]; sz -= A[k][c] * z[c]; }
        y[k] = sy * inv[k];
        z[k] = sz * inv[k];
    }
}

// ---------------------------------------------------------------------------------------------
// fused residual / Jacobian / Schur kernel
//
// MODE_PREP:         U = (0, n^n, E^n); writes g^n = U^n + dt (theta - 1) L(U^n), f(U^n),
//                    and the Schur system at U^n.
// MODE_ITER:         U given; reads g; writes f(U) and the Schur system at U.
// MODE_PREP_PREDICT: writes g^n and the explicit predictor U^n - dt L(U^n) (capped).
// MODE_RESID:        U given; reads g; writes f(U) only (the same arithmetic as MODE_ITER).

// FLUX (limiter_jacobian 1, 2): B.W holds the face fluxes, and the Schur diagonal's face entries
// are left to k_schur_assemble; else B.W holds the coefficients.

template <int NS, int MODE, bool FLUX>
__global__ void __launch_bounds__(CELL_BLOCK) k_cell(const StepParams P, const PhysBuffers B) {
    constexpr int NM = NS + 1, NV = NS + 2;
    const long long c = blockIdx.x * (long long)CELL_BLOCK + threadIdx.x;
    const long long N = P.N;
    double fsq = 0.0;
    if (c < N) {
        int i, j, k;
        cell_coords(P, c, i, j, k);
        const Nbr nb = neighbours(P, c, i, j, k);
        const bool prep = (MODE != MODE_ITER && MODE != MODE_RESID);
        constexpr bool JAC = MODE != MODE_PREP_PREDICT && MODE != MODE_RESID;
        const double* En = prep ? B.E_n : B.E;
        const double* nn = prep ? B.n_n : B.n;
        const double E = En[c];
        double n[NS > 0 ? NS : 1];
#pragma unroll
        for (int s = 0; s < NS; ++s) n[s] = nn[s * N + c];
        const double ec = (prep || B.ec == nullptr) ? 0.0 : B.ec[c];
        const double eh = B.eh[c], nH = B.nH[c], src = B.src[c];
        const double Tfix = P.isothermal ? B.Tiso[c] : 0.0;

        // diffusion, times dt theta: sum over faces W (E_c - E_nb); face part of the diagonal
        double Dterm = 0.0, Wsum = 0.0;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            const double wlo = B.W[ax * N + c];
            const double whi = nb.has_hi[ax] ? B.W[ax * N + nb.hi[ax]] : 0.0;
            if constexpr (FLUX) {
                Dterm += wlo - whi;
            } else {
                Dterm += wlo * (E - En[nb.lo[ax]]) + whi * (E - En[nb.hi[ax]]);
                Wsum += wlo + whi;
            }
        }
        // Dirichlet faces of boundary cells (they carry no entry in the face arrays)
        double kb_term = 0.0;
        if (P.dir_mask) {
            const int q[3] = {i, j, k};
            const int ext[3] = {P.nx, P.ny, P.nz};
            // the cell's opacity at this iterate (the same sum as k_kappa)
            double kc;
            if constexpr (NS == 0) {
                kc = P.kappa_total;
            } else {
                double sk = P.sk[0] * n[0];
                if constexpr (NS == 3) sk += P.sk[1] * n[1] + P.sk[2] * n[2];
                kc = P.ia3 * sk;
            }
#pragma unroll
            for (int d = 0; d < 6; ++d) {
                const int ax = d >> 1;
                if ((P.dir_mask >> d & 1) && q[ax] == ((d & 1) ? ext[ax] - 1 : 0)) {
                    const double Eb = P.Eb[d];
                    const BoundaryFace bf = boundary_face(P, E, Eb, kc);
                    Dterm += bf.W * (E - Eb);
                    Wsum += FLUX ? bf.Qd : bf.W;
                    kb_term += bf.dWdk * (E - Eb);
                }
            }
        }

        Local<NS> lo;
        local_model<NS, JAC>(P, ec, n, E, eh, nH, src, Tfix, lo);
        double Lf[NV];                                      // dt theta L(U)
#pragma unroll
        for (int v = 0; v <= NS; ++v) Lf[v] = lo.L[v];
        Lf[NV - 1] = Dterm + lo.LE;
        double U[NV];
        U[0] = ec;
#pragma unroll
        for (int s = 0; s < NS; ++s) U[1 + s] = n[s];
        U[NV - 1] = E;
        double g[NV];
        if (prep) {
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                g[v] = fma(P.dtm1_dth, Lf[v], U[v]);
                B.g[v * N + c] = g[v];
            }
        } else {
#pragma unroll
            for (int v = 0; v < NV; ++v) g[v] = B.g[v * N + c];
        }

        if (MODE == MODE_PREP_PREDICT || (MODE == MODE_PREP && B.U0)) {
            // explicit Euler predictor U^n - dt L(U^n) (eq. explicit_predictor), positivity cap;
            // MODE_PREP writes it when the step estimates its error against it (Sec. 3.2.3)
            double d[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) d[v] = -P.dt_dth * Lf[v];
            double cap = 1.0;
            auto bound = [&](double q, double dq, double tiny) {
                if (dq < 0.0) cap = fmin(cap, fmax(P.tau * (q + tiny) / (-dq), 0.0));
            };
            bound(eh + ec, d[0], 0.0);
            bound(E, d[NV - 1], 0.0);
            if constexpr (NS >= 1) {
                bound(n[0], d[1], 1e-13 * nH);
                bound(nH - n[0], -d[1], 1e-13 * nH);
            }
            if constexpr (NS == 3) {
                const double nHe = P.y_he * nH;
                bound(n[1], d[2], 1e-13 * nHe);
                bound(n[2], d[3], 1e-13 * nHe);
                bound(nHe - n[1] - n[2], -d[2] - d[3], 1e-13 * nHe);
            }
#pragma unroll
            for (int v = 0; v < NV; ++v) B.U0[v * N + c] = U[v] + cap * d[v];
        }
        if (MODE != MODE_PREP_PREDICT) {
            // scaled residual (eq. nonlinear_residual / eq. scalings)
            double fs[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const double f = (U[v] + Lf[v]) - g[v];
                fs[v] = f * (v == NV - 1 ? P.iu_E : (v == 0 ? P.iu_e : P.iu_n));
                fsq += fs[v] * fs[v];
                if (B.f_out) B.f_out[v * N + c] = fs[v];
            }
            if constexpr (MODE != MODE_RESID) {
            double y[NM], z[NM];
#pragma unroll
            for (int r = 0; r < NM; ++r) { y[r] = fs[r]; z[r] = lo.zU[r]; }
            lu_solve2<NM>(lo.M, y, z);                      // y = M^-1 f_M, z = M^-1 U
            // L M^-1 (U, f_M): L's entries are dt theta (c E + the Dirichlet faces' term of the
            // exact matrix, whose opacity is the cell's) d kappa / d n
            double LMU, LMf;
            if constexpr (NS == 0) {
                LMU = lo.LrE * z[0];
                LMf = lo.LrE * y[0];
            } else {
                double rho = P.ksk[0] * z[1], phi = P.ksk[0] * y[1];
                if constexpr (NS == 3) {
                    rho = fma(P.ksk[1], z[2], fma(P.ksk[2], z[3], rho));
                    phi = fma(P.ksk[1], y[2], fma(P.ksk[2], y[3], phi));
                }
                double cE = P.cdth * E;
                if (P.limiter_newton == 2) cE += kb_term;
                LMU = cE * rho;
                LMf = cE * phi;
                if (FLUX && B.rho) {
                    B.rho[c] = rho;
                    B.phi[c] = phi;
                }
            }
            double dg = (1.0 + lo.dLEE) - LMU;
            for (int go = !FLUX || P.dir_mask; go; go = opaque(0)) dg += Wsum;
            B.diag[c] = dg;
            B.rhs[c] = LMf - fs[NV - 1];
#pragma unroll
            for (int r = 0; r < NM; ++r) {
                B.fMt[r * N + c] = y[r];
                B.MiU[r * N + c] = z[r];
            }
            }
        }
    }
    if (MODE != MODE_PREP_PREDICT) {
        double s, unused;
        if (grid_sum<CELL_BLOCK, false>(fsq, 0.0, B.partials, B.count, s, unused) && threadIdx.x == 0)
            *B.norm_sq = s;
    }
}

template <int NS, bool FLUX>
static void launch_cell_mode(const StepParams& P, int mode, const PhysBuffers& B, int nblocks,
                             cudaStream_t st) {
    const dim3 g(nblocks), b(CELL_BLOCK);
    if (mode == MODE_PREP) k_cell<NS, MODE_PREP, FLUX><<<g, b, 0, st>>>(P, B);
    else if (mode == MODE_ITER) k_cell<NS, MODE_ITER, FLUX><<<g, b, 0, st>>>(P, B);
    else if (mode == MODE_RESID) k_cell<NS, MODE_RESID, FLUX><<<g, b, 0, st>>>(P, B);
    else k_cell<NS, MODE_PREP_PREDICT, FLUX><<<g, b, 0, st>>>(P, B);
}

cudaError_t launch_cell(const StepParams& P, int ns, int mode, const PhysBuffers& B,
                        int nblocks, cudaStream_t st) {
    if (ns == 0) {
        if (B.flux) launch_cell_mode<0, true>(P, mode, B, nblocks, st);
        else launch_cell_mode<0, false>(P, mode, B, nblocks, st);
    } else if (ns == 1) {
        if (B.flux) launch_cell_mode<1, true>(P, mode, B, nblocks, st);
        else launch_cell_mode<1, false>(P, mode, B, nblocks, st);
    } else {
        if (B.flux) launch_cell_mode<3, true>(P, mode, B, nblocks, st);
        else launch_cell_mode<3, false>(P, mode, B, nblocks, st);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Newton update: step (iii) recovery, positivity cap, line-search fraction, new opacity.
// The cap keeps every bounded quantity q (e, E: bound 0; species: bound -1e-13 of the element
// total) above its bound by (1 - tau) of its current distance q + tiny.
//
// Bound by the FP64 pipe.  A cell has a bound in force only where tau (q + tiny) < -dq for one of
// its quantities, which few cells do, so all cells form tau (q + tiny) (one FMA each; of x and
// total - x only the decreasing one) and compare bit patterns on the integer pipe, and only
// the cells with a bound in force take the smallest fraction.  Measured over the launches
// of four 256^3 steps, H + He: 1.35 ms each against 2.27 ms with every bound in FP64.

// the smallest fraction min(1, tau (q + tiny) / (-dq)) over the quantities with a bound in force;
// warps without one go around, and non-negative numbers compare as integers
struct CapFraction {
    double num = 1.0, den = 1.0;
    __device__ __forceinline__ void bound(bool force, double tau, double q, double dq, double tiny) {
        for (int go = force; go; go = opaque(0)) {
            const long long vb = __double_as_longlong(tau * (q + tiny));
            const double v = (vb >= 0 && vb <= 0x7FF0000000000000LL) ? __longlong_as_double(vb) : 0.0;
            const long long lhs = __double_as_longlong(v * den), rhs = __double_as_longlong(num * -dq);
            if (lhs < rhs && rhs <= 0x7FF0000000000000LL) { num = v; den = -dq; }
        }
    }
};

template <int NS>
__global__ void __launch_bounds__(256) k_update(const StepParams P, double lam,
                                                const double* __restrict__ ec0,
                                                const double* __restrict__ n0,
                                                const double* __restrict__ E0,
                                                const double* __restrict__ eh,
                                                const double* __restrict__ nHa,
                                                const double* __restrict__ sE,
                                                const double* __restrict__ fMt,
                                                const double* __restrict__ MiU,
                                                double* __restrict__ ec1, double* __restrict__ n1,
                                                double* __restrict__ E1,
                                                double* __restrict__ kap1) {
    constexpr int NM = NS + 1;
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long N = P.N;
    if (c >= N) return;
    const double se = sE[c];
    double s[NM];
#pragma unroll
    for (int r = 0; r < NM; ++r) s[r] = fma(MiU[r * N + c], se, fMt[r * N + c]) * (r == 0 ? -P.u_e : -P.u_n);
    const double sEp = se * P.u_E;
    const double ec = ec0 ? ec0[c] : 0.0;
    double n[NS > 0 ? NS : 1];
#pragma unroll
    for (int j = 0; j < NS; ++j) n[j] = n0[j * N + c];
    const double E = E0[c], nH = nHa[c], e = eh[c] + ec;
    // v >= 0 and v >= -dq where dq has its sign bit set, on the bit patterns (a negative v, or a
    // dq that is not a number, counts as a bound in force)
    auto in_force = [](double dq, double v) {
        const long long d = __double_as_longlong(dq);
        return d < 0 && __double_as_longlong(v) < (d & 0x7FFFFFFFFFFFFFFFLL);
    };
    const bool fe = in_force(s[0], P.tau * e), fE = in_force(sEp, P.tau * E);
    bool fx = false, f1 = false, f2 = false, f3 = false;
    double qx = 0.0, nHe = 0.0, nHeIII = 0.0, sIII = 0.0;
    if constexpr (NS >= 1) {
        // x decreases or total - x does, by the same amount
        qx = __double_as_longlong(s[1]) < 0 ? n[0] : nH - n[0];
        fx = in_force(-fabs(s[1]), fma(P.tau, qx, P.tau_tiny * nH));
    }
    if constexpr (NS == 3) {
        nHe = P.y_he * nH;
        nHeIII = nHe - n[1] - n[2];
        sIII = -(s[2] + s[3]);
        const double tiny = P.tau_tiny * nHe;
        f1 = in_force(s[2], fma(P.tau, n[1], tiny));
        f2 = in_force(s[3], fma(P.tau, n[2], tiny));
        f3 = in_force(sIII, fma(P.tau, nHeIII, tiny));
    }
    double fr = lam;
    for (int go = fe || fE || fx || f1 || f2 || f3; go; go = opaque(0)) {
        CapFraction cap;
        cap.bound(fe, P.tau, e, s[0], 0.0);
        cap.bound(fE, P.tau, E, sEp, 0.0);
        if constexpr (NS >= 1) cap.bound(fx, P.tau, qx, -fabs(s[1]), 1e-13 * nH);
        if constexpr (NS == 3) {
            cap.bound(f1, P.tau, n[1], s[2], 1e-13 * nHe);
            cap.bound(f2, P.tau, n[2], s[3], 1e-13 * nHe);
            cap.bound(f3, P.tau, nHeIII, sIII, 1e-13 * nHe);
        }
        const double f = cap.num / cap.den;
        fr = __double_as_longlong(f) < __double_as_longlong(lam) ? f : lam;
    }
    ec1[c] = fma(fr, s[0], ec);
    double ksum = 0.0;
#pragma unroll
    for (int j = 0; j < NS; ++j) {
        const double v = fma(fr, s[1 + j], n[j]);
        n1[j * N + c] = v;
        ksum = j == 0 ? P.sk[0] * v : fma(P.sk[j], v, ksum);
    }
    E1[c] = fma(fr, sEp, E);
    kap1[c] = NS == 0 ? P.kappa_total : P.ia3 * ksum;
}

cudaError_t launch_update(const StepParams& P, int ns, double lam, const double* ec0,
                          const double* n0, const double* E0, const double* eh,
                          const double* nH, const double* sE, const double* fMt,
                          const double* MiU, double* ec1, double* n1, double* E1,
                          double* kap1, cudaStream_t st) {
    const int b = 256;
    const unsigned g = (unsigned)((P.N + b - 1) / b);
    if (ns == 0)
        k_update<0><<<g, b, 0, st>>>(P, lam, ec0, n0, E0, eh, nH, sE, fMt, MiU, ec1, n1, E1, kap1);
    else if (ns == 1)
        k_update<1><<<g, b, 0, st>>>(P, lam, ec0, n0, E0, eh, nH, sE, fMt, MiU, ec1, n1, E1, kap1);
    else
        k_update<3><<<g, b, 0, st>>>(P, lam, ec0, n0, E0, eh, nH, sE, fMt, MiU, ec1, n1, E1, kap1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// small state kernels

__global__ void k_finalize(long long N, const double* __restrict__ ec, double* __restrict__ eh) {
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c < N) eh[c] += ec[c];           // e^{n+1} = e_h + e_c (Sec. 3.1)
}

cudaError_t launch_finalize(const StepParams& P, int, const double* ec, double* eh,
                            cudaStream_t st) {
    const int b = 256;
    k_finalize<<<(unsigned)((P.N + b - 1) / b), b, 0, st>>>(P.N, ec, eh);
    return cudaGetLastError();
}

__global__ void k_temperature(const StepParams P, int ns, const double* __restrict__ e,
                              const double* __restrict__ n, const double* __restrict__ nHa,
                              double* __restrict__ T) {
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c >= P.N) return;
    if (ns == 0) { T[c] = P.lte_cT * e[c]; return; }          // LTE
    const double nH = nHa[c], nHe = P.y_he * nH;
    const double nHI = n[c];
    const double nHeI = ns == 3 ? n[P.N + c] : 0.0, nHeII = ns == 3 ? n[2 * P.N + c] : 0.0;
    const double ne = (nH - nHI) + nHeII + 2.0 * (nHe - nHeI - nHeII);
    const double rho = M_H * (nH + 4.0 * nHe);
    T[c] = (GAMMA - 1.0) * rho * e[c] / (K_BOLTZ * (nH + nHe + ne));
}

cudaError_t launch_temperature(const StepParams& P, int ns, const double* e, const double* n,
                               const double* nH, double* T, cudaStream_t st) {
    const int b = 256;
    k_temperature<<<(unsigned)((P.N + b - 1) / b), b, 0, st>>>(P, ns, e, n, nH, T);
    return cudaGetLastError();
}

__global__ void k_check_state(const StepParams P, int ns, const double* __restrict__ E,
                              const double* __restrict__ e, const double* __restrict__ n,
                              const double* __restrict__ nHa, int* bad) {
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c >= P.N) return;
    const double nH = nHa[c], nHe = P.y_he * nH;
    const double nHI = ns >= 1 ? n[c] : 0.0;
    const double nHeI = ns == 3 ? n[P.N + c] : 0.0, nHeII = ns == 3 ? n[2 * P.N + c] : 0.0;
    const bool ok = (E[c] > 0.0) && (e[c] > 0.0) && (nH > 0.0) && (nHI >= 0.0) &&
                    (nH - nHI >= 0.0) && (nHeI >= 0.0) && (nHeII >= 0.0) &&
                    (nHe - nHeI - nHeII >= 0.0) && isfinite(E[c]) && isfinite(e[c]) &&
                    isfinite(nH);
    if (!ok) atomicOr(bad, 1);
}

cudaError_t launch_check_state(const StepParams& P, int ns, const double* E, const double* e,
                               const double* n, const double* nH, int* bad, cudaStream_t st) {
    const int b = 256;
    k_check_state<<<(unsigned)((P.N + b - 1) / b), b, 0, st>>>(P, ns, E, e, n, nH, bad);
    return cudaGetLastError();
}

// Point sources, a batch per launch (one block, a thread per source; the batch rides in the kernel's
// parameters).  Several sources in one cell are added by the first of them, in their order.
__global__ void __launch_bounds__(SOURCE_BATCH) k_deposit(const SourceBatch S, double* src) {
    const int t = (int)threadIdx.x;
    if (t >= S.n) return;
    const long long c = S.cell[t];
    for (int q = 0; q < t; ++q)
        if (S.cell[q] == c) return;
    double v = src[c];
    for (int q = t; q < S.n; ++q)
        if (S.cell[q] == c) v += S.value[q];
    src[c] = v;
}

cudaError_t launch_deposit(const SourceBatch& S, double* src, cudaStream_t st) {
    k_deposit<<<1, SOURCE_BATCH, 0, st>>>(S, src);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Local error estimate of the step against the explicit predictor (eqs. typical_values,
// time_error_estimator): per scaled unknown q = |a - b| / (sqrt|a b| + 1); block partials of
// sum q^p, or of max q when p < 0 (the max norm)

template <int NS>
__global__ void __launch_bounds__(256) k_time_error(const StepParams P, const double* __restrict__ ec,
                                                    const double* __restrict__ n,
                                                    const double* __restrict__ E,
                                                    const double* __restrict__ Up, double pn,
                                                    double* __restrict__ partials) {
    constexpr int NV = NS + 2;
    const long long N = P.N;
    double acc = 0.0;
    for (long long c = blockIdx.x * 256LL + threadIdx.x; c < N; c += (long long)gridDim.x * 256) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const double iu = v == 0 ? P.iu_e : (v == NV - 1 ? P.iu_E : P.iu_n);
            const double a = (v == 0 ? (ec ? ec[c] : 0.0) : (v == NV - 1 ? E[c] : n[(v - 1) * N + c])) * iu;
            const double b = Up[v * N + c] * iu;
            const double q = fabs(a - b) / (sqrt(fabs(a * b)) + 1.0);
            if (pn < 0.0) acc = fmax(acc, q);
            else acc += (pn == 1.0) ? q : (pn == 2.0 ? q * q : pow(q, pn));
        }
    }
    // block reduction (sum or max) in a fixed order
    __shared__ double part[8];
    if (pn < 0.0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc = fmax(acc, __shfl_down_sync(0xffffffffu, acc, o));
    } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    }
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = part[0];
        for (int w = 1; w < 8; ++w) s = pn < 0.0 ? fmax(s, part[w]) : s + part[w];
        partials[blockIdx.x] = s;
    }
}

cudaError_t launch_time_error(const StepParams& P, int ns, const double* ec, const double* n,
                              const double* E, const double* Up, double pn, double* partials,
                              int nblocks, cudaStream_t st) {
    if (ns == 0) k_time_error<0><<<nblocks, 256, 0, st>>>(P, ec, n, E, Up, pn, partials);
    else if (ns == 1) k_time_error<1><<<nblocks, 256, 0, st>>>(P, ec, n, E, Up, pn, partials);
    else k_time_error<3><<<nblocks, 256, 0, st>>>(P, ec, n, E, Up, pn, partials);
    return cudaGetLastError();
}

}  // namespace rhi
