// Learned Newton initial guess (an addition to the paper's method, whose Sec. 3.2 leaves the
// initial iterate free and whose Sec. 3.2.4 uses an explicit predictor): a per-cell MLP
// 13 -> 64 -> 64 -> 64 -> 6 with SiLU that predicts the state at t^{n+1} from the state at
// t^n and the change of the previous step.
//
//   features  log10 E/u_E, log10 e/u_e, log10 x_HI, log10 x_HeI, log10 x_HeII, log10 n_H/u_n,
//             log10(dt Gamma_HI + 1e-30), log10(1 + 4 pi eta dt / E), log10(dt / 1e12 s),
//             log10 E/E^{n-1}, log10 e/e^{n-1}, logit x_HI - logit x_HI^{n-1},
//             log10(dt / dt^{n-1}) (the last four 0 before a first step)
//   outputs   log10 E'/E, log10 e'/e, logit x_HI', He fraction logits (softmax)
//
// Inference runs on the tensor cores (mma.sync m16n8k16, BF16 operands, FP32 accumulation)
// with the layer activations chained in registers; training runs FP32 on the CUDA cores, tiles of
// 32 samples per block, with a deterministic gradient reduction and Adam.
#include <cmath>
#include <cstddef>

#include "rhi_mlp.cuh"

namespace rhi {

namespace {

constexpr int INF_WARPS = 4;                  // warps per inference block
constexpr int TRAIN_BLOCK = 256;

// ------------------------------------------------------------------------------------------
// features of one cell (FP32 from the FP64 state)

__device__ __forceinline__ float log10_clamped(double x) {
    // FP32 logarithm of a positive ratio formed in FP64, clamped into the FP32 range
    return log10f(fminf(fmaxf((float)x, 1e-37f), 1e37f));
}

__device__ __forceinline__ void cell_features(const MlpArgs& A, long long c, float (&f)[MLP_IN]) {
    // ratios in FP64 (the source ratio and the field leave the FP32 range in cells the
    // radiation has not reached), logarithms in FP32
    const double E = A.E[c], e = A.e[c], nH = A.nH[c];
    const double inH = 1.0 / nH;
    f[0] = log10_clamped(E * A.iu_E);
    f[1] = log10_clamped(e * A.iu_e);
    f[2] = log10_clamped(fmax(A.n[c] * inH, 1e-30));
    if (A.ns == 3) {
        const double inHe = inH / A.y_he;
        f[3] = log10_clamped(fmax(A.n[A.N + c] * inHe, 1e-30));
        f[4] = log10_clamped(fmax(A.n[2 * A.N + c] * inHe, 1e-30));
    } else {
        f[3] = 0.0f;
        f[4] = 0.0f;
    }
    f[5] = log10_clamped(nH * A.iu_n);
    f[6] = log10_clamped(A.dt * A.gam_per_E * E + 1e-30);
    f[7] = log10f(1.0f + fminf((float)(A.src[c] * A.dt / E), 1e37f));
    f[8] = log10_clamped(A.dt * 1e-12);
    if (A.E_p) {
        // the previous step's change: ratios in FP64, the logit difference in FP64 (neutral
        // cells sit within 1e-16 of x_HI = 1), rounded to FP32.  One logarithm of the quotient (at most
        // 1e46 either way) instead of four: an FP64 logarithm is some 30 instructions of the FP64
        // pipe, which bounds this kernel, and the sum of four rounded worse (2e-14 against 7e-15)
        f[9] = log10_clamped(E / A.E_p[c]);
        f[10] = log10_clamped(e / A.e_p[c]);
        const double x1 = fmin(fmax(A.n[c] * inH, 1e-30), 1.0 - 1e-16);
        const double x0 = fmin(fmax(A.n_p[c] * inH, 1e-30), 1.0 - 1e-16);
        f[11] = (float)log((x1 * (1.0 - x0)) / ((1.0 - x1) * x0));
        f[12] = A.ldt_ratio;
    } else {
        f[9] = f[10] = f[11] = f[12] = 0.0f;
    }
}

__global__ void k_mlp_features(const MlpArgs A, float* __restrict__ X) {
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c >= A.N) return;
    float f[MLP_IN];
    cell_features(A, c, f);
#pragma unroll
    for (int q = 0; q < MLP_IN; ++q) X[c * MLP_IN + q] = f[q];
}

// targets of the step (E0, e0, n0) -> (E, e, n) of MlpArgs
__global__ void k_mlp_targets(const MlpArgs A, const double* __restrict__ E0,
                              const double* __restrict__ e0, const double* __restrict__ n0,
                              float* __restrict__ Y) {
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c >= A.N) return;
    float* y = Y + c * MLP_OUT;
    y[0] = (float)log10(A.E[c] / E0[c]);
    y[1] = (float)log10(A.e[c] / e0[c]);
    const double nH = A.nH[c];
    const double x = fmin(fmax(A.n[c] / nH, 1e-30), 1.0 - 1e-16);
    y[2] = (float)(log(x) - log1p(-x));
    if (A.ns == 3) {
        const double nHe = A.y_he * nH;
        const double f0 = A.n[A.N + c] / nHe, f1 = A.n[2 * A.N + c] / nHe;
        const double l0 = log(fmax(f0, 1e-30)), l1 = log(fmax(f1, 1e-30));
        const double l2 = log(fmax(1.0 - f0 - f1, 1e-30));
        const double m = (l0 + l1 + l2) / 3.0;
        y[3] = (float)(l0 - m);
        y[4] = (float)(l1 - m);
        y[5] = (float)(l2 - m);
    } else {
        y[3] = y[4] = y[5] = 0.0f;
    }
}

// ------------------------------------------------------------------------------------------
// tensor-core inference

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// one hidden layer on a 16-row tile: in = A fragments over KS k-steps, out = 8 n-tiles
template <int KS, int RS>
__device__ __forceinline__ void hidden_layer(const uint32_t (&a)[4][4], const __nv_bfloat16* W,
                                             const float* b, float (&acc)[8][4], int g, int t) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float b0 = b[8 * j + 2 * t], b1 = b[8 * j + 2 * t + 1];
        acc[j][0] = b0; acc[j][1] = b1; acc[j][2] = b0; acc[j][3] = b1;
#pragma unroll
        for (int s = 0; s < KS; ++s) {
            const uint2 w = *reinterpret_cast<const uint2*>(W + (8 * j + g) * RS + 16 * s + 4 * t);
            mma_bf16(acc[j], a[s], w.x, w.y);
        }
    }
}

// SiLU of 8 n-tiles into the A fragments of the next layer's 4 k-steps
template <bool FAST>
__device__ __forceinline__ void to_fragments(const float (&acc)[8][4], uint32_t (&a)[4][4]) {
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        a[s][0] = pack_bf16(silu_f<FAST>(acc[2 * s][0]), silu_f<FAST>(acc[2 * s][1]));
        a[s][1] = pack_bf16(silu_f<FAST>(acc[2 * s][2]), silu_f<FAST>(acc[2 * s][3]));
        a[s][2] = pack_bf16(silu_f<FAST>(acc[2 * s + 1][0]), silu_f<FAST>(acc[2 * s + 1][1]));
        a[s][3] = pack_bf16(silu_f<FAST>(acc[2 * s + 1][2]), silu_f<FAST>(acc[2 * s + 1][3]));
    }
}

// MODE 0: outputs for given features X (n rows) into Y;  MODE 1: guess for every cell of the
// state (features computed here), decoded into the work iterate (e_c, n, E) and its opacity
template <int MODE>
__global__ void __launch_bounds__(32 * INF_WARPS) k_mlp_infer(const MlpArgs A,
                                                              const MlpPacked* __restrict__ pk,
                                                              const float* __restrict__ X,
                                                              float* __restrict__ Y,
                                                              long long n_rows) {
    __shared__ __align__(16) MlpPacked sw;
    __shared__ __nv_bfloat16 xs[INF_WARPS][32][24];
    __shared__ float os[INF_WARPS][32][8];
    // stage the packed weights
    {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(pk);
        uint32_t* dst = reinterpret_cast<uint32_t*>(&sw);
        for (int q = threadIdx.x; q < (int)(sizeof(MlpPacked) / 4); q += blockDim.x) dst[q] = src[q];
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const long long rows = (MODE == 0) ? n_rows : A.N;
    const long long ntiles = (rows + 31) / 32;
    for (long long tile = blockIdx.x * (long long)INF_WARPS + warp; tile < ntiles;
         tile += (long long)gridDim.x * INF_WARPS) {
        const long long c = tile * 32 + lane;
        float f[MLP_IN];
        if (c < rows) {
            if (MODE == 0) {
#pragma unroll
                for (int q = 0; q < MLP_IN; ++q) f[q] = X[c * MLP_IN + q];
            } else {
                cell_features(A, c, f);
            }
        } else {
#pragma unroll
            for (int q = 0; q < MLP_IN; ++q) f[q] = sw.mean[q];
        }
        bool ood = false;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const float xn = q < MLP_IN ? (f[q] - sw.mean[q]) * sw.iscale[q] : 0.0f;
            ood |= A.ood > 0.0f && fabsf(xn) > A.ood;
            xs[warp][lane][q] = __float2bfloat16_rn(xn);
        }
        __syncwarp();
        // (not unrolled, like the two middle layers: the code then fits the instruction cache, whose misses
        // were a third of the stalls)
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
            const int r0 = 16 * half + g;
            uint32_t a[4][4];
            a[0][0] = *reinterpret_cast<const uint32_t*>(&xs[warp][r0][2 * t]);
            a[0][1] = *reinterpret_cast<const uint32_t*>(&xs[warp][r0 + 8][2 * t]);
            a[0][2] = *reinterpret_cast<const uint32_t*>(&xs[warp][r0][2 * t + 8]);
            a[0][3] = *reinterpret_cast<const uint32_t*>(&xs[warp][r0 + 8][2 * t + 8]);
            float acc[8][4];
            hidden_layer<1, RS1>(a, sw.W1, sw.b1, acc, g, t);
            to_fragments<MODE == 0>(acc, a);
#pragma unroll 1
            for (int layer = 0; layer < 2; ++layer) {
                hidden_layer<4, RS2>(a, layer ? sw.W3 : sw.W2, layer ? sw.b3 : sw.b2, acc, g, t);
                to_fragments<MODE == 0>(acc, a);
            }
            float o[4] = {sw.b4[2 * t], sw.b4[2 * t + 1], sw.b4[2 * t], sw.b4[2 * t + 1]};
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const uint2 w = *reinterpret_cast<const uint2*>(sw.W4 + g * RS2 + 16 * s + 4 * t);
                mma_bf16(o, a[s], w.x, w.y);
            }
            os[warp][r0][2 * t] = o[0];
            os[warp][r0][2 * t + 1] = o[1];
            os[warp][r0 + 8][2 * t] = o[2];
            os[warp][r0 + 8][2 * t + 1] = o[3];
        }
        __syncwarp();
        if (c < rows) {
            const float* o = os[warp][lane];
            if (MODE == 0) {
#pragma unroll
                for (int q = 0; q < MLP_OUT; ++q) Y[c * MLP_OUT + q] = o[q];
            } else {
                // decode (FP32 transcendentals; the logit of the old fraction in FP64, where
                // neutral cells sit within 1e-16 of 1); cells whose predicted change stays
                // below the gate, or whose inputs left the training range, keep U^n
                const double E0 = A.E[c], e0 = A.e[c], nH = A.nH[c];
                const double x0 = fmin(fmax(A.n[c] / nH, 1e-30), 1.0 - 1e-16);
                float change = fmaxf(fabsf(o[0]), fabsf(o[1]));
                change = fmaxf(change, fabsf(o[2] - (float)log(x0 / (1.0 - x0))));
                const double xHI = 1.0 / (1.0 + (double)expf(-o[2]));
                double nHeI = 0.0, nHeII = 0.0;
                if (A.ns == 3) {
                    // softmax normalised in FP64: n_HeI + n_HeII stays below n_He to rounding,
                    // so the derived n_HeIII of the guess is not negative beyond the positivity
                    // cap's tolerance (an FP32 sum can overshoot by 1e-7 n_He and freeze the cell)
                    const double nHe = A.y_he * nH;
                    const float mx = fmaxf(o[3], fmaxf(o[4], o[5]));
                    const double z0 = expf(o[3] - mx), z1 = expf(o[4] - mx), z2 = expf(o[5] - mx);
                    const double iz = 1.0 / (z0 + z1 + z2);
                    const double f0 = A.n[A.N + c] / nHe, f1 = A.n[2 * A.N + c] / nHe;
                    const double f2 = 1.0 - f0 - f1;
                    change = fmaxf(change, fabsf(logf((float)fmax(z0 * iz, 1e-30)) - logf((float)fmax(f0, 1e-30))));
                    change = fmaxf(change, fabsf(logf((float)fmax(z1 * iz, 1e-30)) - logf((float)fmax(f1, 1e-30))));
                    change = fmaxf(change, fabsf(logf((float)fmax(z2 * iz, 1e-30)) - logf((float)fmax(f2, 1e-30))));
                    nHeI = nHe * (z0 * iz);
                    nHeII = nHe * (z1 * iz);
                }
                const long long N = A.N;
                double* U = A.U0;
                if (change < A.gate || ood) {
                    U[c] = 0.0;
                    for (int s = 0; s < A.ns; ++s) U[(1 + s) * N + c] = A.n[s * N + c];
                    U[(1 + A.ns) * N + c] = E0;
                } else {
                    U[c] = A.isothermal ? 0.0 : e0 * (double)expm1f(2.302585093f * o[1]);
                    U[N + c] = nH * xHI;
                    if (A.ns == 3) {
                        U[2 * N + c] = nHeI;
                        U[3 * N + c] = nHeII;
                    }
                    U[(1 + A.ns) * N + c] = E0 * (double)exp10f(o[0]);
                }
            }
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------------------------------
// FP32 training

struct TrainW {
    float W1[MLP_HID * MLP_IN], b1[MLP_HID];
    float W2[MLP_HID * MLP_HID], b2[MLP_HID];
    float W3[MLP_HID * MLP_HID], b3[MLP_HID];
    float W4[MLP_OUT * MLP_HID], b4[MLP_OUT];
    float mean[MLP_IN], scale[MLP_IN];
};
static_assert(sizeof(TrainW) == RHI_MLP_NWEIGHTS * sizeof(float), "weight layout");
// offsets in the weight vector
constexpr int OW1 = 0, OB1 = OW1 + MLP_HID * MLP_IN, OW2 = OB1 + MLP_HID,
              OB2 = OW2 + MLP_HID * MLP_HID, OW3 = OB2 + MLP_HID, OB3 = OW3 + MLP_HID * MLP_HID,
              OW4 = OB3 + MLP_HID, OB4 = OW4 + MLP_OUT * MLP_HID, NTRAIN = OB4 + MLP_OUT;

__device__ __forceinline__ float sig_f(float z) { return 1.0f / (1.0f + expf(-z)); }

// Forward, backward and weight gradient of tiles of 32 samples, one tile at a time per block of 256
// threads, all in shared memory: the weights (rows padded to 68 floats, so that the eight rows a
// warp reads at once fall into different banks), the activations and their derivatives, [sample]
// [feature].  Each matrix product is a 64 x 32 (layers) or 64 x 64 (weight gradients) tile in FP32
// FMAs, 4 x 2 or 4 x 4 results per thread from 16-byte loads.  A block adds the gradients of its
// tiles in registers and writes them once; k_mlp_apply adds the blocks' in order, so a result does
// not depend on timing.
//
// Bound by shared-memory loads (four wavefronts per 16-byte load of a warp).  A minibatch of 4096
// samples: 40 us with its update, against 450 us for one thread per sample with its activations in local memory and a
// gradient pass that walked the samples in one chain per weight.
constexpr int TT = 32;                         // samples per tile
constexpr int PS = MLP_HID + 4;                // padded row
constexpr int PS0 = MLP_IN + 3;                // padded input row (16 floats)
struct TrainSmem {
    float W1[MLP_HID * PS0], W2[MLP_HID * PS], W3[MLP_HID * PS], W4[MLP_OUT * PS];
    float b1[MLP_HID], b2[MLP_HID], b3[MLP_HID], b4[8];
    float mean[16], scale[16];                                      // (MLP_IN of each)
    float h0[TT * PS0], h1[TT * PS], h2[TT * PS], h3[TT * PS];      // activations
    float p1[TT * PS], p2[TT * PS], p3[TT * PS];                    // SiLU', then the deltas
    float g4[TT * 8];
};
// every row that is read or written in 16-byte pieces starts on a 16-byte boundary
static_assert(PS % 4 == 0 && PS0 % 4 == 0 && PS0 >= MLP_IN, "row padding");
static_assert(offsetof(TrainSmem, W1) % 16 == 0 && offsetof(TrainSmem, W2) % 16 == 0 &&
              offsetof(TrainSmem, W3) % 16 == 0 && offsetof(TrainSmem, W4) % 16 == 0 &&
              offsetof(TrainSmem, h0) % 16 == 0 && offsetof(TrainSmem, h1) % 16 == 0 &&
              offsetof(TrainSmem, h2) % 16 == 0 && offsetof(TrainSmem, h3) % 16 == 0 &&
              offsetof(TrainSmem, p1) % 16 == 0 && offsetof(TrainSmem, p2) % 16 == 0 &&
              offsetof(TrainSmem, p3) % 16 == 0, "alignment of the tiles");

// acc[4][2] = rows n0.. of W (64 x K, row stride S) times samples s0, s0 + 1 (row stride S)
template <int K, int S>
__device__ __forceinline__ void tile_fwd(const float* W, const float* h, int n0, int s0, float (&acc)[4][2]) {
#pragma unroll 4
    for (int k = 0; k < K; k += 4) {
        float4 w[4], x[2];
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] = *reinterpret_cast<const float4*>(W + (n0 + q) * S + k);
#pragma unroll
        for (int q = 0; q < 2; ++q) x[q] = *reinterpret_cast<const float4*>(h + (s0 + q) * S + k);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                acc[q][t] = fmaf(w[q].x, x[t].x, acc[q][t]);
                acc[q][t] = fmaf(w[q].y, x[t].y, acc[q][t]);
                acc[q][t] = fmaf(w[q].z, x[t].z, acc[q][t]);
                acc[q][t] = fmaf(w[q].w, x[t].w, acc[q][t]);
            }
    }
}
// SiLU and its derivative of a tile's pre-activations
__device__ __forceinline__ void tile_act(const float (&acc)[4][2], int n0, int s0, float* h, float* p) {
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        float4 hv, pv;
        float* hq = &hv.x;
        float* pq = &pv.x;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float z = acc[q][t], sg = sig_f(z);
            hq[q] = z * sg;
            pq[q] = sg * (1.0f + z * (1.0f - sg));
        }
        *reinterpret_cast<float4*>(h + (s0 + t) * PS + n0) = hv;
        *reinterpret_cast<float4*>(p + (s0 + t) * PS + n0) = pv;
    }
}
// deltas of the layer below: p (SiLU') *= W^T d, columns k0.. of W (64 x 64), samples s0, s0 + 1
__device__ __forceinline__ void tile_bwd(const float* W, const float* d, int k0, int s0, float* p) {
    float acc[2][4] = {};
#pragma unroll 4
    for (int n = 0; n < MLP_HID; n += 4) {
        float4 x[2];
#pragma unroll
        for (int t = 0; t < 2; ++t) x[t] = *reinterpret_cast<const float4*>(d + (s0 + t) * PS + n);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 w = *reinterpret_cast<const float4*>(W + (n + q) * PS + k0);
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const float dv = q == 0 ? x[t].x : (q == 1 ? x[t].y : (q == 2 ? x[t].z : x[t].w));
                acc[t][0] = fmaf(w.x, dv, acc[t][0]);
                acc[t][1] = fmaf(w.y, dv, acc[t][1]);
                acc[t][2] = fmaf(w.z, dv, acc[t][2]);
                acc[t][3] = fmaf(w.w, dv, acc[t][3]);
            }
        }
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        float4* pp = reinterpret_cast<float4*>(p + (s0 + t) * PS + k0);
        float4 v = *pp;
        v.x *= acc[t][0]; v.y *= acc[t][1]; v.z *= acc[t][2]; v.w *= acc[t][3];
        *pp = v;
    }
}
// weight gradient rows n0.., columns k0.. += sum over the tile's samples of d_n h_k
__device__ __forceinline__ void tile_grad(const float* d, const float* h, int n0, int k0, float (&g)[4][4]) {
#pragma unroll 4
    for (int s = 0; s < TT; ++s) {
        const float4 a = *reinterpret_cast<const float4*>(d + s * PS + n0);
        const float4 x = *reinterpret_cast<const float4*>(h + s * PS + k0);
        const float av[4] = {a.x, a.y, a.z, a.w}, xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int t = 0; t < 4; ++t) g[q][t] = fmaf(av[q], xv[t], g[q][t]);
    }
}

__global__ void __launch_bounds__(TRAIN_BLOCK) k_mlp_train(const float* __restrict__ w,
                                                           const float* __restrict__ X,
                                                           const float* __restrict__ Y,
                                                           long long m, float inv_norm,
                                                           float* __restrict__ gpart,
                                                           double* __restrict__ partials) {
    extern __shared__ __align__(16) unsigned char train_smem[];
    TrainSmem& S = *reinterpret_cast<TrainSmem*>(train_smem);
    const int tid = (int)threadIdx.x;
    for (int q = tid; q < MLP_HID * MLP_HID; q += TRAIN_BLOCK) {
        const int n = q >> 6, k = q & 63;
        S.W2[n * PS + k] = w[OW2 + q];
        S.W3[n * PS + k] = w[OW3 + q];
        if (n < MLP_OUT) S.W4[n * PS + k] = w[OW4 + q];
    }
    for (int q = tid; q < MLP_HID * PS0; q += TRAIN_BLOCK) {
        const int n = q / PS0, k = q % PS0;
        S.W1[q] = k < MLP_IN ? w[OW1 + n * MLP_IN + k] : 0.0f;
    }
    if (tid < MLP_HID) {
        S.b1[tid] = w[OB1 + tid];
        S.b2[tid] = w[OB2 + tid];
        S.b3[tid] = w[OB3 + tid];
        if (tid < MLP_OUT) S.b4[tid] = w[OB4 + tid];
        if (tid < MLP_IN) { S.mean[tid] = w[NTRAIN + tid]; S.scale[tid] = w[NTRAIN + MLP_IN + tid]; }
    }
    // layer tiles: 16 groups of 4 neurons x 16 pairs of samples, 8 x 4 of them per warp; gradient tiles:
    // 16 x 16 groups of 4 x 4
    const int lane = tid & 31, warp = tid >> 5;
    const int n0 = 4 * ((lane & 7) + 8 * (warp & 1)), s0 = 2 * ((lane >> 3) + 4 * (warp >> 1));
    const int gn = 4 * (tid >> 4), gk = 4 * (tid & 15);
    float g2[4][4] = {}, g3[4][4] = {}, g1[4] = {}, gw4[2] = {}, gb = 0.0f, gb4 = 0.0f;
    double se = 0.0;
    const long long tiles = (m + TT - 1) / TT;
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const long long base = tile * TT;
        const int cnt = (int)(m - base < TT ? m - base : TT);
        __syncthreads();                                    // the last tile's arrays are free
        for (int q = tid; q < TT * PS0; q += TRAIN_BLOCK) {
            const int s = q / PS0, k = q % PS0;
            float v = 0.0f;
            if (k < MLP_IN && s < cnt) v = (X[(base + s) * MLP_IN + k] - S.mean[k]) / S.scale[k];
            S.h0[q] = v;
        }
        __syncthreads();
        float acc[4][2];
        auto bias = [&](const float* b) {
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q][0] = acc[q][1] = b[n0 + q];
        };
        bias(S.b1);
        tile_fwd<PS0, PS0>(S.W1, S.h0, n0, s0, acc);
        tile_act(acc, n0, s0, S.h1, S.p1);
        __syncthreads();
        bias(S.b2);
        tile_fwd<MLP_HID, PS>(S.W2, S.h1, n0, s0, acc);
        tile_act(acc, n0, s0, S.h2, S.p2);
        __syncthreads();
        bias(S.b3);
        tile_fwd<MLP_HID, PS>(S.W3, S.h2, n0, s0, acc);
        tile_act(acc, n0, s0, S.h3, S.p3);
        __syncthreads();
        // outputs: thread (sample, n); the delta of a sample beyond the last is 0
        {
            const int s = tid >> 3, n = tid & 7;
            float gv = 0.0f;
            if (n < MLP_OUT && s < cnt) {
                float a = S.b4[n];
#pragma unroll 4
                for (int k = 0; k < MLP_HID; k += 4) {
                    const float4 wv = *reinterpret_cast<const float4*>(S.W4 + n * PS + k);
                    const float4 hv = *reinterpret_cast<const float4*>(S.h3 + s * PS + k);
                    a = fmaf(wv.x, hv.x, a);
                    a = fmaf(wv.y, hv.y, a);
                    a = fmaf(wv.z, hv.z, a);
                    a = fmaf(wv.w, hv.w, a);
                }
                const float d = a - Y[(base + s) * MLP_OUT + n];
                se += (double)d * d;
                gv = 2.0f * d * inv_norm;
            }
            S.g4[s * 8 + n] = gv;
        }
        __syncthreads();
        // deltas d3 (in p3), then d2, d1
        for (int q = tid; q < TT * MLP_HID; q += TRAIN_BLOCK) {
            const int s = q >> 6, k = q & 63;
            float a = 0.0f;
#pragma unroll
            for (int n = 0; n < MLP_OUT; ++n) a = fmaf(S.W4[n * PS + k], S.g4[s * 8 + n], a);
            S.p3[s * PS + k] *= a;
        }
        __syncthreads();
        tile_bwd(S.W3, S.p3, n0, s0, S.p2);
        __syncthreads();
        tile_bwd(S.W2, S.p2, n0, s0, S.p1);
        __syncthreads();
        // gradients: W3 and W2 tiles, W1 (thread: neuron, 4 inputs), W4 (384 entries) and the biases
        tile_grad(S.p3, S.h2, gn, gk, g3);
        tile_grad(S.p2, S.h1, gn, gk, g2);
        {
            const int n = tid >> 2, k = 4 * (tid & 3);
#pragma unroll 4
            for (int s = 0; s < TT; ++s) {
                const float d = S.p1[s * PS + n];
                const float4 x = *reinterpret_cast<const float4*>(S.h0 + s * PS0 + k);
                g1[0] = fmaf(d, x.x, g1[0]);
                g1[1] = fmaf(d, x.y, g1[1]);
                g1[2] = fmaf(d, x.z, g1[2]);
                g1[3] = fmaf(d, x.w, g1[3]);
            }
            const int k4 = tid & 63, n4 = tid >> 6;          // W4: rows n4 and, for n4 < 2, n4 + 4
#pragma unroll 4
            for (int s = 0; s < TT; ++s) {
                const float hv = S.h3[s * PS + k4];
                gw4[0] = fmaf(S.g4[s * 8 + n4], hv, gw4[0]);
                if (n4 < 2) gw4[1] = fmaf(S.g4[s * 8 + n4 + 4], hv, gw4[1]);
            }
            // biases: b1, b2, b3 by threads 0-191, b4 by threads 192-197
            const float* d = tid < 64 ? S.p1 : (tid < 128 ? S.p2 : S.p3);
            if (tid < 192) {
#pragma unroll 4
                for (int s = 0; s < TT; ++s) gb += d[s * PS + (tid & 63)];
            } else if (tid < 192 + MLP_OUT) {
#pragma unroll 4
                for (int s = 0; s < TT; ++s) gb4 += S.g4[s * 8 + tid - 192];
            }
        }
    }
    // this block's gradient
    float* g = gpart + (long long)blockIdx.x * NTRAIN;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            g[OW2 + (gn + q) * MLP_HID + gk + t] = g2[q][t];
            g[OW3 + (gn + q) * MLP_HID + gk + t] = g3[q][t];
        }
    {
        const int n = tid >> 2, k = 4 * (tid & 3);
#pragma unroll
        for (int t = 0; t < 4; ++t)
            if (k + t < MLP_IN) g[OW1 + n * MLP_IN + k + t] = g1[t];
        const int k4 = tid & 63, n4 = tid >> 6;
        g[OW4 + n4 * MLP_HID + k4] = gw4[0];
        if (n4 < 2) g[OW4 + (n4 + 4) * MLP_HID + k4] = gw4[1];
        if (tid < 192) g[(tid < 64 ? OB1 : (tid < 128 ? OB2 : OB3)) + (tid & 63)] = gb;
        else if (tid < 192 + MLP_OUT) g[OB4 + tid - 192] = gb4;
    }
    const double bs = block_sum<TRAIN_BLOCK>(se);
    if (tid == 0) partials[blockIdx.x] = bs;
}

// Sum of the blocks' gradients in a fixed order, then the Adam update (ADAM) or the gradient itself.
// 32 weights per block, 8 threads for each.
template <bool ADAM>
__global__ void __launch_bounds__(256) k_mlp_apply(const float* __restrict__ gpart, int nb,
                                                   float* __restrict__ w, float* __restrict__ g,
                                                   float* __restrict__ m1, float* __restrict__ m2,
                                                   float lr, float b1t, float b2t) {
    __shared__ float part[8][32];
    const int q = blockIdx.x * 32 + (threadIdx.x & 31), grp = threadIdx.x >> 5;
    float a = 0.0f;
    if (q < NTRAIN) {
#pragma unroll 4
        for (int b = grp; b < nb; b += 8) a += gpart[(long long)b * NTRAIN + q];
    }
    part[grp][threadIdx.x & 31] = a;
    __syncthreads();
    if (grp != 0 || q >= NTRAIN) return;
    float gv = a;
#pragma unroll
    for (int t = 1; t < 8; ++t) gv += part[t][threadIdx.x];
    if (!ADAM) {
        g[q] = gv;
        return;
    }
    const float b1 = 0.9f, b2 = 0.999f;
    const float u = b1 * m1[q] + (1.0f - b1) * gv;
    const float v = b2 * m2[q] + (1.0f - b2) * gv * gv;
    m1[q] = u;
    m2[q] = v;
    w[q] -= lr * (u / (1.0f - b1t)) / (sqrtf(v / (1.0f - b2t)) + 1e-8f);
}

// FP32 master weights to the padded BF16 inference layout (one block)
__global__ void __launch_bounds__(1024) k_mlp_pack(const float* __restrict__ w, MlpPacked* __restrict__ out) {
    const int tid = (int)threadIdx.x;
    const __nv_bfloat16 zero = __float2bfloat16_rn(0.0f);
    for (int q = tid; q < MLP_HID * RS1; q += 1024) {
        const int n = q / RS1, k = q % RS1;
        out->W1[n * RS1 + packed_k(k)] = k < MLP_IN ? __float2bfloat16_rn(w[OW1 + n * MLP_IN + k]) : zero;
    }
    for (int q = tid; q < MLP_HID * RS2; q += 1024) {
        const int n = q / RS2, k = q % RS2, at = n * RS2 + packed_k(k);
        out->W2[at] = k < MLP_HID ? __float2bfloat16_rn(w[OW2 + n * MLP_HID + k]) : zero;
        out->W3[at] = k < MLP_HID ? __float2bfloat16_rn(w[OW3 + n * MLP_HID + k]) : zero;
        if (n < 8) out->W4[at] = n < MLP_OUT && k < MLP_HID ? __float2bfloat16_rn(w[OW4 + n * MLP_HID + k]) : zero;
    }
    if (tid < MLP_HID) {
        out->b1[tid] = w[OB1 + tid];
        out->b2[tid] = w[OB2 + tid];
        out->b3[tid] = w[OB3 + tid];
    }
    if (tid < 8) out->b4[tid] = tid < MLP_OUT ? w[OB4 + tid] : 0.0f;
    if (tid < MLP_IN) {
        out->mean[tid] = w[NTRAIN + tid];
        out->iscale[tid] = 1.0f / w[NTRAIN + MLP_IN + tid];
    }
}

}  // namespace

// ------------------------------------------------------------------------------------------
// launchers

cudaError_t launch_mlp_features(const MlpArgs& A, float* X, cudaStream_t st) {
    k_mlp_features<<<(unsigned)((A.N + 255) / 256), 256, 0, st>>>(A, X);
    return cudaGetLastError();
}

cudaError_t launch_mlp_targets(const MlpArgs& A, const double* E0, const double* e0,
                               const double* n0, float* Y, cudaStream_t st) {
    k_mlp_targets<<<(unsigned)((A.N + 255) / 256), 256, 0, st>>>(A, E0, e0, n0, Y);
    return cudaGetLastError();
}

cudaError_t launch_mlp_infer(const MlpArgs& A, const MlpPacked* pk, const float* X, float* Y,
                             long long n_rows, int guess, cudaStream_t st) {
    const long long rows = guess ? A.N : n_rows;
    const long long tiles = (rows + 31) / 32;
    long long blocks = (tiles + INF_WARPS - 1) / INF_WARPS;
    // one wave of the 6 blocks an SM holds (their shared memory): with more, the few that start late
    // would take as long as the first ones
    if (blocks > 152LL * 6) blocks = 152LL * 6;
    if (blocks < 1) blocks = 1;
    if (guess) k_mlp_infer<1><<<(unsigned)blocks, 32 * INF_WARPS, 0, st>>>(A, pk, X, Y, n_rows);
    else k_mlp_infer<0><<<(unsigned)blocks, 32 * INF_WARPS, 0, st>>>(A, pk, X, Y, n_rows);
    return cudaGetLastError();
}

// two blocks per SM hold a tile each; more tiles go round
int mlp_train_blocks(long long m) {
    const long long tiles = (m + TT - 1) / TT;
    return (int)(tiles < 304 ? tiles : 304);
}
int mlp_ntrain() { return NTRAIN; }

cudaError_t launch_mlp_train(const float* w, const float* X, const float* Y, long long m, float* gpart,
                             double* partials, cudaStream_t st) {
    const size_t sm = sizeof(TrainSmem);
    cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    k_mlp_train<<<mlp_train_blocks(m), TRAIN_BLOCK, sm, st>>>(w, X, Y, m, 1.0f / (float)(m * MLP_OUT),
                                                            gpart, partials);
    return cudaGetLastError();
}

cudaError_t launch_mlp_grad(const float* gpart, int nb, float* grad, cudaStream_t st) {
    k_mlp_apply<false><<<(NTRAIN + 31) / 32, 256, 0, st>>>(gpart, nb, nullptr, grad, nullptr, nullptr, 0.0f,
                                                          0.0f, 0.0f);
    return cudaGetLastError();
}

cudaError_t launch_mlp_adam(const float* gpart, int nb, float* w, float* m1, float* m2, float lr,
                            float b1t, float b2t, cudaStream_t st) {
    k_mlp_apply<true><<<(NTRAIN + 31) / 32, 256, 0, st>>>(gpart, nb, w, nullptr, m1, m2, lr, b1t, b2t);
    return cudaGetLastError();
}

cudaError_t launch_mlp_pack(const float* w, MlpPacked* out, cudaStream_t st) {
    k_mlp_pack<<<1, 1024, 0, st>>>(w, out);
    return cudaGetLastError();
}

}  // namespace rhi
