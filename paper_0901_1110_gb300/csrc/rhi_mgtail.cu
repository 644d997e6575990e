// The coarse end of a multigrid V-cycle in one launch.
//
// Below about 40^3 cells a level's kernel is shorter than the gap between two launches: a V-cycle of
// a 32^3 grid is 20 launches of 3 to 4 us each whatever they compute.  Here one thread-block
// cluster runs the whole cycle from a level of few enough cells down to the coarsest and back.
// Its barriers are the hardware's cluster barrier, so nothing spins.
//
//  * The cells of a "wide" level are split into one contiguous chunk per block; x (two buffers) and b
//    of a chunk live in the block's shared memory, and neighbours in other chunks are read
//    through distributed shared memory.  A barrier follows each sweep.
//  * A level of at most NARROW cells runs in block 0 alone, where __syncthreads is the barrier (the
//    coarsest level's 16 sweeps above all).  FP64 sweeps are bound by the FP64 pipe (two
//    instructions a clock per SM), so their narrow levels are smaller.
//  * A thread keeps its cells' couplings and the addresses of their neighbours in registers: those of
//    the first level (CELLS per thread) for the whole cycle, those of the others (one per
//    thread) while it works on the level.  They are fetched one level ahead, because a cluster barrier
//    also empties L1 and every fetch goes to L2.
//
// Measured: a whole cycle of a 32^3 FP32 grid (4 levels) 24.6 us, against about 75 us for its 20
// launches inside a CUDA graph; a 16^3 FP64 cycle (5 levels) 34.8 us against about 90 us.  What is left is
// latency: about 0.4 us for each of about twelve cluster barriers (5 of the 25 us; the rest is not attributed),
// and in FP64 64 cycles for each instruction of a warp.
// Larger levels stay with the level kernels, which use all SMs: at 64^3 FP32 a sweep moves 10 MB.
//
// Where the whole cycle is one such launch, BiCGStab's p is updated as it is read (given): a launch and
// the gap before it less per iteration, 37.3 -> 36.7 ms for 377 iterations on 32^3.
//
// The arithmetic of a sweep, the residual, the restriction (sum of the children's residuals / 8) and
// the injection is that of the level kernels in rhi_linear.cu.  Sweeps alternate between the two
// buffers with a barrier between, so no buffer is written while it is read.
#include <cooperative_groups.h>

#include "rhi_linear.cuh"

namespace cg = cooperative_groups;

namespace rhi {

namespace {

// a block holds THREADS x CELLS cells of the first level and THREADS of each other
template <typename T> struct TailTraits;
template <> struct TailTraits<float> { static constexpr int THREADS = 512, CELLS = 4, NARROW = 512; };
template <> struct TailTraits<double> { static constexpr int THREADS = 512, CELLS = 1, NARROW = 128; };

constexpr int TAIL_CLUSTER = 16;

template <typename T>
struct TailLevel {
    int nx, ny, nz, N;
    FastDiv fd_nx, fd_nxy, fd_chunk;
    int chunk;               // cells per block (narrow: N, all in block 0)
    int buf[2], b;           // offsets in shared memory, in elements
    const T *diag, *wid, *W[3], *Wp[3];
};

template <typename T>
struct TailArgs {
    TailLevel<T> lv[MG_TAIL_LEVELS];
    int n, wide;             // levels; the first `wide` of them are split over the blocks
    int per[3];
    int pre, post, coarse;
    T om1;                   // 1 - omega
    const T* b;              // right-hand side of the first level, in T or (b64) FP64
    const double* b64;
    T* x;                    // result in T (may be null) and FP64 (may be null)
    double* x64;
    const double* skip;
    BicgP up;                // with up.scal, the right-hand side is the p this launch updates
};

// shared memory of a block of the cluster by its address in the cluster's window (the block's own too:
// one instruction, no branch, so that a thread's loads are in flight together)
__device__ __forceinline__ float ld_tail(unsigned a, float) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ double ld_tail(unsigned a, double) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}

// one cell of a level as its owner keeps it in registers
template <typename T>
struct TailCell {
    T w[6];                  // couplings to the six neighbours (0 where there is none)
    unsigned a[6];           // their x in buffer 0, in the cluster's window
    T wid, b, x;
    bool on;                 // the thread has such a cell
};

// A thread's work on its one cell of a level stays a branch (opaque): warps without a cell go around it.
#define TAIL_CELL(on) for (int go_ = (on) ? 1 : 0; go_; go_ = M == 1 ? opaque(0) : 0)

template <typename T>
struct TailBlock {
    static constexpr int THREADS = TailTraits<T>::THREADS;
    const TailArgs<T>& A;
    const TailLevel<T>* lv;  // in shared memory: indexed by level, which kernel parameters serve slowly
    T* sm;
    unsigned me, base;       // rank; address of sm as of ld.shared

    // where value q of the array at element offset `at` of level v sits
    __device__ __forceinline__ unsigned where(const TailLevel<T>& v, int at, int q) const {
        const unsigned r = fdiv((unsigned)q, v.fd_chunk);
        const unsigned a = base + (unsigned)(at + (q - (int)r * v.chunk)) * (unsigned)sizeof(T);
        unsigned m;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(m) : "r"(a), "r"(r));
        return m;
    }
    __device__ __forceinline__ static void coords(const TailLevel<T>& v, int c, int& i, int& j, int& k) {
        k = (int)fdiv((unsigned)c, v.fd_nxy);
        const int r = c - k * v.nx * v.ny;
        j = (int)fdiv((unsigned)r, v.fd_nx);
        i = r - j * v.nx;
    }
    // cell u of this thread in the chunk
    __device__ __forceinline__ static int at(int u) { return (int)threadIdx.x + u * THREADS; }
    __device__ __forceinline__ int cell(const TailLevel<T>& v, int u) const { return (int)me * v.chunk + at(u); }

    // fetches this thread's cells of level v (couplings, omega / diagonal, neighbours' addresses)
    template <int M>
    __device__ __forceinline__ void cells(const TailLevel<T>& v, TailCell<T> (&r)[M]) const {
        const int c0 = (int)me * v.chunk, c1 = min(c0 + v.chunk, v.N);
        const int n[3] = {v.nx, v.ny, v.nz}, s[3] = {1, v.nx, v.nx * v.ny};
#pragma unroll
        for (int u = 0; u < M; ++u) {
            const int c = c0 + at(u);
            r[u].on = c < c1;
            if (!r[u].on) continue;
            int q[3];
            coords(v, c, q[0], q[1], q[2]);
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) {
                const bool lo = q[ax] > 0 || A.per[ax], hi = q[ax] < n[ax] - 1 || A.per[ax];
                const int cl = q[ax] > 0 ? c - s[ax] : (lo ? c + (n[ax] - 1) * s[ax] : c);
                const int ch = q[ax] < n[ax] - 1 ? c + s[ax] : (hi ? c - (n[ax] - 1) * s[ax] : c);
                r[u].w[2 * ax] = lo ? __ldg(v.W[ax] + c) : T(0);
                r[u].w[2 * ax + 1] = hi ? __ldg(v.Wp[ax] + ch) : T(0);
                r[u].a[2 * ax] = where(v, v.buf[0], cl);
                r[u].a[2 * ax + 1] = where(v, v.buf[0], ch);
            }
            r[u].wid = __ldg(v.wid + c);
        }
    }
    // b plus the sum over the six neighbours of coupling times x, of the buffer `d` bytes above the first
    __device__ __forceinline__ static void neighbours(unsigned d, const TailCell<T>& r, T (&x)[6]) {
#pragma unroll
        for (int f = 0; f < 6; ++f) x[f] = ld_tail(r.a[f] + d, T(0));
    }
    __device__ __forceinline__ static T row(const TailCell<T>& r, const T (&x)[6]) {
        T acc = r.b;
#pragma unroll
        for (int f = 0; f < 6; ++f) acc += r.w[f] * x[f];
        return acc;
    }
    __device__ __forceinline__ static void sync(bool wide) {
        if (wide) cg::this_cluster().sync();
        else __syncthreads();
    }
    // The first level's right-hand side: given, or BiCGStab's p, updated here (k_bicg_p's formulas; the
    // thread that owns a cell is the only one to read or write its p).
    template <int M>
    __device__ __forceinline__ void given(TailCell<T> (&r)[M]) const {
        const BicgP& P = A.up;
        if (!P.scal) {
#pragma unroll
            for (int u = 0; u < M; ++u)
                if (r[u].on) {
                    const int c = cell(lv[0], u);
                    r[u].b = A.b64 ? (T)A.b64[c] : A.b[c];
                }
            return;
        }
        const double beta = P.scal[S_BETA], omega = P.scal[S_OMEGA];
        const bool restart = P.scal[S_RST] != 0.0;
        const bool first = P.scal[S_ITS] == 0.0 || restart;
        double rv[M], pv[M], vv[M];
#pragma unroll
        for (int u = 0; u < M; ++u)
            if (r[u].on) {
                const int c = cell(lv[0], u);
                rv[u] = P.r[c];
                if (!first) {
                    pv[u] = P.p[c];
                    vv[u] = P.v[c];
                }
            }
#pragma unroll
        for (int u = 0; u < M; ++u)
            TAIL_CELL(r[u].on) {
                const int c = cell(lv[0], u);
                const double p = first ? rv[u] : fma(beta, fma(-omega, vv[u], pv[u]), rv[u]);
                P.p[c] = p;
                if (restart) P.rh[c] = rv[u];
                r[u].b = (T)p;
            }
    }
    // right-hand side of a coarse cell: the children's residuals, which sit in buffer `rb` of the level above
    __device__ __forceinline__ T rhs(int l, int rb, int c) const {
        const TailLevel<T>& f = lv[l - 1];
        int I, J, K;
        coords(lv[l], c, I, J, K);
        T x[8];
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            const int i = 2 * I + (d & 1), j = 2 * J + ((d >> 1) & 1), k = 2 * K + (d >> 2);
            const bool in = i < f.nx && j < f.ny && k < f.nz;
            // (a missing child reads the first one)
            const int q = in ? i + f.nx * (j + f.ny * k) : 2 * I + f.nx * (2 * J + f.ny * 2 * K);
            const T val = ld_tail(where(f, f.buf[rb], q), T(0));
            x[d] = in ? val : T(0);
        }
        T b = T(0);
#pragma unroll
        for (int d = 0; d < 8; ++d) b += x[d];
        return b * T(0.125);
    }
    // one weighted-Jacobi sweep of level v from buffer `in` into the other
    template <int M>
    __device__ __forceinline__ void sweep(const TailLevel<T>& v, int in, TailCell<T> (&r)[M]) const {
        T* dst = sm + (in ? v.buf[0] : v.buf[1]);
        const unsigned d = in ? (unsigned)v.chunk * (unsigned)sizeof(T) : 0u;
        T x[M][6];
#pragma unroll
        for (int u = 0; u < M; ++u)
            if (M > 1 && r[u].on) neighbours(d, r[u], x[u]);      // all cells' loads in flight
#pragma unroll
        for (int u = 0; u < M; ++u)
            TAIL_CELL(r[u].on) {
                if (M == 1) neighbours(d, r[u], x[u]);
                r[u].x = A.om1 * r[u].x + r[u].wid * row(r[u], x[u]);
                dst[at(u)] = r[u].x;
            }
    }
    // Down the level: right-hand side, first sweep from x = 0 into buffer 0, further sweeps and, above
    // the coarsest level, the residual into the buffer they leave free.  r: fetched cells
    template <int M>
    __device__ __forceinline__ void down(int l, bool w, int sweeps, bool last, int rb, TailCell<T> (&r)[M]) const {
        const TailLevel<T>& v = lv[l];
        T dg[M];
        if (l == 0) given(r);
#pragma unroll
        for (int u = 0; u < M; ++u)
            TAIL_CELL(r[u].on) {
                if (l > 0) r[u].b = rhs(l, rb, cell(v, u));
                if (!last) dg[u] = __ldg(v.diag + cell(v, u));
                r[u].x = r[u].wid * r[u].b;
                if (M == 1) sm[v.b + at(u)] = r[u].b;       // (the first level's b stays in its registers)
                sm[v.buf[0] + at(u)] = r[u].x;
            }
        for (int s = 1; s < sweeps; ++s) {
            sync(w);
            sweep(v, (s - 1) & 1, r);
        }
        sync(w);
        if (last) return;
        const int in = (sweeps - 1) & 1;
        T* dst = sm + (in ? v.buf[0] : v.buf[1]);
        const unsigned d = in ? (unsigned)v.chunk * (unsigned)sizeof(T) : 0u;
#pragma unroll
        for (int u = 0; u < M; ++u)
            TAIL_CELL(r[u].on) {
                T x[6];
                neighbours(d, r[u], x);
                dst[at(u)] = row(r[u], x) - dg[u] * r[u].x;
            }
        sync(w);
    }
    // Up: the coarse correction (buffer `cin` of the level below) and the post-sweeps, from buffer
    // `in`; returns the buffer that holds x.  b and x of a level other than the first are read back
    template <int M>
    __device__ __forceinline__ int up(int l, bool w, int in, int cin, bool keep, TailCell<T> (&r)[M]) const {
        const TailLevel<T>& v = lv[l];
        const TailLevel<T>& f = lv[l + 1];
#pragma unroll
        for (int u = 0; u < M; ++u)
            TAIL_CELL(r[u].on) {
                int i, j, k;
                coords(v, cell(v, u), i, j, k);
                const T pc = ld_tail(where(f, f.buf[cin], (i >> 1) + f.nx * ((j >> 1) + f.ny * (k >> 1))), T(0));
                if (!keep) {
                    r[u].b = sm[v.b + at(u)];
                    r[u].x = sm[(in ? v.buf[1] : v.buf[0]) + at(u)];
                }
                r[u].x += pc;
                sm[(in ? v.buf[1] : v.buf[0]) + at(u)] = r[u].x;
            }
        for (int s = 0; s < A.post; ++s, in ^= 1) {
            sync(w);
            sweep(v, in, r);
        }
        if (l > 0) sync(w);
        return in;
    }
};

// the buffer that holds x of a level after its first sweep and s - 1 more
__device__ __forceinline__ int after(int sweeps) { return (sweeps - 1) & 1; }

template <typename T>
__global__ void __launch_bounds__(TailTraits<T>::THREADS) k_mg_tail(const __grid_constant__ TailArgs<T> A) {
    if (A.skip && *A.skip != 0.0) return;             // every block reads the same flag
    extern __shared__ __align__(16) unsigned char tail_smem[];
    __shared__ TailLevel<T> lv[MG_TAIL_LEVELS];
    const cg::cluster_group cl = cg::this_cluster();
    const TailBlock<T> B{A, lv, reinterpret_cast<T*>(tail_smem), cl.block_rank(),
                         static_cast<unsigned>(__cvta_generic_to_shared(tail_smem))};
    const int n = A.n, wide = A.wide, pre = after(A.pre);
    for (unsigned q = threadIdx.x; q < n * (unsigned)(sizeof(TailLevel<T>) / 4); q += TailTraits<T>::THREADS)
        reinterpret_cast<unsigned*>(lv)[q] = reinterpret_cast<const unsigned*>(A.lv)[q];
    __syncthreads();
    // levels this block works on: the wide ones, and in block 0 all
    const int mine = B.me == 0 ? n : wide;
    TailCell<T> r0[TailTraits<T>::CELLS];             // the first level, for the whole cycle
    TailCell<T> r1[1], rn[1];                         // another level, and the next one on the way
    if (mine > 0) B.cells(lv[0], r0);
    if (mine > 1) B.cells(lv[1], r1);
    // (a block reads another's memory only after a barrier of all, so after all have started)
    // down
    if (mine > 0) B.down(0, wide > 0, n == 1 ? A.coarse : A.pre, n == 1, 0, r0);
    for (int l = 1; l < mine; ++l) {
        if (l + 1 < mine) B.cells(lv[l + 1], rn);
        B.down(l, l < wide, l == n - 1 ? A.coarse : A.pre, l == n - 1, pre ^ 1, r1);
        if (l + 1 < mine) r1[0] = rn[0];
    }
    // up: x of every level above the coarsest is in buffer `pre`; its post-sweeps alternate
    const int done = (pre + A.post) & 1;
    int top = min(mine, n - 1) - 1;                   // first level of this block's way up
    if (top > 0) B.cells(lv[top], r1);
    for (int l = top; l > 0; --l) {
        if (l > 1) B.cells(lv[l - 1], rn);
        if (l + 1 == wide && wide < n) cl.sync();     // the narrow levels are done
        B.up(l, l < wide, pre, l + 1 == n - 1 ? after(A.coarse) : done, false, r1);
        if (l > 1) r1[0] = rn[0];
    }
    if (n > 1 && mine > 0) {
        if (wide == 1) cl.sync();
        B.up(0, wide > 0, pre, n == 2 ? after(A.coarse) : done, true, r0);
    }
    // no block leaves while its memory may be read: all have arrived here, their last reads done
    if (wide > 0) cl.barrier_arrive();
    if (mine > 0) {
#pragma unroll
        for (int u = 0; u < TailTraits<T>::CELLS; ++u)
            if (r0[u].on) {
                const int c = B.cell(lv[0], u);
                if (A.x) A.x[c] = r0[u].x;
                if (A.x64) A.x64[c] = (double)r0[u].x;
            }
    }
    if (wide > 0) cl.barrier_wait();
}

// blocks of the cluster on the current device: 16 where such a cluster (a non-portable size) fits,
// else 8
template <typename T>
cudaError_t tail_init(int* blocks) {
    cudaError_t e = cudaFuncSetAttribute(k_mg_tail<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         MG_TAIL_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_mg_tail<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = TAIL_CLUSTER;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(TAIL_CLUSTER);
    cfg.blockDim = dim3(TailTraits<T>::THREADS);
    cfg.dynamicSmemBytes = MG_TAIL_SMEM;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int clusters = 0;
    e = cudaOccupancyMaxActiveClusters(&clusters, k_mg_tail<T>, &cfg);
    if (e != cudaSuccess) { cudaGetLastError(); clusters = 0; }
    *blocks = clusters >= 1 ? TAIL_CLUSTER : 8;
    return cudaSuccess;
}

}  // namespace

cudaError_t mg_tail_init(int* blocks32, int* blocks64) {
    cudaError_t e = tail_init<float>(blocks32);
    if (e == cudaSuccess) e = tail_init<double>(blocks64);
    return e;
}

// Sizes: a block's THREADS x CELLS cells of the first level; below it one cell per thread
template <typename T>
bool mg_tail_fits(long long N, long long N_next, int blocks) {
    return N <= (long long)TailTraits<T>::THREADS * TailTraits<T>::CELLS * blocks &&
           N_next <= (long long)TailTraits<T>::THREADS * blocks;
}
template bool mg_tail_fits<float>(long long, long long, int);
template bool mg_tail_fits<double>(long long, long long, int);

template <typename T>
cudaError_t LinLaunch::mg_tail(const MgTail<T>& M) {
    TailArgs<T> A{};
    const int blocks = M.blocks;
    A.n = M.n;
    size_t at = 0;
    for (int l = 0; l < M.n; ++l) {
        const Op<T>& o = M.op[l];
        TailLevel<T>& v = A.lv[l];
        v.nx = o.nx; v.ny = o.ny; v.nz = o.nz; v.N = (int)o.N;
        v.fd_nx = o.fd_nx; v.fd_nxy = o.fd_nxy;
        const bool wide = o.N > TailTraits<T>::NARROW;
        if (wide) A.wide = l + 1;
        v.chunk = wide ? (v.N + blocks - 1) / blocks : v.N;
        v.fd_chunk = make_fastdiv((unsigned)v.chunk);
        v.buf[0] = (int)at;
        v.buf[1] = (int)(at + v.chunk);
        v.b = (int)(at + 2 * (size_t)v.chunk);
        at += 3 * (size_t)v.chunk;
        v.diag = o.diag; v.wid = o.wid;
        for (int a = 0; a < 3; ++a) { v.W[a] = o.W[a]; v.Wp[a] = o.Wp[a]; A.per[a] = o.per[a]; }
    }
    if (at * sizeof(T) > (size_t)MG_TAIL_SMEM) return cudaErrorInvalidValue;
    A.pre = M.pre; A.post = M.post; A.coarse = M.coarse;
    A.om1 = T(1) - M.omega;
    A.up = M.up;
    A.b = M.b; A.b64 = M.b64; A.x = M.x; A.x64 = M.x64;
    A.skip = skip;
    begin(sizeof(T) == 4 ? "mg_tail_f32" : "mg_tail_f64");
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = blocks;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(TailTraits<T>::THREADS);
    cfg.dynamicSmemBytes = at * sizeof(T);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_mg_tail<T>, A);
    const cudaError_t e2 = end();
    return e != cudaSuccess ? e : e2;
}

template cudaError_t LinLaunch::mg_tail<float>(const MgTail<float>&);
template cudaError_t LinLaunch::mg_tail<double>(const MgTail<double>&);

}  // namespace rhi
