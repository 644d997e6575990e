// Allocation-free RMS norm: the block-partial reduction of the residual norm with its scratch
// in a file-scope device array instead of memory from cudaMalloc.
//
// Callers that may not allocate device memory (code running while a CUDA stream is being
// captured into a graph, where cudaMalloc is not allowed, or a host application that owns all
// device memory through its own pool) can still evaluate the convergence measure of a
// residual they hold.  The scratch below is reserved on every GPU that loads the library, for
// the life of the process.
#include <mutex>

#include "rhi_internal.cuh"

namespace {

constexpr int NA_BLOCK = 256;
constexpr int NA_BLOCKS = 152 * 4;             // blocks of a large input, 4 per SM

// one partial sum per block of the first kernel (the result goes to the caller's `out`)
static __device__ __align__(256) double na_scratch[NA_BLOCKS];

// Sum of squares of this block's share: four independent 16-byte loads per thread and turn, then single
// values.  Bound by HBM and the FP64 pipe alike (one FMA per 8 bytes): 2^25 values 72 us, against 478 us
// with one value per thread in 131072 blocks, each of which reduced its 256 values.
__device__ __forceinline__ double na_sum(const double* __restrict__ v, long long n, bool aligned) {
    double a0 = 0.0, a1 = 0.0;
    const long long stride = (long long)gridDim.x * NA_BLOCK;
    const long long i0 = blockIdx.x * (long long)NA_BLOCK + threadIdx.x;
    long long done = 0;
    if (aligned) {
        const double2* v2 = reinterpret_cast<const double2*>(v);
        const long long n2 = n / 2;
        long long i = i0;
        for (; i + 3 * stride < n2; i += 4 * stride) {
            double2 x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = __ldg(v2 + i + q * stride);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                a0 = fma(x[q].x, x[q].x, a0);
                a1 = fma(x[q].y, x[q].y, a1);
            }
        }
        for (; i < n2; i += stride) {
            const double2 x = __ldg(v2 + i);
            a0 = fma(x.x, x.x, a0);
            a1 = fma(x.y, x.y, a1);
        }
        done = 2 * n2;
    }
    for (long long i = done + i0; i < n; i += stride) {
        const double x = __ldg(v + i);
        a0 = fma(x, x, a0);
    }
    return rhi::block_sum<NA_BLOCK>(a0 + a1);
}

__global__ void __launch_bounds__(NA_BLOCK) k_na_partials(const double* __restrict__ v, long long n,
                                                          bool aligned, double* __restrict__ part) {
    const double s = na_sum(v, n, aligned);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

__global__ void __launch_bounds__(NA_BLOCK) k_na_finish(const double* __restrict__ part, int np,
                                                        double inv_count, double* __restrict__ out) {
    double acc = 0.0;
    for (int q = threadIdx.x; q < np; q += NA_BLOCK) acc += part[q];
    const double s = rhi::block_sum<NA_BLOCK>(acc);
    if (threadIdx.x == 0) out[0] = sqrt(s * inv_count);
}

// device address of the scratch, looked up once per device with that device current
constexpr int NA_MAX_DEVICES = 64;
double* na_addr[NA_MAX_DEVICES] = {nullptr};
std::mutex na_mutex;

}  // namespace

extern "C" int rhi_rms_norm_noalloc(const double* v, long long n, long long count,
                                    double* out, void* stream) {
    if (!v || !out || n < 1 || count < 1) return RHI_ERR_ARG;
    if (n > RHI_NOALLOC_MAX_COUNT) return RHI_ERR_ARG;       // the documented limit
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) return RHI_ERR_CUDA;
    double* part = nullptr;
    {
        std::lock_guard<std::mutex> lock(na_mutex);
        if (!na_addr[dev]) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, na_scratch) != cudaSuccess || !p) return RHI_ERR_CUDA;
            na_addr[dev] = (double*)p;
        }
        part = na_addr[dev];
    }
    const cudaStream_t st = (cudaStream_t)stream;
    // four values per thread at least, and no more blocks than fill the GPU, which is what the scratch holds
    const long long want = (n + 4 * NA_BLOCK - 1) / (4 * NA_BLOCK);
    const long long nb = want < NA_BLOCKS ? want : NA_BLOCKS;
    const bool aligned = ((unsigned long long)v & 15ull) == 0;
    // a launch error left pending by earlier work of this host thread is cleared here, so that
    // each launch below is judged on its own status
    (void)cudaGetLastError();
    k_na_partials<<<(unsigned)nb, NA_BLOCK, 0, st>>>(v, n, aligned, part);
    if (cudaGetLastError() != cudaSuccess) return RHI_ERR_CUDA;
    k_na_finish<<<1, NA_BLOCK, 0, st>>>(part, (int)nb, 1.0 / (double)count, out);
    if (cudaGetLastError() != cudaSuccess) return RHI_ERR_CUDA;
    return RHI_OK;
}
