// Allocation-free variant of the diagonal-block step:
// Dinv = L_KK^{-T} D_K^{-1} L_KK^{-1} for one unit-lower diagonal block.
//
// Some callers cannot allocate device memory: code in a latency-critical
// loop (cudaMalloc and cudaFree synchronize the whole device and take an
// unbounded amount of time), code whose device memory is entirely owned by
// another allocator (a framework's caching allocator or a fixed arena sized
// up front), and code running where allocation is not permitted at all
// (inside a host callback).  For them this entry point keeps its scratch --
// the s x s block L_KK^{-1} -- in a file-scope static device array of fixed
// size instead of plan- or caller-allocated memory; the caller still passes
// the input block, D and the output.
#include <cuda_runtime.h>

#include <mutex>

#include "selinv.h"
#include "tri_rows.cuh"

namespace {

using namespace selinv;

constexpr int kMaxS = SELINV_NOALLOC_MAX_S;
constexpr int kMaxDevices = 64;

// L_KK^{-1} of the current call, column-major s x s.  Every GPU that loads
// the library holds this array (kMaxS^2 doubles = 128 KB) until the process
// exits.  All calls share it.
static __device__ __align__(256) double g_linv_scratch[kMaxS * kMaxS];

// Two kernels, both spread over SMs (one CTA walking the block in global
// memory took 1325 us at s = 96).  First the columns of L_KK^{-1}, 8 per CTA
// (they are independent), into the scratch block: every entry is written, so
// nothing needs clearing between calls.
__global__ void __launch_bounds__(kTriThreads) k_noalloc_linv(int s, const double *__restrict__ L, int64_t ld,
                                                              double *__restrict__ X) {
    grid_dep_wait();   // the previous call's k_noalloc_dinv may still read the scratch block
    extern __shared__ __align__(16) double Ls[];
    const int j0 = blockIdx.x * kTriCols;
    tri_store(Ls, L, ld, s, j0 / 32);
    __syncthreads();
    tri_inverse<double, false>(Ls, nullptr, X, s, s, j0);
}

// Then Dinv(i, j) = sum_{k >= max(i, j)} X(k, i) / D_k X(k, j), one 16 x 16 tile
// (i0 >= j0) of the lower triangle per CTA, mirrored: k over 16 lanes at a time.
// The terms are quotients: a product with 1 / D_k rounds twice, and 1 / D_k
// overflows where the quotient does not.  Each sum starts at its own k: a zero
// of X above the diagonal times an infinite or undefined 1 / D_k is no term.
// A quotient is x r + x r', r the rounded reciprocal and r' its residual over D_k:
// one rounding, to within 2^-100 of the product.  Both kernels: 34.8 us at s = 96
// and 51.2 at 128 (with divisions 36.9 and 55.2; products with r alone 32.8 and
// 49.2).  Where a magnitude is near the ends of the range, the CTA divides.
constexpr int kMidLo = 1023 - 400, kMidHi = 1023 + 400;   // biased exponents
__device__ __forceinline__ bool mid(double v) {
    const int e = (int)((__double_as_longlong(v) >> 52) & 0x7FF);
    return e >= kMidLo && e <= kMidHi;
}

__global__ void __launch_bounds__(256) k_noalloc_dinv(int s, const double *__restrict__ X, const double *__restrict__ D,
                                                      double *__restrict__ Dinv, int64_t ldo) {
    grid_dep_wait();
    __shared__ double As[128][17], Bs[128][17], rd[128], rl[128];
    int ti = 0, tj = blockIdx.x;
    while (tj > ti) { tj -= ti + 1; ti++; }
    const int i0 = ti * 16, j0 = tj * 16, n = s - i0;
    bool far = false;
    for (int q = threadIdx.x; q < n; q += 256) {
        const double d = D[i0 + q], r = 1.0 / d;
        far = !mid(d);
        rd[q] = r;
        rl[q] = fma(-d, r, 1.0) * r;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 16 * n; e += 256) {
        const int q = e % n, r = e / n, k = i0 + q;   // k fastest: contiguous in X's columns
        const double x = r <= q ? X[(int64_t)(i0 + r) * s + k] : 0.0;
        far = far || !(mid(x) || x == 0.0);
        As[q][r] = fma(x, rd[q], x * rl[q]);
        Bs[q][r] = j0 + r < s ? X[(int64_t)(j0 + r) * s + k] : 0.0;
    }
    if (__syncthreads_or(far)) {
        for (int e = threadIdx.x; e < 16 * n; e += 256) {
            const int q = e % n, r = e / n, k = i0 + q;
            if (r <= q) As[q][r] = X[(int64_t)(i0 + r) * s + k] / D[k];
        }
        __syncthreads();
    }
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16, i = i0 + ty, j = j0 + tx;
    if (i >= s || i < j) return;
    double acc = 0.0;
    for (int q = ty; q < n; q++) acc = fma(As[q][ty], Bs[q][tx], acc);
    Dinv[(int64_t)j * ldo + i] = acc;
    Dinv[(int64_t)i * ldo + j] = acc;
}

// Device address of g_linv_scratch per device ordinal, looked up once per
// device (in host code the symbol is only a host-side stand-in).  The
// address belongs to the device's primary context: after cudaDeviceReset
// the module is loaded again and the cached address is stale, so a process
// that resets a device must not call this entry point on it afterwards.
std::mutex g_lock;
double *g_addr[kMaxDevices] = {nullptr};

int scratch_address(double **out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return SELINV_ERR_CUDA;
    std::lock_guard<std::mutex> g(g_lock);
    if (!g_addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_linv_scratch) != cudaSuccess || !p) return SELINV_ERR_CUDA;
        // (with the first call's address goes the kernel's shared-memory opt-in)
        if (cudaFuncSetAttribute(k_noalloc_linv, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(double) * tri_store_elems(kMaxS)) != cudaSuccess)
            return SELINV_ERR_CUDA;
        g_addr[dev] = static_cast<double *>(p);
    }
    *out = g_addr[dev];
    return SELINV_OK;
}

}  // namespace

extern "C" int selinv_dinv_noalloc(int32_t s, const double *Lkk, int64_t ld, const double *D,
                                   double *Dinv, int64_t ldo, void *cuda_stream) {
    if (s < 0 || s > kMaxS) return SELINV_ERR_INVALID_ARG;  // beyond the static scratch
    if (s == 0) return SELINV_OK;
    if (!Lkk || !D || !Dinv || ld < s || ldo < s) return SELINV_ERR_INVALID_ARG;
    double *scratch = nullptr;
    int rc = scratch_address(&scratch);
    if (rc) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const int nt = (s + 15) / 16;
    k_noalloc_linv<<<(s + kTriCols - 1) / kTriCols, kTriThreads, sizeof(double) * tri_store_elems(s), st>>>(s, Lkk, ld, scratch);
    k_noalloc_dinv<<<nt * (nt + 1) / 2, 256, 0, st>>>(s, scratch, D, Dinv, ldo);
    return cudaGetLastError() == cudaSuccess ? SELINV_OK : SELINV_ERR_CUDA;
}
