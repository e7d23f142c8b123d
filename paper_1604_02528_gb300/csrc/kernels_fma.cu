// FP64 / complex products of the level schedule for the supernodes that run
// neither on the tensor cores nor in k_selinv_narrow: every supernode of the
// LU form wider than 16 columns, those of the FP64-only options, and narrow
// ones with a long C.  The FP64 pipe bounds them all (2 products per clock and
// SM), so what counts is that every SM has its share: small tiles, both sides
// of the LU form and the diagonal block as items of their own.  (A CTA per 64
// rows of C doing both sides and its part of the diagonal block left all but a
// few SMs idle at the top of the tree: a 22 x 20 x 21 grid's LU form took
// 12.8 ms for products that need 3 ms of the whole chip.)
//
//   k_fma_lhat   Lhat_{C,K} = L_{C,K} L_KK^{-1} (Uhat^T = U_{K,C}^T (U_KK^T)^{-1})
//   k_fma_rows   A^{-1}_{C,K} = -A^{-1}_{C,C} Lhat with the gather (LU: and
//                A^{-1}_{K,C}^T = -A^{-1}(C,C)^T Uhat^T)
//   k_fma_diag   A^{-1}_KK = Dinv_K - Lhat^T A^{-1}_{C,K}, symmetrized (LU:
//                U_KK^{-1} L_KK^{-1} - Uhat A^{-1}_{C,K})
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "launch.h"
#include "tile_gemm.cuh"

namespace selinv {

namespace cg = cooperative_groups;

constexpr int kFmThreads = 128;
constexpr int kFmK = 32;                     // k per stage
static_assert(kFmaCols == 32, "the widest column tile below");

// acc += A(R x 32) B(32 x TN) from shared memory; thread (tx, ty): rows
// tx + 16 i, columns ty + 8 j
template <typename T, int R, int TN>
__device__ __forceinline__ void fma_stage(const T (&As)[kFmK][R + 1], const T (&Bs)[kFmK][TN + 1], int kk,
                                          T (&acc)[R / 16][TN / 8]) {
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
#pragma unroll 4
    for (int k = 0; k < kk; k++) {
        T a[R / 16], b[TN / 8];
#pragma unroll
        for (int i = 0; i < R / 16; i++) a[i] = As[k][tx + 16 * i];
#pragma unroll
        for (int j = 0; j < TN / 8; j++) b[j] = Bs[k][ty + 8 * j];
#pragma unroll
        for (int i = 0; i < R / 16; i++)
#pragma unroll
            for (int j = 0; j < TN / 8; j++) madd(acc[i][j], a[i], b[j]);
    }
}

// items: tile = row tile of R rows, ntiles = (column tile of TN) << 1 | side; a
// cluster shares the rows q of C, the partial sums meeting in its first CTA
// (where a level has a few narrow supernodes with a long C: 34 tiles of
// c = 500 took 123 us)
template <typename T, int R, int TN>
__global__ void __launch_bounds__(kFmThreads) k_fma_rows(const ProbDesc *__restrict__ descs,
                                                         const Item *__restrict__ items, int nitems) {
    grid_dep_wait();
    __shared__ T As[kFmK][R + 1], Bs[kFmK][TN + 1];
    static_assert(kFmK * (R + 1) >= R * TN || kFmK * (TN + 1) >= R * TN, "a tile's sums fit a stage");
    __shared__ int64_t tile_cb[R], tile_rb[R];
    __shared__ int ymax[TN];
    cg::cluster_group cl = cg::this_cluster();
    const int CL = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int w = blockIdx.x / CL;
    if (w >= nitems) return;                 // the grid is nitems clusters: never taken by a part of one
    const Item it = items[w];
    const ProbDesc &P = descs[it.prob];
    const int K = it.K, side = it.ntiles & 1, j0 = (it.ntiles >> 1) * TN, p0 = it.tile * R;
    const int fc = P.super_ptr[K];
    const int s = P.super_ptr[K + 1] - fc;
    const int64_t ld = P.rowptr[K + 1] - P.rowptr[K];
    const int c = (int)(ld - s);
    const int64_t pos0 = P.rowptr[K] + s, off = P.panel_off[K];
    const bool herm = P.herm != 0;
    const T *Zlow = static_cast<const T *>(side ? P.Zu : P.Z);
    const T *Zup = P.lu ? static_cast<const T *>(side ? P.Z : P.Zu) : Zlow;
    const T *B = static_cast<const T *>(side ? P.LDu : P.LD) + off + s;
    const int64_t *pcb = P.colbase + pos0, *prb = P.relbase + pos0;
    const GatherCheck chk = gather_check(P);
    const int tid = threadIdx.x;
    for (int r = tid; r < R; r += kFmThreads) {
        tile_cb[r] = p0 + r < c ? P.colbase[pos0 + p0 + r] : 0;
        tile_rb[r] = p0 + r < c ? P.relbase[pos0 + p0 + r] : 0;
    }
    if (tid < TN) ymax[tid] = 0;
    T acc[R / 16][TN / 8];
#pragma unroll
    for (int i = 0; i < R / 16; i++)
#pragma unroll
        for (int j = 0; j < TN / 8; j++) acc[i][j] = Sc<T>::zero();
    constexpr int NA = R * kFmK / kFmThreads, NB = TN * kFmK / kFmThreads;
    // entry u of this thread in the stage at k0: contiguous down the stored
    // columns, rows fastest below the diagonal, k fastest above it
    auto place = [&](int k0, int u, int &r, int &kk) {
        const int e = tid + kFmThreads * u;
        if (k0 >= p0 + R) { kk = e % kFmK; r = e / kFmK; }
        else { r = e % R; kk = e / R; }
    };
    const int per = ((c + CL - 1) / CL + kFmK - 1) / kFmK * kFmK;     // this CTA's range of q
    const int ka = rank * per, kb = c < ka + per ? c : ka + per;
    __syncthreads();
    int64_t addr[NA];            // of the next stage
    auto find = [&](int k0) {
#pragma unroll
        for (int u = 0; u < NA; u++) {
            int r, kk;
            place(k0, u, r, kk);
            const int p = p0 + r, q = k0 + kk;
            addr[u] = -1;
            if (p < c && q < kb) {
                const int64_t a = p >= q ? pcb[q] + P.relidx[prb[q] + p] : tile_cb[r] + P.relidx[tile_rb[r] + q];
                if (chk.ok(a)) addr[u] = a;
            }
        }
    };
    T va[NA], vb[NB];
    auto load = [&](int k0) {
#pragma unroll
        for (int u = 0; u < NA; u++) {
            int r, kk;
            place(k0, u, r, kk);
            const bool up = p0 + r < k0 + kk;
            T v = addr[u] >= 0 ? (up ? Zup : Zlow)[addr[u]] : Sc<T>::zero();
            va[u] = up ? cjif(v, herm) : v;
        }
#pragma unroll
        for (int u = 0; u < NB; u++) {
            const int e = tid + kFmThreads * u, kk = e % kFmK, j = e / kFmK;
            vb[u] = k0 + kk < kb && j0 + j < s ? B[(int64_t)(j0 + j) * ld + k0 + kk] : Sc<T>::zero();
        }
    };
    find(ka);
    load(ka);
    find(ka + kFmK);
    for (int k0 = ka; k0 < kb; k0 += kFmK) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < NA; u++) {
            int r, kk;
            place(k0, u, r, kk);
            As[kk][r] = va[u];
        }
#pragma unroll
        for (int u = 0; u < NB; u++) {
            const int e = tid + kFmThreads * u;
            Bs[e % kFmK][e / kFmK] = vb[u];
        }
        __syncthreads();
        if (k0 + kFmK < kb) {    // the next stage's values and the addresses after them, under the products
            load(k0 + kFmK);
            find(k0 + 2 * kFmK);
        }
        fma_stage<T, R, TN>(As, Bs, kb - k0 < kFmK ? kb - k0 : kFmK, acc);
    }
    T *out = static_cast<T *>(side ? P.Zu : P.Z) + off + s;
    const int tx = tid % 16, ty = tid / 16;
    if (CL > 1) {                // the partial sums through shared memory, added in rank order
        T *Pt = kFmK * (R + 1) >= R * TN ? &As[0][0] : &Bs[0][0];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < R / 16; i++)
#pragma unroll
            for (int j = 0; j < TN / 8; j++) Pt[(ty + 8 * j) * R + tx + 16 * i] = acc[i][j];
        cl.sync();
        if (rank == 0)
            for (int q = 1; q < CL; q++) {
                const T *pq = cl.map_shared_rank(Pt, q);
#pragma unroll
                for (int i = 0; i < R / 16; i++)
#pragma unroll
                    for (int j = 0; j < TN / 8; j++) acc[i][j] = add(acc[i][j], pq[(ty + 8 * j) * R + tx + 16 * i]);
            }
        cl.sync();
        if (rank) return;
    }
#pragma unroll
    for (int j = 0; j < TN / 8; j++) {
        const int col = j0 + ty + 8 * j;
        int e = 0;
#pragma unroll
        for (int i = 0; i < R / 16; i++) {
            const int p = p0 + tx + 16 * i;
            if (p < c && col < s) {
                out[(int64_t)col * ld + p] = neg(acc[i][j]);
                e = max(e, bexp(acc[i][j]));
            }
        }
        if (e) atomicMax(&ymax[ty + 8 * j], e);
    }
    if (side) return;
    __syncthreads();
    // whole-column exponents for the row bounds of later tensor-core gathers (zeroed at the start of the call)
    if (tid < TN && ymax[tid]) atomicMax(&P.colexpZ[fc + j0 + tid], ymax[tid]);
}

// items: tile = row tile of 32 rows, ntiles = (column tile of 32) << 1 | side
template <typename T>
__global__ void __launch_bounds__(kFmThreads) k_fma_lhat(const ProbDesc *__restrict__ descs,
                                                         const Item *__restrict__ items, int nitems) {
    grid_dep_wait();
    constexpr int R = 32;
    __shared__ T As[kFmK][R + 1], Bs[kFmK][kFmaCols + 1];
    const int w = blockIdx.x;
    if (w >= nitems) return;
    const Item it = items[w];
    const ProbDesc &P = descs[it.prob];
    const int K = it.K, side = it.ntiles & 1, j0 = (it.ntiles >> 1) * kFmaCols, p0 = it.tile * R;
    const int s = P.super_ptr[K + 1] - P.super_ptr[K];
    const int64_t ld = P.rowptr[K + 1] - P.rowptr[K], off = P.panel_off[K];
    const int c = (int)(ld - s);
    const T *L = static_cast<const T *>(side ? P.Ut : P.L) + off + s;
    const T *X = static_cast<const T *>(side ? P.Vt : P.Linv) + P.linv_off[K];
    T *out = static_cast<T *>(side ? P.LDu : P.LD) + off + s;
    const int tid = threadIdx.x;
    T acc[R / 16][4];
#pragma unroll
    for (int i = 0; i < R / 16; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = Sc<T>::zero();
    for (int k0 = j0; k0 < s; k0 += kFmK) {      // X is lower triangular: k >= j0 only
        __syncthreads();
#pragma unroll
        for (int u = 0; u < R * kFmK / kFmThreads; u++) {
            const int e = tid + kFmThreads * u, r = e % R, kk = e / R;
            As[kk][r] = k0 + kk < s && p0 + r < c ? L[(int64_t)(k0 + kk) * ld + p0 + r] : Sc<T>::zero();
        }
#pragma unroll
        for (int u = 0; u < kFmaCols * kFmK / kFmThreads; u++) {
            const int e = tid + kFmThreads * u, kk = e % kFmK, j = e / kFmK;
            Bs[kk][j] = k0 + kk < s && j0 + j < s ? X[(int64_t)(j0 + j) * s + k0 + kk] : Sc<T>::zero();
        }
        __syncthreads();
        fma_stage<T, R, kFmaCols>(As, Bs, s - k0 < kFmK ? s - k0 : kFmK, acc);
    }
    const int tx = tid % 16, ty = tid / 16;
#pragma unroll
    for (int i = 0; i < R / 16; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int p = p0 + tx + 16 * i, col = j0 + ty + 8 * j;
            if (p < c && col < s) out[(int64_t)col * ld + p] = acc[i][j];
        }
}

// Narrow ones (s <= 16): a thread per row of C and exactly the triangle's
// products (a 64 x 8 tile over 16 k spent four times as many).
// items: tile = tile of 128 rows, ntiles = side
template <typename T>
__global__ void __launch_bounds__(kFmThreads) k_fma_lhat_narrow(const ProbDesc *__restrict__ descs,
                                                                const Item *__restrict__ items, int nitems) {
    grid_dep_wait();
    __shared__ T Xs[kNarrowS * kNarrowS];
    const int w = blockIdx.x;
    if (w >= nitems) return;
    const Item it = items[w];
    const ProbDesc &P = descs[it.prob];
    const int K = it.K, side = it.ntiles & 1;
    const int s = P.super_ptr[K + 1] - P.super_ptr[K];
    const int64_t ld = P.rowptr[K + 1] - P.rowptr[K], off = P.panel_off[K];
    const T *X = static_cast<const T *>(side ? P.Vt : P.Linv) + P.linv_off[K];
    for (int e = threadIdx.x; e < s * s; e += kFmThreads) Xs[e] = X[e];
    __syncthreads();
    const int p = it.tile * kFmThreads + threadIdx.x;
    if (p >= (int)(ld - s)) return;
    const T *L = static_cast<const T *>(side ? P.Ut : P.L) + off + s + p;
    T *out = static_cast<T *>(side ? P.LDu : P.LD) + off + s + p;
    for (int j = 0; j < s; j++) {
        T acc = mul(L[(int64_t)j * ld], Xs[j * s + j]);
        for (int k = j + 1; k < s; k++) madd(acc, L[(int64_t)k * ld], Xs[j * s + k]);
        out[(int64_t)j * ld] = acc;
    }
}

// items: tile = 16 x 16 tile of the s x s block (row-major over the lower
// triangle, LU: over the square); a cluster shares the rows of C
template <typename T>
__global__ void __launch_bounds__(kFmThreads) k_fma_diag(const ProbDesc *__restrict__ descs,
                                                         const Item *__restrict__ items, int nitems) {
    grid_dep_wait();
    // [p][16] of Lhat (LU: Uhat^T) and of A^{-1}_{C,K}, columns i0.. and j0..
    __shared__ T Li[kFmK][17], Lj[kFmK][17], Yi[kFmK][17], Yj[kFmK][17];
    __shared__ T Pt[2][256];
    cg::cluster_group cl = cg::this_cluster();
    const int CL = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int w = blockIdx.x / CL;
    if (w >= nitems) return;                 // the grid is nitems clusters: never taken by a part of one
    const Item it = items[w];
    const ProbDesc &P = descs[it.prob];
    const int K = it.K;
    const int fc = P.super_ptr[K];
    const int s = P.super_ptr[K + 1] - fc;
    const int64_t ld = P.rowptr[K + 1] - P.rowptr[K], off = P.panel_off[K];
    const int c = (int)(ld - s);
    const bool lu = P.lu != 0, herm = P.herm != 0;
    int ti = 0, tj = it.tile;
    if (lu) {
        const int nt = (s + 15) / 16;
        ti = it.tile / nt;
        tj = it.tile % nt;
    } else {
        while (tj > ti) { tj -= ti + 1; ti++; }
    }
    const int i0 = ti * 16, j0 = tj * 16;
    const T *LD = static_cast<const T *>(P.LD) + off;
    const T *Lh = (lu ? static_cast<const T *>(P.LDu) : static_cast<const T *>(P.LD)) + off + s;
    T *Zk = static_cast<T *>(P.Z) + off;
    const int per = ((c + CL - 1) / CL + kFmK - 1) / kFmK * kFmK;
    const int pa = rank * per, pb = c < pa + per ? c : pa + per;
    const int tid = threadIdx.x;
    T d[2] = {Sc<T>::zero(), Sc<T>::zero()}, m[2] = {Sc<T>::zero(), Sc<T>::zero()};   // (i, j) and (j, i)
    for (int k0 = pa; k0 < pb; k0 += kFmK) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 16 * kFmK / kFmThreads; u++) {
            const int e = tid + kFmThreads * u, kk = e % kFmK, x = e / kFmK, p = k0 + kk;
            const bool oi = p < pb && i0 + x < s, oj = p < pb && j0 + x < s;
            Li[kk][x] = oi ? cjif(Lh[(int64_t)(i0 + x) * ld + p], herm) : Sc<T>::zero();
            Yj[kk][x] = oj ? Zk[(int64_t)(j0 + x) * ld + s + p] : Sc<T>::zero();
            if (!lu) {
                Lj[kk][x] = oj ? cjif(Lh[(int64_t)(j0 + x) * ld + p], herm) : Sc<T>::zero();
                Yi[kk][x] = oi ? Zk[(int64_t)(i0 + x) * ld + s + p] : Sc<T>::zero();
            }
        }
        __syncthreads();
        const int kk = pb - k0 < kFmK ? pb - k0 : kFmK, x = tid % 16, y = tid / 16;
#pragma unroll 4
        for (int k = 0; k < kk; k++) {
            const T a = Li[k][x];
            madd(d[0], a, Yj[k][y]);
            madd(d[1], a, Yj[k][y + 8]);
            if (!lu) {
                const T b = Yi[k][x];
                madd(m[0], Lj[k][y], b);
                madd(m[1], Lj[k][y + 8], b);
            }
        }
    }
#pragma unroll
    for (int v = 0; v < 2; v++) {
        const int x = tid % 16 + 16 * (tid / 16 + 8 * v);
        Pt[0][x] = d[v];
        Pt[1][x] = m[v];
    }
    if (CL > 1) cl.sync();
    else __syncthreads();
    if (rank == 0)
        for (int x = tid; x < 256; x += kFmThreads) {
            const int i = i0 + x % 16, j = j0 + x / 16;
            if (i >= s || j >= s || (!lu && i < j)) continue;
            T a = LD[(int64_t)j * ld + i], b = LD[(int64_t)i * ld + j];
            for (int q = 0; q < CL; q++) {
                const T *pq = CL > 1 ? cl.map_shared_rank(&Pt[0][0], q) : &Pt[0][0];
                a = sub(a, pq[x]);
                if (!lu) b = sub(b, pq[256 + x]);
            }
            if (lu) {
                Zk[(int64_t)j * ld + i] = a;
                (static_cast<T *>(P.Zu) + off)[(int64_t)i * ld + j] = a;
                continue;
            }
            if (P.symmetrize) {   // (X + X^T) / 2, or (X + X^H) / 2
                a = half(add(a, cjif(b, herm)));
                b = cjif(a, herm);
            }
            Zk[(int64_t)j * ld + i] = a;
            Zk[(int64_t)i * ld + j] = b;
            const int ea = bexp(a), eb = bexp(b);
            if (ea) atomicMax(&P.colexpZ[fc + j], ea);
            if (eb) atomicMax(&P.colexpZ[fc + i], eb);
        }
    if (CL > 1) cl.sync();   // no CTA leaves while the first may still read its sums
}

template <typename... A>
static cudaError_t launch_cluster(void (*kernel)(A...), int n, int cl, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n * cl));
    cfg.blockDim = dim3(kFmThreads);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cl;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename T>
static cudaError_t launch_fma_rows_t(int rows, int cols, int cl, const ProbDesc *d, const Item *items, int n, cudaStream_t st) {
    if (rows == 16)
        return cols == 16 ? launch_cluster(k_fma_rows<T, 16, 16>, n, cl, st, d, items, n)
                          : launch_cluster(k_fma_rows<T, 16, 32>, n, cl, st, d, items, n);
    return cols == 16 ? launch_cluster(k_fma_rows<T, 32, 16>, n, cl, st, d, items, n)
                      : launch_cluster(k_fma_rows<T, 32, 32>, n, cl, st, d, items, n);
}

cudaError_t launch_fma_rows(int dtype, int rows, int cols, int cl, const ProbDesc *d, const Item *items, int n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    return dtype == SELINV_C128 ? launch_fma_rows_t<zd>(rows, cols, cl, d, items, n, st)
                                : launch_fma_rows_t<double>(rows, cols, cl, d, items, n, st);
}

cudaError_t launch_fma_lhat(int dtype, int narrow, const ProbDesc *d, const Item *items, int n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (dtype == SELINV_C128) {
        if (narrow) k_fma_lhat_narrow<zd><<<n, kFmThreads, 0, st>>>(d, items, n);
        else k_fma_lhat<zd><<<n, kFmThreads, 0, st>>>(d, items, n);
    } else {
        if (narrow) k_fma_lhat_narrow<double><<<n, kFmThreads, 0, st>>>(d, items, n);
        else k_fma_lhat<double><<<n, kFmThreads, 0, st>>>(d, items, n);
    }
    return cudaGetLastError();
}

cudaError_t launch_fma_diag(int dtype, int cl, const ProbDesc *d, const Item *items, int n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    return dtype == SELINV_C128 ? launch_cluster(k_fma_diag<zd>, n, cl, st, d, items, n)
                                : launch_cluster(k_fma_diag<double>, n, cl, st, d, items, n);
}

}  // namespace selinv
