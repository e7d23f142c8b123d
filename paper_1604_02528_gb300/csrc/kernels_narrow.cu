// The whole of Alg. 1's second loop for a narrow supernode -- s <= 16 columns,
// its part of A^{-1}_{C,C} in shared memory -- by one CTA or one thread-block
// cluster: the gather of A^{-1}_{C,C}, A^{-1}_{C,K} = -A^{-1}_{C,C} Lhat, and
// A^{-1}_KK = Dinv_K - Lhat^T A^{-1}_{C,K}, symmetrized (Sec. II-C; Lhat^H for a
// Hermitian problem).  The deep levels of a nested-dissection tree hold
// hundreds to thousands of these.
//
// The FP64 pipe bounds it: an SM sub-partition issues one FP64 instruction per
// 64 clocks whatever the number of active lanes, so a warp per supernode (an
// earlier form) ran c^2 s / 32 of them in one chain on one of the SM's four
// sub-partitions -- 135 us for a complex supernode of 8 columns and 64 rows --
// and the warp sums of the diagonal block were as many again.  Here the c s
// outputs are dealt to the threads one by one, so that every lane of every
// instruction is a product term and all sub-partitions work; on levels with
// few supernodes a cluster of up to 8 CTAs shares the rows of C, the partial
// sums of the diagonal block meeting in the first CTA (distributed shared
// memory).  The pass over the outputs takes ceil(warps / 4) x terms of one
// instruction slot each, which the measurements follow (c = 61, s = 6 complex:
// 25,000 clocks, 31,700 by that count),
// so a sum is split over neighbouring lanes where that fills the last pass;
// levels of up to a CTA per SM take 512 threads and an SM each, longer ones 256
// threads and, alone on their rows, the stored triangle instead of the square.
// 40^3: 6.06 ms without the three, 5.38 with; a batch of 8 matrices (6 poles of
// 18 x 19 x 17 and two real meshes) 4.78 and 3.53; a 2-D grid of 63^2 0.46 and
// 0.43; factoring, inverting and summing 4 poles of 16 x 17 x 15 12.5 and 11.9.
// Every stored entry of A^{-1}_{C,C} is read once, down the columns of
// its panel (contiguous runs of rows), and serves both (p, q) and (q, p).
//
// LU form (nonsymmetric values): entries above the diagonal come from the
// transposed upper panels at the same addresses; a second product with the
// transposed gather gives A^{-1}(K,C)^T = -A^{-1}(C,C)^T Uhat^T, and
// A^{-1}_KK = U_KK^{-1} L_KK^{-1} - Uhat A^{-1}_{C,K} is not symmetrized.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "launch.h"
#include "tile_gemm.cuh"

namespace selinv {

namespace cg = cooperative_groups;

constexpr int kNrBatch = 8;      // gathered runs in flight per warp

// Elements of dynamic shared memory of one CTA: the rows of the gather (twice:
// LU; one CTA alone keeps the stored triangle only, packed, so that levels of
// a thousand supernodes are resident in one wave), Lhat (and Uhat^T),
// A^{-1}_{C,K} of the CTA's rows, its sums of the diagonal block.
__host__ __device__ inline int nr_rows(int c, int cl) { return (c + cl - 1) / cl; }
int narrow_elems(int s, int c, int cl, int lu) {
    const int rows = nr_rows(c, cl), two = lu ? 2 : 1;
    const int gather = cl == 1 && !lu ? c * (c + 1) / 2 : two * c * (rows | 1);
    return gather + two * c * s + rows * s + s * s;
}
__device__ __forceinline__ int tri_at(int p, int q) { return p * (p + 1) / 2 + q; }   // p >= q

// Lanes per sum of len terms, a power of two up to 8: the one whose passes over
// the threads take least (a pass costs a sub-partition its warps' terms).
template <int NT> __device__ __forceinline__ int nr_lanes(int n, int len) {
    int best = 1, least = 1 << 30;
#pragma unroll
    for (int nl = 1, lg = 0; nl <= 8; nl *= 2, lg++) {
        const int warps = (n * nl + 31) / 32, cost = (warps + 3) / 4 * ((len + nl - 1) / nl + lg);
        if (cost < least) {
            least = cost;
            best = nl;
        }
    }
    return best;
}

__device__ __forceinline__ double shfl_xor_elem(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ zd shfl_xor_elem(zd v, int o) {
    return make_zd(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}

// NT threads; PACK: a CTA alone, not the LU form
template <typename T, int NT, bool PACK>
__global__ void __launch_bounds__(NT) k_selinv_narrow(const ProbDesc *__restrict__ descs,
                                                              const Item *__restrict__ items, int nitems) {
    grid_dep_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int ymax[2][kNarrowS], zmax[kNarrowS];
    cg::cluster_group cl = cg::this_cluster();
    const int CL = PACK ? 1 : (int)cl.num_blocks(), rank = PACK ? 0 : (int)cl.block_rank();
    const int w = blockIdx.x / CL;
    if (w >= nitems) return;                 // the grid is nitems clusters: never taken by a part of one
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    const Item it = items[w];
    const ProbDesc &P = descs[it.prob];
    const int K = it.K;
    const int fc = P.super_ptr[K];
    const int s = P.super_ptr[K + 1] - fc;
    const int64_t r0 = P.rowptr[K];
    const int ld = (int)(P.rowptr[K + 1] - r0);
    const int c = ld - s;
    const bool herm = P.herm != 0, lu = !PACK && P.lu != 0;
    const int64_t off = P.panel_off[K];
    const T *LDk = static_cast<const T *>(P.LD) + off;
    const T *LDu = lu ? static_cast<const T *>(P.LDu) + off : LDk;
    T *Zk = static_cast<T *>(P.Z) + off;
    T *Zuk = lu ? static_cast<T *>(P.Zu) + off : nullptr;
    const int rows = nr_rows(c, CL), p0 = rank * rows, p1 = min(c, p0 + rows), np = max(0, p1 - p0);
    const int ldg = rows | 1;
    T *G = reinterpret_cast<T *>(smem_raw);          // [c][ldg]: entry (p0 + r, q) of A^{-1}_{C,C} at q ldg + r
    T *Gt = G + (lu ? c * ldg : 0);                  // LU: entry (q, p0 + r)
    T *Ls = Gt + (PACK ? c * (c + 1) / 2 : c * ldg);                          // [s][c] Lhat
    T *Us = Ls + (lu ? c * s : 0);                   // LU: Uhat^T (else Lhat again)
    T *Y = Us + c * s;                               // [s][rows] A^{-1}_{C,K} of this CTA's rows
    T *Pt = Y + rows * s;                            // [s][s] this CTA's sums of the diagonal block
    // Lhat on its way while the gather's addresses are followed
    for (int e = tid; e < c * s; e += NT) {
        const int q = e % c, j = e / c;
        cp_async_elem(Ls + e, LDk + (int64_t)j * ld + s + q);
        if (lu) cp_async_elem(Us + e, LDu + (int64_t)j * ld + s + q);
    }
    cp_async_commit();
    if (tid < kNarrowS) ymax[0][tid] = ymax[1][tid] = zmax[tid] = 0;
    // the stored entries (a, b), a >= b, with a or b among this CTA's rows:
    // runs of 32 rows a down the columns b, a warp per run
    {
        const T *Z = static_cast<const T *>(P.Z), *Zu = static_cast<const T *>(P.Zu);
        const int64_t *pcb = P.colbase + r0 + s, *prb = P.relbase + r0 + s;
        const GatherCheck chk = gather_check(P);
        const int nblk = (c + 31) / 32, total = c * nblk;
        for (int t0 = warp; t0 < total; t0 += kNrBatch * (NT / 32)) {
            int64_t addr[kNrBatch];
            bool use[kNrBatch];
#pragma unroll
            for (int u = 0; u < kNrBatch; u++) {
                const int t = t0 + u * (NT / 32), b = t / nblk, a = (t % nblk) * 32 + lane;
                use[u] = t < total && a < c && a >= b && ((a >= p0 && a < p1) || (b >= p0 && b < p1));
                addr[u] = use[u] ? pcb[b] + P.relidx[prb[b] + a] : 0;
                if (use[u] && !chk.ok(addr[u])) addr[u] = -1;
            }
            T v[kNrBatch], vu[kNrBatch];
#pragma unroll
            for (int u = 0; u < kNrBatch; u++) {
                const bool ok = use[u] && addr[u] >= 0;
                v[u] = ok ? Z[addr[u]] : Sc<T>::zero();
                vu[u] = lu && ok ? Zu[addr[u]] : Sc<T>::zero();
            }
#pragma unroll
            for (int u = 0; u < kNrBatch; u++) {
                if (!use[u]) continue;
                const int t = t0 + u * (NT / 32), b = t / nblk, a = (t % nblk) * 32 + lane;
                if (PACK) {
                    G[tri_at(a, b)] = v[u];
                    continue;
                }
                // (a, b) as stored; (b, a) its mirror (conjugate: Hermitian), or the upper entry (LU)
                const T m = lu ? vu[u] : cjif(v[u], herm);
                if (a >= p0 && a < p1) {
                    G[b * ldg + a - p0] = v[u];
                    if (lu) Gt[b * ldg + a - p0] = m;
                }
                if (a != b && b >= p0 && b < p1) {
                    G[a * ldg + b - p0] = m;
                    if (lu) Gt[a * ldg + b - p0] = v[u];
                }
            }
        }
    }
    cp_async_wait<0>();
    __syncthreads();
    // A^{-1}_{C,K} = -A^{-1}_{C,C} Lhat on this CTA's rows (LU: and A^{-1}(K,C)^T),
    // a sum over q split over neighbouring lanes where there are few
    for (int side = 0; side < (lu ? 2 : 1); side++) {
        const T *A = side ? Gt : G, *B = side ? Us : Ls;
        T *out = side ? Zuk : Zk;
        const int n = np * s, nl = nr_lanes<NT>(n, c), part = tid & (nl - 1);
        for (int e0 = 0; e0 < n * nl; e0 += NT) {      // (whole warps take part in the sums)
            const int e = (e0 + tid) / nl, r = e < n ? e % np : 0, j = e < n ? e / np : 0;
            T acc = Sc<T>::zero();
            const T *a = A + r, *b = B + j * c;
            if (e < n) {
                if (PACK) {
                    const T *ar = A + tri_at(r, 0), *ac = A + r;   // (r, q) for q <= r, (q, r) beyond
#pragma unroll 4
                    for (int q = part; q < c; q += nl)
                        madd(acc, q <= r ? ar[q] : cjif(ac[tri_at(q, 0)], herm), b[q]);
                } else {
#pragma unroll 4
                    for (int q = part; q < c; q += nl) madd(acc, a[q * ldg], b[q]);
                }
            }
            for (int o = 1; o < nl; o <<= 1) acc = add(acc, shfl_xor_elem(acc, o));
            if (e >= n || part) continue;
            acc = neg(acc);
            out[(int64_t)j * ld + s + p0 + r] = acc;
            if (!side) Y[j * rows + r] = acc;
            atomicMax(&ymax[side][j], bexp(acc));
        }
    }
    __syncthreads();
    // this CTA's rows of sum_p Lhat(p, i) A^{-1}_{C,K}(p, j) (Lhat conjugated:
    // Hermitian; Uhat^T: LU), likewise
    const int ss = s * s;
    {
        const int nl = nr_lanes<NT>(ss, np), part = tid & (nl - 1);
        for (int e0 = 0; e0 < ss * nl; e0 += NT) {
            const int e = (e0 + tid) / nl, i = e < ss ? e % s : 0, j = e < ss ? e / s : 0;
            T acc = Sc<T>::zero();
            if (e < ss)
                for (int r = part; r < np; r += nl) madd(acc, cjif(Us[i * c + p0 + r], herm), Y[j * rows + r]);
            for (int o = 1; o < nl; o <<= 1) acc = add(acc, shfl_xor_elem(acc, o));
            if (e < ss && !part) Pt[e] = acc;
        }
    }
    if (CL > 1) cl.sync();
    else __syncthreads();
    if (rank == 0) {
        // A^{-1}_KK = Dinv_K - the sums, in CTA order; each thread forms an entry and its mirror
        for (int x = tid; x < ss; x += NT) {
            const int i = x % s, j = x / s;
            if (!lu && i < j) continue;
            T d = LDk[(int64_t)j * ld + i], m = LDk[(int64_t)i * ld + j];
            T pd[8], pm[8];                            // every CTA's sums on their way together (CL <= 8)
#pragma unroll
            for (int q = 0; q < 8; q++)
                if (q < CL) {
                    const T *pq = CL > 1 ? cl.map_shared_rank(Pt, q) : Pt;
                    pd[q] = pq[j * s + i];
                    pm[q] = pq[i * s + j];
                }
#pragma unroll
            for (int q = 0; q < 8; q++)
                if (q < CL) {
                    d = sub(d, pd[q]);
                    if (!lu) m = sub(m, pm[q]);
                }
            if (lu) {
                Zk[(int64_t)j * ld + i] = d;
                Zuk[(int64_t)i * ld + j] = d;
                continue;
            }
            if (P.symmetrize) {   // (X + X^T) / 2, or (X + X^H) / 2
                d = half(add(d, cjif(m, herm)));
                m = cjif(d, herm);
            }
            Zk[(int64_t)j * ld + i] = d;
            Zk[(int64_t)i * ld + j] = m;
            atomicMax(&zmax[j], bexp(d));
            atomicMax(&zmax[i], bexp(m));
        }
        __syncthreads();
        // the largest exponent of each whole column, for the row bounds of later tensor-core gathers
        if (tid < s) {
            int y = zmax[tid];
            for (int q = 0; q < CL; q++) y = max(y, CL > 1 ? cl.map_shared_rank(&ymax[0][0], q)[tid] : ymax[0][tid]);
            P.colexpZ[fc + tid] = y;
        }
    }
    if (CL > 1) cl.sync();   // no CTA leaves while the first may still read its sums
}

template <typename T>
static cudaError_t configure_narrow_t() {
    cudaError_t e = cudaFuncSetAttribute(k_selinv_narrow<T, 512, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kNarrowAlone);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_selinv_narrow<T, 512, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kNarrowAlone);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_selinv_narrow<T, 256, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kNarrowSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_selinv_narrow<T, 256, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kNarrowSmem);
    return e;
}

cudaError_t configure_narrow_kernels() {
    const cudaError_t e = configure_narrow_t<double>();
    return e == cudaSuccess ? configure_narrow_t<zd>() : e;
}

template <typename T>
static cudaError_t launch_narrow_t(int cl, int lu, int smem, const ProbDesc *d, const Item *items, int n, cudaStream_t st) {
    // up to a CTA per SM: 512 threads, and shared memory for one alone (the
    // CTAs of a cluster may otherwise share an SM and its FP64 pipe)
    const bool few = n * cl <= 152, pack = cl == 1 && !lu;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n * cl));
    cfg.blockDim = dim3(few ? 512 : 256);
    cfg.dynamicSmemBytes = (size_t)(few ? std::max(smem, kNarrowAlone) : smem);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cl;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (few)
        return pack ? cudaLaunchKernelEx(&cfg, k_selinv_narrow<T, 512, true>, d, items, n)
                    : cudaLaunchKernelEx(&cfg, k_selinv_narrow<T, 512, false>, d, items, n);
    return pack ? cudaLaunchKernelEx(&cfg, k_selinv_narrow<T, 256, true>, d, items, n)
                : cudaLaunchKernelEx(&cfg, k_selinv_narrow<T, 256, false>, d, items, n);
}

cudaError_t launch_selinv_narrow(int dtype, int cl, int lu, int smem, const ProbDesc *d, const Item *items, int n,
                                 cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    return dtype == SELINV_C128 ? launch_narrow_t<zd>(cl, lu, smem, d, items, n, st)
                                : launch_narrow_t<double>(cl, lu, smem, d, items, n, st);
}

}  // namespace selinv
