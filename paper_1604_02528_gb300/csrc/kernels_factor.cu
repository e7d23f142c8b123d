// Prerequisite factorization A = L D L^T without pivoting, supernodal, level
// by level from the leaves (Sec. IV of the paper uses a supernodal
// factorization with a symmetric permutation and no dynamic pivoting; Sec.
// II-C: LDL^T for symmetric A, L D L^H for a Hermitian one, where every
// transposed factor below is conjugated), in multifrontal form:
//
//   k_assemble  scatter A's CSC values into the panels (after a memset)
//   k_fasm      extend-add of each child's update matrix U_child into its
//               parent J: entries whose column is one of J's columns go to
//               J's panel, the rest into U_J (one launch per child rank, so
//               no two writers meet; fixed order: deterministic)
//   k_fsmall    a whole narrow supernode: the next three steps at once
//   k_fdiag     dense LDL^T of J's diagonal block in place (a cluster of CTAs)
//   k_ftrsm     L(C,J) = A(C,J) L_JJ^{-T} D_J^{-1}, row tiles
//   k_fupd      U_J -= L_CJ D_J L_CJ^T (lower c x c, tiles); large real ones
//               on the tensor cores: k_fupd_digits (digit planes of L_CJ D_J)
//               and the SYRK mode of the transposed tcgen05 kernel
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "digit_rows.cuh"
#include "launch.h"
#include "nvtx.h"
#include "plan.h"
#include "put.cuh"
#include "seg_update.cuh"
#include "tri_rows.cuh"

namespace selinv {

namespace cg = cooperative_groups;

constexpr int kFSmallS = 16;        // widest supernode of k_fsmall
constexpr int kFSmallElems = 3400;  // ... and its largest panel (both copies of a complex one in 109 KB)
// narrowest supernode (with the caller's oz_min_s, if that is wider) and
// shortest C of the tcgen05 update: one of its
// CTAs takes about as long as the FP64 pipe of an SM needs for 16 columns of
// a 128 x 64 tile, and below 96 rows most of that tile is padding
constexpr int kFTcS = 17, kFTcC = 96;

template <typename T>
__global__ void k_assemble(const int64_t *__restrict__ pos, const T *__restrict__ vals, int64_t nnz,
                           T *__restrict__ L) {
    grid_dep_wait();
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz;
         e += (int64_t)gridDim.x * blockDim.x)
        L[pos[e]] = vals[e];
}

// Extend-add of one child's update matrix into its parent J: entry (a, b),
// a >= b, of U_child lands at rows(J) positions (pa, pb) -- in J's panel when
// the column C_child[b] is one of J's columns, else in U_J.  One launch per
// child rank: two children of one parent never run together.
template <typename T>
__global__ void __launch_bounds__(256) k_fasm(const FactorDesc *__restrict__ fd, const int2 *__restrict__ items,
                                              int nitems) {
    grid_dep_wait();
    const int w = blockIdx.x;
    if (w >= nitems) return;
    const FactorDesc &F = *fd;
    const int ch = items[w].x, chunk = items[w].y;
    const int J = F.sparent[ch];
    const int sch = F.super_ptr[ch + 1] - F.super_ptr[ch];
    const int cch = (int)(F.rowptr[ch + 1] - F.rowptr[ch] - sch);
    const int sJ = F.super_ptr[J + 1] - F.super_ptr[J];
    const int64_t ldJ = F.rowptr[J + 1] - F.rowptr[J];
    const int cJ = (int)(ldJ - sJ);
    const int32_t *pos = F.chpos + F.rowptr[ch] + sch;
    const T *Uc = static_cast<const T *>(F.U) + F.u_off[ch];
    T *UJ = static_cast<T *>(F.U) + F.u_off[J];
    T *PJ = static_cast<T *>(F.L) + F.panel_off[J];
    const int64_t cc = (int64_t)cch * cch;
    for (int64_t e = (int64_t)chunk * kAsmChunk + threadIdx.x; e < cc && e < (int64_t)(chunk + 1) * kAsmChunk; e += 256) {
        const int a = (int)(e % cch), b = (int)(e / cch);
        if (a < b) continue;
        const T v = Uc[e];
        const int pa = pos[a], pb = pos[b];
        T *dst = pb < sJ ? PJ + (int64_t)pb * ldJ + pa : UJ + (int64_t)(pb - sJ) * cJ + (pa - sJ);
        *dst = add(*dst, v);
    }
}

// U_J -= L_CJ D_J L_CJ^T on one B x B tile of the lower c x c triangle
template <typename T, int B>
__global__ void __launch_bounds__(256) k_fupd(const FactorDesc *__restrict__ fd, const int4 *__restrict__ items,
                                              int nitems) {
    grid_dep_wait();
    __shared__ SegSmem<T, B> sm;
    const int w = blockIdx.x;
    if (w >= nitems) return;
    const FactorDesc &F = *fd;
    const int J = items[w].x, ti = items[w].y, tj = items[w].z;
    const int sJ = F.super_ptr[J + 1] - F.super_ptr[J];
    const int64_t ld = F.rowptr[J + 1] - F.rowptr[J];
    const int c = (int)(ld - sJ);
    const T *LC = static_cast<const T *>(F.L) + F.panel_off[J] + sJ;   // L(p, k) = LC[k*ld + p]
    const T *DJ = static_cast<const T *>(F.D) + F.super_ptr[J];
    T *UJ = static_cast<T *>(F.U) + F.u_off[J];
    const int pa = ti * B, st = tj * B;
    const int np = c - pa < B ? c - pa : B, nq = c - st < B ? c - st : B;
    auto x = [&](int pl, int k) { return mul(LC[(int64_t)k * ld + pa + pl], DJ[k]); };
    auto y = [&](int ql, int k) { return cjif(LC[(int64_t)k * ld + st + ql], F.herm != 0); };
    auto out = [&](int pl, int ql, T v) {
        T *dst = UJ + (int64_t)(st + ql) * c + pa + pl;
        *dst = sub(*dst, v);
    };
    seg_update<T, decltype(x), decltype(y), decltype(out), B>(pa, np, st, nq, sJ, x, y, out, sm);
}

// Digit planes of the rows of L_CJ D_J (undivided rows of the panel solve, up
// to rounding) for the tcgen05 form of the update.  work: (J, 32-row block).
__global__ void __launch_bounds__(256) k_fupd_digits(const FactorDesc *__restrict__ fd, const int2 *__restrict__ work,
                                                     int nwork) {
    grid_dep_wait();
    const int w = blockIdx.x;
    if (w >= nwork) return;
    const FactorDesc &F = *fd;
    const int J = work[w].x, b = work[w].y;
    const int s = F.super_ptr[J + 1] - F.super_ptr[J];
    const int64_t ld = F.rowptr[J + 1] - F.rowptr[J];
    const double *LC = static_cast<const double *>(F.L) + F.panel_off[J] + s;
    const double *DJ = static_cast<const double *>(F.D) + F.super_ptr[J];
    auto x = [&](int p, int k) -> double { return LC[(int64_t)k * ld + p] * DJ[k]; };
    auto add = [&](int k) { return 2 * kBalBias - k_balance(bexp(DJ[k])); };
    digit_rows<true>(x, add, s, (int)(ld - s), b, F.up.linvd + F.up.linvd_off[J], F.up.linvexp + F.rowptr[J] + s);
}

// ---------------------------------------------------------------------------
// k_fdiag: dense LDL^T of J's diagonal block by one thread-block cluster.
// GB300 issues one FP64 instruction per SM sub-partition in 64 clocks, and a
// dependent one no later, so two things bound it: the s^3 / 6 products (85 us
// for 128 columns on one SM), and the chain pivot, reciprocal, scale, update
// of every column (5 instructions at least, 20 us).  The levels near the root
// hold one to eight such blocks: a cluster (8 CTAs there, 1 where a level has
// blocks enough for every SM) keeps the rows cyclically, four at a time, in
// its CTAs' shared memory.  Per block of 32 columns:
//   - every CTA reads the 32 x 32 diagonal block from the owners (distributed
//     shared memory) and factors it by itself, the triangle's entries dealt to
//     four warps (no lane idle, little else on the pipe than the chain);
//   - its own rows below are solved against it, a warp per two rows;
//   - the solved rows are exchanged and the CTA's rows of the trailing block
//     updated.
// Two cluster barriers per block.  (Panels of 8 columns factored on all rows
// by every CTA put 3.5 more instructions per column on the chain: 114 us for
// 128 columns, against 600 us for one CTA in global memory.)
// ---------------------------------------------------------------------------
constexpr int kFdThreads = 256;
constexpr int kFdChain = 128;      // threads that factor the diagonal block
constexpr int kFdNB = 32;          // columns per block
constexpr int kFdLd = kFdNB + 1;   // row stride of the exchanged rows
constexpr int kFdSlots = (kFdNB * (kFdNB + 1) / 2 + kFdChain - 1) / kFdChain;   // entries per chain thread

// 1 / d: the hardware's approximate reciprocal r0 (relative error below
// 2^-19), then one step r0 (1 + e + e^2), e = 1 - d r0, of the hyperpower
// iteration of third order (M. Altman, Pacific J. Math. 10, 1960): e^3 < 2^-57
// beside the last rounding, 0.5625 units in the last place where the division
// has 0.5.  Three dependent FP64 operations, 240 clocks with the seed, where
// the division takes 385.  Magnitudes near the ends of the exponent range (and
// zero, infinities, NaN) go through the division.
// The division is a call: inlined, its own FP64 operations would run beside
// the others in every lane.
__device__ __noinline__ double full_recip(double d) { return 1.0 / d; }
__device__ __forceinline__ double fast_recip(double d) {
    const int e = (int)((__double_as_longlong(d) >> 52) & 0x7FF);
    if (e < 64 || e > 1982) return full_recip(d);
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    const double x = fma(-d, r, 1.0);
    return fma(fma(x, x, x), r, r);
}
__device__ __noinline__ zd full_recip(zd d) { return recip(d); }
// complex: conj(d) / |d|^2 while |d|^2 and its reciprocal stay in range
__device__ __forceinline__ zd fast_recip(zd d) {
    const int ex = (int)((__double_as_longlong(d.x) >> 52) & 0x7FF), ey = (int)((__double_as_longlong(d.y) >> 52) & 0x7FF);
    const int e = ex > ey ? ex : ey;
    if (e < 623 || e > 1423) return full_recip(d);
    const double r = fast_recip(fma(d.x, d.x, d.y * d.y));
    return make_zd(d.x * r, -d.y * r);
}

// elements of a CTA's row store for s columns, clusters of cl CTAs: groups of
// four rows, group g as 4 rows of 4 (g + 1) entries
__host__ __device__ inline int fd_rows_elems(int s, int cl) {
    const int groups = (s + 3) / 4, mine = (groups + cl - 1) / cl;   // at most, rank cl - 1
    return 16 * (cl * (mine * (mine - 1) / 2) + mine * cl);
}
// ... and of everything: the rows below a block, the block's columns (y and L), the row store
__host__ __device__ inline int fd_elems(int s, int cl) {
    return (s > kFdNB ? s - kFdNB : 0) * kFdLd + 2 * kFdNB * kFdLd + fd_rows_elems(s, cl);
}

template <typename T>
__global__ void __launch_bounds__(kFdThreads) k_fdiag(const FactorDesc *__restrict__ fd, const int *__restrict__ js,
                                                      int nj) {
    grid_dep_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ T rD[kFdNB];
    cg::cluster_group cl = cg::this_cluster();
    const int CL = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int lc = 31 - __clz(CL);           // CL = 1 << lc
    const int w = blockIdx.x >> lc;
    if (w >= nj) return;                     // the grid is nj clusters: never taken by a part of one
    const FactorDesc &F = *fd;
    const int J = js[w];
    const int fc = F.super_ptr[J];
    const int s = F.super_ptr[J + 1] - fc;
    const int64_t ld = F.rowptr[J + 1] - F.rowptr[J];
    T *P = static_cast<T *>(F.L) + F.panel_off[J];
    T *D = static_cast<T *>(F.D) + fc;
    const bool herm = F.herm != 0;
    T *Yd = reinterpret_cast<T *>(smem_raw);            // [column][row] of the diagonal block, undivided (y = l d)
    T *Ld = Yd + kFdNB * kFdLd;                         // [column][row] of its L
    T *Yp = Ld + kFdNB * kFdLd;                         // [row below the block][column] undivided
    T *A = Yp + (s > kFdNB ? s - kFdNB : 0) * kFdLd;    // this CTA's rows
    const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
    // row i = 4 g + u lives in rank g % CL at (local group g / CL)
    auto off = [&](int i) {
        const int g = i >> 2, lg = g >> lc, r = g & (CL - 1);
        return 16 * (((lg * (lg - 1) / 2) << lc) + lg * (r + 1)) + (i & 3) * 4 * (g + 1);
    };
    const int groups = (s + 3) / 4;
    const int myg = groups > rank ? (groups - rank + CL - 1) >> lc : 0;   // row groups of this CTA
    auto row_of = [&](int lr) { return (((lr >> 2) << lc) + rank) * 4 + (lr & 3); };
    auto owner = [&](int i) { return (i >> 2) & (CL - 1); };
    for (int k = warp; k < s; k += kFdThreads / 32)
        for (int lr = lane; lr < 4 * myg; lr += 32) {
            const int i = row_of(lr);
            if (i < s && k <= i) cp_async_elem(A + off(i) + k, P + (int64_t)k * ld + i);
        }
    cp_async_commit();
    cp_async_wait<0>();
    // the block's rows of L into the row store, when every CTA has read them
    auto keep = [&](int b0) {
        const int nb = s - b0 < kFdNB ? s - b0 : kFdNB;
        for (int e = tid; e < nb * nb; e += kFdThreads) {
            const int i = e % nb, j = e / nb;
            if (i > j && owner(b0 + i) == rank) A[off(b0 + i) + b0 + j] = Ld[j * kFdLd + i];
        }
    };
    // the chain threads' entries of a block's triangle, column after column
    // (as the chain moves on, whole slots fall done): row and column, and the
    // last column in the warp's slot
    T a[kFdSlots];
    int ei[kFdSlots], ek[kFdSlots], last[kFdSlots];
    auto deal = [&](int nb) {
        const int ne = nb * (nb + 1) / 2;
        int k = 0, q = tid;
#pragma unroll
        for (int u = 0; u < kFdSlots; u++) {
            const bool on = tid + u * kFdChain < ne;
            while (on && q >= nb - k) q -= nb - k++;
            ek[u] = on ? k : -1;
            ei[u] = on ? k + q : 0;
            last[u] = __reduce_max_sync(0xffffffffu, ek[u]);
            q += kFdChain;
        }
    };
    if (tid < kFdChain) deal(s < kFdNB ? s : kFdNB);
    for (int b0 = 0; b0 < s; b0 += kFdNB) {
        const int nb = s - b0 < kFdNB ? s - b0 : kFdNB;
        if (CL > 1) cl.sync();
        else __syncthreads();
        if (tid < kFdChain) {
            if (b0 && nb < kFdNB) deal(nb);
#pragma unroll
            for (int u = 0; u < kFdSlots; u++) {
                const int i = b0 + ei[u];
                a[u] = ek[u] >= 0 ? (CL > 1 ? cl.map_shared_rank(A, owner(i)) : A)[off(i) + b0 + ek[u]] : Sc<T>::zero();
            }
            for (int j = 0; j < nb; j++) {
#pragma unroll
                for (int u = 0; u < kFdSlots; u++)
                    if (ek[u] == j) Yd[j * kFdLd + ei[u]] = a[u];
                asm volatile("bar.sync 1, 128;\n" ::: "memory");
                const T dj = Yd[j * kFdLd + j], r = fast_recip(dj);
                const T l = mul(Yd[j * kFdLd + (lane > j && lane < nb ? lane : j)], r);   // row `lane` of L's column
#pragma unroll
                for (int u = 0; u < kFdSlots; u++) {
                    if (last[u] <= j) continue;                  // the whole warp's slot is done
                    const T li = shfl_elem(l, ei[u]);
                    if (ek[u] > j) msub(a[u], li, cjif(Yd[j * kFdLd + ek[u]], herm));
                }
                if (warp == 3 && lane >= j && lane < nb) {
                    if (lane > j) Ld[j * kFdLd + lane] = l;
                    else rD[j] = r;
                }
            }
        }
        __syncthreads();
        if (rank == 0 && warp == 7 && lane < nb) {               // the pivots, off the chain
            const T d = Yd[lane * kFdLd + lane];
            if (is_zero(d) || !finite_val(d)) atomicCAS(F.status, 0, SELINV_ERR_ZERO_PIVOT);
            D[b0 + lane] = d;
        }
        const int b1 = b0 + kFdNB, below = s - b1;
        if (below <= 0) break;                                   // (a full block otherwise: nb = 32)
        // own rows below the block: y L^T = a, lanes over the block's columns, two rows per warp
        for (int lr = 2 * warp; lr < 4 * myg; lr += 2 * (kFdThreads / 32)) {
            const int i0 = row_of(lr), i1 = row_of(lr + 1);      // (of one group of four)
            if (i1 < b1 || i0 >= s) continue;
            const bool second = i1 < s;
            T y0 = A[off(i0) + b0 + lane], y1 = second ? A[off(i1) + b0 + lane] : Sc<T>::zero();
#pragma unroll 4
            for (int j = 0; j < kFdNB; j++) {
                const T v0 = shfl_elem(y0, j), v1 = shfl_elem(y1, j);
                if (lane > j) {
                    const T l = cjif(Ld[j * kFdLd + lane], herm);
                    msub(y0, v0, l);
                    msub(y1, v1, l);
                }
            }
            const T r = rD[lane];
            Yp[(i0 - b1) * kFdLd + lane] = y0;
            A[off(i0) + b0 + lane] = mul(y0, r);
            if (second) {
                Yp[(i1 - b1) * kFdLd + lane] = y1;
                A[off(i1) + b0 + lane] = mul(y1, r);
            }
        }
        if (CL > 1) {
            cl.sync();
            for (int i = b1 + warp; i < s; i += kFdThreads / 32) {
                const int o = owner(i);
                if (o != rank) Yp[(i - b1) * kFdLd + lane] = cl.map_shared_rank(Yp, o)[(i - b1) * kFdLd + lane];
            }
        }
        __syncthreads();
        keep(b0);
        // own rows of the trailing block: a_ik -= l_i y_k, columns b1 .. i of row i
        // -- entries dealt to the threads one by one (an idle lane costs as much
        // as a busy one), all lanes of a warp brought to their entry before the
        // products start
        int total = 0;
        for (int lr = 0; lr < 4 * myg; lr++) {
            const int r = row_of(lr);
            total += r < s && r >= b1 ? r - b1 + 1 : 0;
        }
        int lr = 0, q = tid, r = row_of(0), cnt = r < s && r >= b1 ? r - b1 + 1 : 0;
        for (int e = tid; e < total; e += kFdThreads) {
            while (q >= cnt) {                         // to the q-th column of local row lr
                q -= cnt;
                r = row_of(++lr);
                cnt = r < s && r >= b1 ? r - b1 + 1 : 0;
            }
            __syncwarp(__activemask());
            T *row = A + off(r);
            T acc = row[b1 + q];
            const T *lrow = row + b0, *yrow = Yp + q * kFdLd;
#pragma unroll 8
            for (int j = 0; j < kFdNB; j++) msub(acc, lrow[j], cjif(yrow[j], herm));
            row[b1 + q] = acc;
            q += kFdThreads;
        }
    }
    if (CL > 1) cl.sync();   // the last block is read no more, and no CTA leaves while another may still read its rows
    keep((s - 1) / kFdNB * kFdNB);
    __syncthreads();
    for (int k = warp; k < s; k += kFdThreads / 32)
        for (int lr = lane; lr < 4 * myg; lr += 32) {
            const int i = row_of(lr);
            if (i < s) P[(int64_t)k * ld + i] = i > k ? A[off(i) + k] : (i == k ? Sc<T>::one() : Sc<T>::zero());
        }
}

// ---------------------------------------------------------------------------
// k_ftrsm: X D L_JJ^T = A for the rows of C (D L_JJ^H for a Hermitian matrix):
// with y = x D, step j broadcasts y_j and every later column subtracts
// y_j L(k, j); the rows are scaled by 1 / D once at the end.  L_JJ's lower
// triangle waits in shared memory (columns from their 32-block's first row on,
// zeros above the diagonal).  The FP64 pipe bounds it, so a warp packs four
// rows of its share into its lanes, then two, then one (tri_rows), and the row
// tiles are made small enough that every SM gets one.
// 40^3: the panel solves of all levels 3.95 ms with one row to a lane block of
// 32 columns, 3.53 so.
// items {J, first row of C, rows}
// ---------------------------------------------------------------------------
constexpr int kFtThreads = kTriThreads;

template <typename T, int W, int NC>
__device__ __forceinline__ void ftrsm_group(const T *Ls, const T *rD, T *P, int64_t ld, int s, int row, int end, bool herm) {
    constexpr int NT = NC * 32 / W;
    const int c = threadIdx.x % W;
    row += threadIdx.x % 32 / W;
    T a[NT];
#pragma unroll
    for (int t = 0; t < NT; t++) {
        const int k = c + W * t;
        a[t] = row < end && k < s ? P[(int64_t)k * ld + row] : Sc<T>::zero();
    }
    tri_rows<T, W, NC, false>(a, Ls, nullptr, (s + W - 1) / W, 0, 0, herm);
#pragma unroll
    for (int t = 0; t < NT; t++) {
        const int k = c + W * t;
        if (row < end && k < s) P[(int64_t)k * ld + row] = mul(a[t], rD[k]);
    }
}

template <typename T, int NC>
__device__ void ftrsm_rows(const T *Ls, const T *rD, T *P, int64_t ld, int s, int row0, int nrows, bool herm) {
    constexpr int kWarps = kFtThreads / 32;
    const int share = (nrows + kWarps - 1) / kWarps, warp = threadIdx.x / 32;
    const int end = row0 + min(nrows, (warp + 1) * share);
    for (int row = row0 + warp * share; row < end;) {
        const int left = end - row;
        if (left > 2) ftrsm_group<T, 8, NC>(Ls, rD, P, ld, s, row, end, herm);
        else if (left == 2) ftrsm_group<T, 16, NC>(Ls, rD, P, ld, s, row, end, herm);
        else ftrsm_group<T, 32, NC>(Ls, rD, P, ld, s, row, end, herm);
        row += left > 2 ? 4 : left;
    }
}

template <typename T>
__global__ void __launch_bounds__(kFtThreads) k_ftrsm(const FactorDesc *__restrict__ fd,
                                                      const int4 *__restrict__ items, int nitems) {
    grid_dep_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ T rD[128];
    T *Ls = reinterpret_cast<T *>(smem_raw);
    const int w = blockIdx.x;
    if (w >= nitems) return;
    const FactorDesc &F = *fd;
    const int4 it = items[w];
    const int J = it.x;
    const int fc = F.super_ptr[J];
    const int s = F.super_ptr[J + 1] - fc;
    const int64_t ld = F.rowptr[J + 1] - F.rowptr[J];
    T *P = static_cast<T *>(F.L) + F.panel_off[J];
    const T *D = static_cast<const T *>(F.D) + fc;
    const bool h = F.herm != 0;
    const int nc = (s + 31) / 32;
    for (int k = threadIdx.x; k < s; k += kFtThreads) rD[k] = recip(D[k]);
    tri_store(Ls, P, ld, s, 0);
    __syncthreads();
    T *Pc = P + s;
    if (nc == 1) ftrsm_rows<T, 1>(Ls, rD, Pc, ld, s, it.y, it.z, h);
    else if (nc == 2) ftrsm_rows<T, 2>(Ls, rD, Pc, ld, s, it.y, it.z, h);
    else if (nc == 3) ftrsm_rows<T, 3>(Ls, rD, Pc, ld, s, it.y, it.z, h);
    else ftrsm_rows<T, 4>(Ls, rD, Pc, ld, s, it.y, it.z, h);
}

// ---------------------------------------------------------------------------
// k_fsmall: a whole narrow supernode (s <= kFSmallS columns, its panel twice
// in shared memory): LDL^T of the diagonal block and the rows of C together,
// column by column (one barrier each), then U_J -= (L D) L^T over exactly the
// entries of the lower triangle, 2 x 2 per thread.  One launch where the
// blocks' own kernels would each be launch-bound, and no 64 x 64 x 16 tile
// for a 20 x 20 x 3 product.
// ---------------------------------------------------------------------------
constexpr int kFsThreads = 128;

template <typename T>
__global__ void __launch_bounds__(kFsThreads) k_fsmall(const FactorDesc *__restrict__ fd, const int *__restrict__ js,
                                                       int nj) {
    grid_dep_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int w = blockIdx.x;
    if (w >= nj) return;
    const FactorDesc &F = *fd;
    const int J = js[w];
    const int fc = F.super_ptr[J];
    const int s = F.super_ptr[J + 1] - fc;
    const int ld = (int)(F.rowptr[J + 1] - F.rowptr[J]);
    const int c = ld - s;
    T *P = static_cast<T *>(F.L) + F.panel_off[J];
    T *D = static_cast<T *>(F.D) + fc;
    const bool herm = F.herm != 0;
    T *Y = reinterpret_cast<T *>(smem_raw);   // [s][ld] columns: the panel, then y = l d
    T *Lp = Y + s * ld;                       // [s][ld] columns of L
    const int tid = threadIdx.x;
    for (int e = tid; e < s * ld; e += kFsThreads) Y[e] = P[e];
    for (int j = 0; j < s; j++) {
        __syncthreads();                      // column j is final on the rows of the diagonal block
        const T d = Y[j * ld + j];
        const T r = recip(d);
        if (tid == 0) {
            if (is_zero(d) || !finite_val(d)) atomicCAS(F.status, 0, SELINV_ERR_ZERO_PIVOT);
            D[j] = d;
        }
        for (int i = j + 1 + tid; i < ld; i += kFsThreads) {
            const T l = mul(Y[j * ld + i], r);
            Lp[j * ld + i] = l;
            for (int k = j + 1; k < s && k <= i; k++) msub(Y[k * ld + i], l, cjif(Y[j * ld + k], herm));
        }
    }
    __syncthreads();
    for (int e = tid; e < s * ld; e += kFsThreads) {
        const int j = e / ld, i = e % ld;
        P[e] = i > j ? Lp[e] : (i == j ? Sc<T>::one() : Sc<T>::zero());
    }
    // U_J(p, q) -= sum_k y_p l_q, p >= q, in 2 x 2 blocks of the lower triangle
    T *UJ = static_cast<T *>(F.U) + F.u_off[J];
    const int nt = (c + 1) / 2;
    int tj = 0, ti = tid;                     // block row ti (from the diagonal on) of block column tj
    for (int e = tid; e < nt * (nt + 1) / 2; e += kFsThreads) {
        while (ti >= nt - tj) {
            ti -= nt - tj;
            tj++;
        }
        __syncwarp(__activemask());           // all lanes at their block before the products start
        const int p = 2 * (tj + ti), q = 2 * tj;
        const bool p1 = p + 1 < c, q1 = q + 1 < c;
        T a00 = Sc<T>::zero(), a10 = Sc<T>::zero(), a01 = Sc<T>::zero(), a11 = Sc<T>::zero();
        for (int k = 0; k < s; k++) {
            const T *yk = Y + k * ld + s, *lk = Lp + k * ld + s;
            const T y0 = yk[p], y1 = p1 ? yk[p + 1] : Sc<T>::zero();
            const T l0 = cjif(lk[q], herm), l1 = q1 ? cjif(lk[q + 1], herm) : Sc<T>::zero();
            madd(a00, y0, l0);
            madd(a10, y1, l0);
            madd(a01, y0, l1);
            madd(a11, y1, l1);
        }
        T *u = UJ + (int64_t)q * c + p;
        u[0] = sub(u[0], a00);
        if (p1) u[1] = sub(u[1], a10);
        if (q1 && p > q) u[c] = sub(u[c], a01);
        if (p1 && q1) u[c + 1] = sub(u[c + 1], a11);
        ti += kFsThreads;
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
void FactorLists::release() {
    for (void *q : {(void *)d_tiles, (void *)d_js, (void *)d_uitems, (void *)d_tcitems, (void *)d_tcwork, (void *)d_digoff})
        if (q) cudaFree(q);
}

void factor_release(selinv_plan_s *plan) {
    FactorData *f = plan->factor;
    if (!f) return;
    auto fr = [](void *p) { if (p) cudaFree(p); };
    fr(f->d_a_pos); fr(f->d_desc);
    fr(f->d_asm); fr(f->d_uoff); fr(f->d_chpos); fr(f->U);
    fr(f->digits); fr(f->digexp);
    for (auto &l : f->lists)
        if (l.second) l.second->release();
    for (CapturedLoop &g : f->loop) g.release();
    adjoint_release(f->adj);
    delete f;
    plan->factor = nullptr;
}

template <typename X>
static int up(X **d, const std::vector<X> &h) {
    *d = nullptr;
    if (dev_malloc((void **)d, sizeof(X) * std::max<size_t>(1, h.size())) != cudaSuccess) return SELINV_ERR_OOM;
    if (!h.empty() && cudaMemcpy(*d, h.data(), sizeof(X) * h.size(), cudaMemcpyHostToDevice) != cudaSuccess)
        return SELINV_ERR_CUDA;
    return SELINV_OK;
}

// the factorization's launch lists for the narrowest tensor-core supernode tc_s:
// made once for each value that the caller sets, and kept (a caller's own
// graph may hold their addresses)
static int factor_lists(selinv_plan_s *plan, int tc_s, FactorLists **out) {
    FactorData *f = plan->factor;
    const PlanData &p = plan->data;
    std::unique_ptr<FactorLists> &slot = f->lists[tc_s];
    if (slot) {
        *out = slot.get();
        return SELINV_OK;
    }
    std::unique_ptr<FactorLists> made(new FactorLists());
    FactorLists *q = made.get();
    int64_t dig_total = 0;   // of every supernode that some tc_s takes
    // per-level launch lists, leaves first: the narrow supernodes, then the
    // others' diagonal blocks and row tiles
    std::vector<int> js;
    std::vector<int4> tiles, uitems;
    std::vector<Item> tcitems;
    std::vector<int2> tcwork;
    std::vector<int64_t> digoff(std::max(p.ns, 1), 0);
    auto width = [&](int32_t J) { return p.super_ptr[J + 1] - p.super_ptr[J]; };
    auto below = [&](int32_t J) { return (int)(p.rowptr[J + 1] - p.rowptr[J]) - width(J); };
    for (int l = p.nlevels - 1; l >= 0; l--) {
        FactorLevel v;
        std::vector<int32_t> wide;
        v.small0 = (int64_t)js.size();
        // one CTA for a whole supernode while its update's c^2 s / 2 products take
        // under 10 us of an SM (c = 64, s = 16), or up to twice that where the
        // level has supernodes for two CTAs on every SM.  Limits of 16384, 65536
        // and 400000 on the shorter levels: 40^3 11.42, 11.42 and 11.50 ms, 16^3
        // 0.92 each, 20^3 Hermitian 4.36, 4.41 and 4.70, 240^2 2.38, 2.78 and
        // 2.91; on the longer ones 32768 to 400000 differ by under 2 % anywhere
        const int64_t small_prod = p.level_ptr[l + 1] - p.level_ptr[l] >= 304 ? 150000 : 65536;
        for (int64_t e = p.level_ptr[l]; e < p.level_ptr[l + 1]; e++) {
            const int32_t J = p.level_list[e];
            const int s = width(J), elems = s * (s + below(J));
            const int64_t prod = (int64_t)s * below(J) * below(J);
            if (s <= kFSmallS && elems <= kFSmallElems && prod <= small_prod) {
                js.push_back(J);
                v.small_elems = std::max(v.small_elems, elems);
            } else {
                wide.push_back(J);
            }
        }
        v.wide0 = (int64_t)js.size();
        v.wide1 = v.wide0 + (int64_t)wide.size();
        js.insert(js.end(), wide.begin(), wide.end());
        int64_t rows = 0;
        for (int32_t J : wide) {
            v.wide_s = std::max(v.wide_s, width(J));
            rows += below(J);
        }
        // a cluster of 8 CTAs per diagonal block while all of them find an SM;
        // wide levels have blocks enough by themselves.  At most 8, 4, 2 and 1
        // CTAs: 40^3 11.3, 11.6, 12.3 and 14.0 ms, 20^3 Hermitian 4.4, 4.7, 5.4 and
        // 6.8, 16^3 complex 2.05, 2.24, 2.68 and 3.54 (one 128-column block of 40^3
        // takes 105 us on 8 SMs, cold caches)
        const int64_t nw = (int64_t)wide.size();
        v.cl = v.wide_s <= 32 ? 1 : (nw * 8 <= 152 ? 8 : (nw * 4 <= 152 ? 4 : (nw * 2 <= 152 ? 2 : 1)));
        // rows per tile: the number whose tiles, dealt to the SMs, take least --
        // a warp's groups of four, two and one row cost about 34, 18 and 10 us
        // of an SM sub-partition at 128 columns, a tile's L_JJ 5 us more for
        // each of the two CTAs in flight; the ratios serve every width (weights
        // scaled to the level's widest supernode choose no better: 24^3 2.93
        // against 2.89 ms).  Tiles of 4, 8, 16 and 64 rows throughout: 40^3 12.35,
        // 11.53, 11.72 and 15.26 ms against 11.42, 16^3 0.93, 0.94, 1.01 and 1.45
        // against 0.92, 20^3 Hermitian 4.57, 4.55, 4.96 and 8.21 against 4.41,
        // 24^3 2.80, 2.81, 3.04 and 4.85 against 2.89
        int rt = 4;
        int64_t least = INT64_MAX;
        for (int t = 4; t <= 64; t += 4) {
            int64_t nt = 0;
            for (int32_t J : wide) nt += (below(J) + t - 1) / t;
            constexpr int rest[4] = {0, 10, 18, 34};
            const int64_t per = (nt + 151) / 152, cost = per * (t / 16 * 34 + rest[t / 4 % 4]) + (per + 1) / 2 * 5;
            if (cost < least) {
                least = cost;
                rt = t;
            }
        }
        v.tile0 = (int64_t)tiles.size();
        for (int32_t J : wide)
            for (int r = 0, c = below(J); r < c; r += rt) tiles.push_back(make_int4(J, r, std::min(rt, c - r), 0));
        v.tile1 = (int64_t)tiles.size();
        // update tiles: the side (64, 32, 16) whose waves over the SMs multiply
        // least, for all of them and for those that the tcgen05 form leaves
        auto tc = [&](int32_t J) { return width(J) >= tc_s && below(J) >= kFTcC; };
        for (int part = 0; part < 2; part++) {
            FactorLevel::Upd &u = v.upd[part];
            int64_t best = INT64_MAX;
            for (int B : {64, 32, 16}) {
                int64_t nt = 0;
                for (int32_t J : wide) {
                    const int64_t t = part && tc(J) ? 0 : (below(J) + B - 1) / B;
                    nt += t * (t + 1) / 2;
                }
                const int64_t cost = (nt + 151) / 152 * (B * B + 4 * B);
                if (cost < best) {
                    best = cost;
                    u.b = B;
                }
            }
            u.i0 = (int64_t)uitems.size();
            for (int32_t J : wide) {
                if (part && tc(J)) continue;
                const int nt = (below(J) + u.b - 1) / u.b;
                for (int ti = 0; ti < nt; ti++)
                    for (int tj = 0; tj <= ti; tj++) uitems.push_back(make_int4(J, ti, tj, 0));
            }
            u.i1 = (int64_t)uitems.size();
        }
        // tcgen05 form: 128 x 64 tiles on or below the diagonal, the digit
        // planes of a level one after the other in one buffer
        v.tc0 = (int64_t)tcitems.size();
        v.tw0 = (int64_t)tcwork.size();
        int64_t dig = 0;
        int64_t any = 0;
        for (int32_t J : wide) {
            const int64_t planes = (int64_t)((below(J) + 127) / 128) * 7 * 128 * ((width(J) + 15) / 16 * 16);
            if (width(J) >= kFTcS && below(J) >= kFTcC) any += planes;
            if (!tc(J)) continue;
            const int c = below(J), n2 = (c + 63) / 64;
            for (int m = 0; m < (c + 127) / 128; m++)
                for (int t = 0; t < n2 && 64 * t <= 128 * m + 127; t++) tcitems.push_back(Item{0, J, m * n2 + t, 1});
            for (int b = 0; b < (c + 31) / 32; b++) tcwork.push_back(make_int2(J, b));
            digoff[J] = dig;
            dig += planes;
        }
        v.tc1 = (int64_t)tcitems.size();
        q->tc = q->tc || v.tc1 > v.tc0;
        v.tw1 = (int64_t)tcwork.size();
        dig_total = std::max(dig_total, any);
        q->lev.push_back(v);
    }
    int rc;
    if ((rc = up(&q->d_tiles, tiles)) || (rc = up(&q->d_js, js)) || (rc = up(&q->d_uitems, uitems)) ||
        (rc = up(&q->d_tcitems, tcitems)) || (rc = up(&q->d_tcwork, tcwork)) || (rc = up(&q->d_digoff, digoff))) {
        q->release();
        return rc;
    }
    f->dig_total = dig_total;
    slot = std::move(made);
    *out = q;
    return SELINV_OK;
}

// update-matrix tables, shared by the factorization and the selected-inversion
// adjoint
int factor_tables(selinv_plan_s *plan) {
    FactorData *f = plan->factor;
    if (f->d_desc) return SELINV_OK;
    const PlanData &p = plan->data;
    int rc = ensure_device(plan->data);
    if (rc) return rc;
    // update matrices: offsets; the position of every C_K entry in its
    // parent's row list (closure: C_K lies inside rows(parent)); children by rank
    f->u_off.assign(p.ns + 1, 0);
    for (int32_t K = 0; K < p.ns; K++) {
        const int64_t c = p.rowptr[K + 1] - p.rowptr[K] - (p.super_ptr[K + 1] - p.super_ptr[K]);
        f->u_off[K + 1] = f->u_off[K] + c * c;
    }
    f->chpos.assign(std::max<int64_t>(p.rowptr[p.ns], 1), 0);
    std::vector<int> rank(p.ns, 0), nchild(p.ns, 0);
    for (int32_t K = 0; K < p.ns; K++) {
        const int32_t P = p.sparent[K];
        if (P < 0) continue;
        rank[K] = nchild[P]++;
        const int s = p.super_ptr[K + 1] - p.super_ptr[K];
        const int32_t *RP = p.rows.data() + p.rowptr[P];
        const int64_t mP = p.rowptr[P + 1] - p.rowptr[P];
        int64_t t = 0;
        for (int64_t r = p.rowptr[K] + s; r < p.rowptr[K + 1]; r++) {   // both lists ascending
            while (t < mP && RP[t] < p.rows[r]) t++;
            f->chpos[r] = (int32_t)t;
        }
    }
    f->npass = 1;
    for (int32_t K = 0; K < p.ns; K++) f->npass = std::max(f->npass, nchild[K]);
    std::vector<int64_t> kid_ptr(p.ns + 1, 0);
    for (int32_t K = 0; K < p.ns; K++) kid_ptr[K + 1] = kid_ptr[K] + nchild[K];
    std::vector<int32_t> kids(std::max<int64_t>(kid_ptr[p.ns], 1));
    for (int32_t K = 0; K < p.ns; K++)
        if (p.sparent[K] >= 0) kids[kid_ptr[p.sparent[K]] + rank[K]] = K;
    f->asm_items.clear();
    f->asm_lptr.assign(1, 0);
    for (int l = p.nlevels - 1; l >= 0; l--) {
        for (int r = 0; r < f->npass; r++) {
            for (int64_t e = p.level_ptr[l]; e < p.level_ptr[l + 1]; e++) {
                const int32_t K = p.level_list[e];
                if (r >= nchild[K]) continue;
                const int32_t ch = kids[kid_ptr[K] + r];
                const int64_t cc = f->u_off[ch + 1] - f->u_off[ch];
                for (int64_t ck = 0; ck < (cc + kAsmChunk - 1) / kAsmChunk; ck++) f->asm_items.push_back(make_int2(ch, (int)ck));
            }
            f->asm_lptr.push_back((int64_t)f->asm_items.size());
        }
    }
    if ((rc = up(&f->d_asm, f->asm_items))) return rc;
    if ((rc = up(&f->d_uoff, f->u_off))) return rc;
    if ((rc = up(&f->d_chpos, f->chpos))) return rc;
    if (dev_malloc((void **)&f->d_desc, sizeof(FactorDesc)) != cudaSuccess) return SELINV_ERR_OOM;
    return SELINV_OK;
}

static FactorDesc *factor_desc(selinv_plan_s *plan, const FactorLists *q, void *L, void *D, cudaStream_t st, int herm) {
    FactorData *f = plan->factor;
    const PlanData &p = plan->data;
    FactorDesc h = {};
    // the tcgen05 update's view: L's panels, digit planes of L D, the update matrices
    h.up.super_ptr = p.d_super_ptr;
    h.up.rowptr = p.d_rowptr;
    h.up.panel_off = p.d_panel_off;
    h.up.L = L;
    h.up.D = D;
    h.up.linvd = f->digits;
    h.up.linvd_off = q->d_digoff;
    h.up.linvexp = f->digexp;
    h.up.Yout = f->U;
    h.up.part_off = f->d_uoff;
    h.up.status = p.d_status;
    h.super_ptr = p.d_super_ptr;
    h.sparent = p.d_sparent;
    h.rowptr = p.d_rowptr;
    h.rows = p.d_rows;
    h.panel_off = p.d_panel_off;
    h.u_off = f->d_uoff;
    h.chpos = f->d_chpos;
    h.U = f->U;
    h.L = L;
    h.D = D;
    h.status = p.d_status;
    h.herm = herm;
    put(f->d_desc, &h, 1, st);
    return f->d_desc;
}

// the dynamic shared memory of the widest blocks, on the plan's device
template <typename T> static cudaError_t configure_factor_kernels() {
    const int diag = (int)(sizeof(T) * (size_t)fd_elems(128, 1));
    const int trsm = (int)(sizeof(T) * (size_t)tri_store_elems(128)), small = (int)(2 * sizeof(T) * kFSmallElems);
    cudaError_t e = cudaFuncSetAttribute(k_fdiag<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, diag);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_ftrsm<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, trsm);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_fsmall<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, small);
    return e;
}

template <typename T>
static int factor_t(selinv_plan_s *plan, const void *A, void *L, void *D, cudaStream_t st, int herm) {
    FactorData *f = plan->factor;
    const int tc_s = std::max(kFTcS, plan->data.asked.oz_min_s);
    FactorLists *q = nullptr;
    if (const int rc = factor_lists(plan, tc_s, &q)) return rc;
    const PlanData &p = plan->data;
    const size_t ubytes = sizeof(T) * (size_t)std::max<int64_t>(f->u_off[p.ns], 1);
    if (f->U_bytes < ubytes) {
        if (f->U) cudaFree(f->U);
        f->U = nullptr;
        f->U_bytes = 0;
        if (dev_malloc((void **)&f->U, ubytes) != cudaSuccess) return SELINV_ERR_OOM;
        f->U_bytes = ubytes;
    }
    // real updates on the tensor cores unless the plan asks for FP64 FMA
    const bool tc = sizeof(T) == 8 && p.asked.fast_contraction == 1 && q->tc;
    if (tc && !f->digits) {
        if (!f->digexp && dev_malloc((void **)&f->digexp, sizeof(int) * (size_t)p.rowptr[p.ns]) != cudaSuccess) return SELINV_ERR_OOM;
        if (dev_malloc((void **)&f->digits, sizeof(uint16_t) * (size_t)f->dig_total) != cudaSuccess) return SELINV_ERR_OOM;
    }
    FactorDesc *fd = factor_desc(plan, q, L, D, st, herm);
    if (cudaMemsetAsync(L, 0, sizeof(T) * (size_t)p.nnz, st) != cudaSuccess) return SELINV_ERR_CUDA;
    if (cudaMemsetAsync(f->U, 0, ubytes, st) != cudaSuccess) return SELINV_ERR_CUDA;
    if (f->nnzA > 0) {
        const int blocks = (int)std::min<int64_t>((f->nnzA + 255) / 256, 152 * 8);
        k_assemble<T><<<blocks, 256, 0, st>>>(f->d_a_pos, static_cast<const T *>(A), f->nnzA, static_cast<T *>(L));
        note_launch();
    }
    if (!f->configured[sizeof(T) > 8]) {
        if (configure_factor_kernels<T>() != cudaSuccess) return SELINV_ERR_CUDA;
        f->configured[sizeof(T) > 8] = true;
    }
    auto levels = [&](cudaStream_t st) {
        for (size_t l = 0; l < q->lev.size(); l++) {
            // the children's update matrices complete J's panel and start U_J
            for (int r = 0; r < f->npass; r++) {
                const int64_t x0 = f->asm_lptr[l * f->npass + r], x1 = f->asm_lptr[l * f->npass + r + 1];
                if (x1 > x0) { k_fasm<T><<<(int)(x1 - x0), 256, 0, st>>>(fd, f->d_asm + x0, (int)(x1 - x0)); note_launch(); }
            }
            const FactorLevel &v = q->lev[l];
            if (v.wide0 > v.small0) {
                k_fsmall<T><<<(int)(v.wide0 - v.small0), kFsThreads, 2 * sizeof(T) * (size_t)v.small_elems, st>>>(
                    fd, q->d_js + v.small0, (int)(v.wide0 - v.small0));
                note_launch();
            }
            if (v.wide1 > v.wide0) {
                cudaLaunchConfig_t cfg = {};
                cfg.gridDim = dim3((unsigned)((v.wide1 - v.wide0) * v.cl));
                cfg.blockDim = dim3(kFdThreads);
                cfg.dynamicSmemBytes = sizeof(T) * (size_t)fd_elems(v.wide_s, v.cl);
                cfg.stream = st;
                cudaLaunchAttribute at[1];
                at[0].id = cudaLaunchAttributeClusterDimension;
                at[0].val.clusterDim.x = (unsigned)v.cl;
                at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
                cfg.attrs = at;
                cfg.numAttrs = 1;
                cudaLaunchKernelEx(&cfg, k_fdiag<T>, (const FactorDesc *)fd, (const int *)(q->d_js + v.wide0),
                                   (int)(v.wide1 - v.wide0));   // (an error stays for cudaGetLastError)
                note_launch();
            }
            if (v.tile1 > v.tile0) {
                k_ftrsm<T><<<(int)(v.tile1 - v.tile0), kFtThreads, sizeof(T) * (size_t)tri_store_elems(v.wide_s), st>>>(
                    fd, q->d_tiles + v.tile0, (int)(v.tile1 - v.tile0));
                note_launch();
            }
            const FactorLevel::Upd &u = v.upd[tc];
            if (u.i1 > u.i0) {
                const int nu = (int)(u.i1 - u.i0);
                if (u.b == 64) k_fupd<T, 64><<<nu, 256, 0, st>>>(fd, q->d_uitems + u.i0, nu);
                else if (u.b == 32) k_fupd<T, 32><<<nu, 256, 0, st>>>(fd, q->d_uitems + u.i0, nu);
                else k_fupd<T, 16><<<nu, 256, 0, st>>>(fd, q->d_uitems + u.i0, nu);
                note_launch();
            }
            if (tc && v.tc1 > v.tc0) {
                const int nw = (int)(v.tw1 - v.tw0);
                k_fupd_digits<<<nw, 256, 0, st>>>(fd, q->d_tcwork + v.tw0, nw);
                launch_syrk_tcw(2, &fd->up, q->d_tcitems + v.tc0, (int)(v.tc1 - v.tc0), p.opts.spin_limit, st);
                note_launch(2);
            }
        }
    };
    if (cudaGetLastError() != cudaSuccess) return SELINV_ERR_CUDA;
    return f->loop[sizeof(T) > 8].run({2 * tc_s + tc, p.opts.spin_limit}, f, st, p.opts.use_graph != 0, levels);
}

}  // namespace selinv

using namespace selinv;

extern "C" int selinv_plan_set_matrix(selinv_plan plan, int32_t n, const int64_t *colptr,
                                      const int32_t *rowind) {
    if (!plan || !colptr || (n > 0 && !rowind) || n != plan->data.n) return SELINV_ERR_INVALID_ARG;
    const PlanData &p = plan->data;
    std::vector<int32_t> col2s(n);
    for (int32_t K = 0; K < p.ns; K++)
        for (int32_t j = p.super_ptr[K]; j < p.super_ptr[K + 1]; j++) col2s[j] = K;
    std::vector<int64_t> pos(colptr[n] > 0 ? colptr[n] : 0);
    for (int32_t j = 0; j < n; j++) {
        const int32_t K = col2s[j];
        const int32_t *R = p.rows.data() + p.rowptr[K];
        const int64_t m = p.rowptr[K + 1] - p.rowptr[K];
        int64_t t = j - p.super_ptr[K];
        for (int64_t e = colptr[j]; e < colptr[j + 1]; e++) {
            const int32_t i = rowind[e];
            if (i < j || i >= n) return SELINV_ERR_BAD_PATTERN;
            while (t < m && R[t] < i) t++;
            if (t >= m || R[t] != i) return SELINV_ERR_BAD_PATTERN;  // A not inside L's pattern
            pos[e] = p.panel_off[K] + (int64_t)(j - p.super_ptr[K]) * m + t;
        }
    }
    if (!plan->factor) plan->factor = new FactorData();
    FactorData *f = plan->factor;
    if (f->d_a_pos) cudaFree(f->d_a_pos);
    f->d_a_pos = nullptr;
    f->n = n;
    f->nnzA = (int64_t)pos.size();
    f->a_pos = pos;
    int rc = ensure_device(plan->data);
    if (rc) return rc;
    return up(&f->d_a_pos, f->a_pos);
}

extern "C" int selinv_factor(selinv_plan plan, selinv_dtype dtype, const void *A, void *L, void *D,
                             void *stream) {
    NvtxRange nvtx_range("selinv_factor");
    if (!plan || !plan->factor || (dtype != SELINV_F64 && dtype != SELINV_C128 && dtype != SELINV_C128H))
        return SELINV_ERR_INVALID_ARG;
    if (plan->data.ns == 0) return SELINV_OK;
    if (!L || !D || (plan->factor->nnzA > 0 && !A)) return SELINV_ERR_INVALID_ARG;
    int rc = factor_tables(plan);
    if (rc) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    plan->last_stream = st;
    return dtype == SELINV_F64 ? factor_t<double>(plan, A, L, D, st, 0)
                               : factor_t<zd>(plan, A, L, D, st, dtype == SELINV_C128H);
}
