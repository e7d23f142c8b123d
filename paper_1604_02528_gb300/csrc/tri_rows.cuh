// Triangular solves with rows dealt to warps, lanes over the columns: shared
// by the factorization's panel solve and by the inverses of the diagonal blocks.
//
// GB300's FP64 pipe issues one warp instruction per SM sub-partition in 64
// clocks whatever the number of active lanes, and a dependent one no later:
// a chain of s steps is therefore best run by as many sub-partitions as the
// problem has rows.  A warp holds 32 / W rows in registers, W lanes to a row,
// so that lane l has the columns l % W, l % W + W, ... of row l / W.  Step j
// touches the blocks of W columns from its own on: at 128 columns 320
// instructions a row for W = 32, 288 for 16, 272 for 8 (half the last block is
// idle lanes), and a width is rounded up to W.  Few rows are spread one to a
// warp, many are packed.
#pragma once

#include "common.cuh"

namespace selinv {

template <int W = 32> __device__ __forceinline__ double shfl_elem(double v, int src) { return __shfl_sync(0xffffffffu, v, src, W); }
template <int W = 32> __device__ __forceinline__ zd shfl_elem(zd v, int src) {
    return make_zd(__shfl_sync(0xffffffffu, v.x, src, W), __shfl_sync(0xffffffffu, v.y, src, W));
}

// Shared-memory store of a lower triangle of nc blocks of 32 columns: block b
// holds its 32 columns one after the other, rows 32 b .. 32 nc - 1 of each.
__host__ __device__ inline int tri_store_elems(int s) {
    const int nc = (s + 31) / 32;
    return 32 * 32 * (nc * (nc + 1) / 2);
}

// Fills the store with the strict lower triangle of an s x s column-major
// block, columns 32 b0 on (zeros past s; the entries on and above the
// diagonal are never used).  All threads; followed by a barrier of the caller.
template <typename T>
__device__ __forceinline__ void tri_store(T *dst, const T *L, int64_t ld, int s, int b0) {
    const int nc = (s + 31) / 32;
    for (int b = b0; b < nc; b++) {
        const int rows = 32 * (nc - b);
        for (int e = threadIdx.x; e < 32 * rows; e += blockDim.x) {
            const int j = 32 * b + e / rows, k = 32 * b + e % rows;
            if (k < s && k > j) cp_async_elem(dst + e, L + (int64_t)j * ld + k);
            else dst[e] = Sc<T>::zero();
        }
        dst += 32 * rows;
    }
    cp_async_commit();
    cp_async_wait<0>();
}

// y L^T = a for the warp's 32 / W rows a (unit lower L; conj(L) in place of L
// when herm) of nt blocks of W columns, from column j0 on: y_j, final after step
// j - 1, is taken from every later column k as y_j L(k, j).  Finished columns
// are not touched, and a row takes the steps from `own` on, which is among the
// warp's first 32 / W (the columns of an inverse: what lies before is zero, which
// an infinite or undefined entry of L would not keep so).  SCALED: L has the diagonal 1 / rd: y_j = a_j rd[j] is what
// the later columns lose, and what is left in a is the undivided a_j.
template <typename T, int W, int NC, bool SCALED>
__device__ __forceinline__ void tri_rows(T (&a)[NC * 32 / W], const T *Ls, const T *rd, int nt, int j0, int own, bool herm) {
    constexpr int NT = NC * 32 / W;
    const int c = threadIdx.x % W;
#pragma unroll
    for (int b = 0; b < NT; b++) {
        if (b >= nt) break;
        if (W * (b + 1) <= j0) continue;
        const int q = b * W / 32;                       // the store's block of 32 columns
        const T *Lb = Ls + 32 * 32 * (q * NC - q * (q - 1) / 2) + b * W % 32 * 32 * (NC - q) + c - 32 * q;
        auto step = [&](int jj, bool on) {
            T y = shfl_elem<W>(a[b], jj);
            if (SCALED) y = mul(y, rd[W * b + jj]);
            const T *l = Lb + jj * 32 * (NC - q);
#pragma unroll
            for (int t = b; t < NT; t++)
                if (on && (t > b || c > jj) && (t <= NT - 32 / W || t < nt)) msub(a[t], y, cjif(l[W * t], herm));
        };
        int jj = max(0, j0 - W * b);
        for (; jj < W && W * b + jj < j0 + 32 / W - 1; jj++) step(jj, W * b + jj >= own);   // up to the warp's last own step
#pragma unroll 2
        for (; jj < W; jj++) step(jj, true);
    }
}

// A column per row of the warp: columns j0 .. j0 + kTriCols - 1 (all in the
// 32-block j0 / 32) of the inverse of a lower triangle staged from that block
// on, written to the column-major block X (ld ldx) in full: zeros above the
// diagonal.  rd: reciprocals of the diagonal (SCALED), by column.
constexpr int kTriThreads = 128;
constexpr int kTriW = 16;                                       // lanes per column
constexpr int kTriCols = 32 / kTriW * kTriThreads / 32;         // columns of an inverse per CTA

template <typename T, int NC, bool SCALED>
__device__ __forceinline__ void tri_inverse_cols(const T *Ls, const T *rd, T *X, int64_t ldx, int s, int j0) {
    constexpr int W = kTriW, NT = NC * 32 / W;
    const int c0 = 32 * (j0 / 32), j = j0 + threadIdx.x / 32 * (32 / W), c = threadIdx.x % W;
    if (j >= s) return;
    const int col = j + threadIdx.x % 32 / W;
    T a[NT];
#pragma unroll
    for (int t = 0; t < NT; t++) a[t] = c0 + c + W * t == col ? Sc<T>::one() : Sc<T>::zero();
    tri_rows<T, W, NC, SCALED>(a, Ls, SCALED ? rd + c0 : rd, (s - c0 + W - 1) / W, j - c0, col - c0, false);
    if (col >= s) return;
    T *x = X + (int64_t)col * ldx;
    for (int i = c; i < c0; i += W) x[i] = Sc<T>::zero();
#pragma unroll
    for (int t = 0; t < NT; t++) {
        const int i = c0 + c + W * t;
        if (i < s) x[i] = i < col ? Sc<T>::zero() : (SCALED ? mul(a[t], rd[i]) : a[t]);
    }
}

template <typename T, bool SCALED>
__device__ __forceinline__ void tri_inverse(const T *Ls, const T *rd, T *X, int64_t ldx, int s, int j0) {
    const int nc = (s + 31) / 32 - j0 / 32;
    if (nc == 1) tri_inverse_cols<T, 1, SCALED>(Ls, rd, X, ldx, s, j0);
    else if (nc == 2) tri_inverse_cols<T, 2, SCALED>(Ls, rd, X, ldx, s, j0);
    else if (nc == 3) tri_inverse_cols<T, 3, SCALED>(Ls, rd, X, ldx, s, j0);
    else tri_inverse_cols<T, 4, SCALED>(Ls, rd, X, ldx, s, j0);
}

}  // namespace selinv
