// Triangular solves with a row per warp, lanes over the columns: shared by
// the factorization's panel solve and by the inverses of the diagonal blocks.
//
// GB300's FP64 pipe issues one warp instruction per SM sub-partition in 64
// clocks whatever the number of active lanes, and a dependent one no later:
// a chain of s steps is therefore best run by as many sub-partitions as the
// problem has rows, each warp holding a row (or two, which then share the
// loads of the triangle) in registers, NC = ceil(s / 32) values per lane.
#pragma once

#include "common.cuh"

namespace selinv {

template <typename T> __device__ __forceinline__ T shfl_elem(T v, int src);
template <> __device__ __forceinline__ double shfl_elem(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
template <> __device__ __forceinline__ zd shfl_elem(zd v, int src) {
    return make_zd(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
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

// y L^T = a for R rows a (unit lower L; conj(L) in place of L when herm),
// from column j0 of the first 32 on: y_j, final after step j - 1, is taken
// from every later column k as y_j L(k, j).  Finished columns are not touched.
// SCALED: L has the diagonal 1 / rd: y_j = a_j rd[j] is what the later columns
// lose, and what is left in a is the undivided a_j.
template <typename T, int NC, int R, bool SCALED>
__device__ __forceinline__ void tri_rows(T (&a)[R][NC], const T *Ls, const T *rd, int j0, bool herm) {
    const int lane = threadIdx.x % 32;
    const T *Lb = Ls;
#pragma unroll
    for (int b = 0; b < NC; b++) {
#pragma unroll 2
        for (int jj = b ? 0 : j0; jj < 32; jj++) {
            T l[NC];
#pragma unroll
            for (int t = b; t < NC; t++) l[t] = cjif(Lb[jj * 32 * (NC - b) + lane + 32 * (t - b)], herm);
#pragma unroll
            for (int r = 0; r < R; r++) {
                T y = shfl_elem(a[r][b], jj);
                if (SCALED) y = mul(y, rd[32 * b + jj]);
#pragma unroll
                for (int t = b; t < NC; t++)
                    if (t > b || lane > jj) msub(a[r][t], y, l[t]);
            }
        }
        Lb += 32 * 32 * (NC - b);
    }
}

// Columns j0 .. j0 + 4 R - 1 (a warp for R of them; all in the 32-block j0 / 32)
// of the inverse of a lower triangle staged from that block on, written to the
// column-major block X (ld ldx) in full: zeros above the diagonal.
// rd: reciprocals of the diagonal (SCALED), by column.
template <typename T, int NC, int R, bool SCALED>
__device__ __forceinline__ void tri_inverse_cols(const T *Ls, const T *rd, T *X, int64_t ldx, int s, int j0) {
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, c0 = 32 * (j0 / 32), j = j0 + warp * R;
    if (j >= s) return;
    T a[R][NC];
#pragma unroll
    for (int r = 0; r < R; r++)
#pragma unroll
        for (int t = 0; t < NC; t++) a[r][t] = c0 + lane + 32 * t == j + r ? Sc<T>::one() : Sc<T>::zero();
    tri_rows<T, NC, R, SCALED>(a, Ls, SCALED ? rd + c0 : rd, j - c0, false);
#pragma unroll
    for (int r = 0; r < R; r++) {
        if (j + r >= s) break;
        T *x = X + (int64_t)(j + r) * ldx;
        for (int i = lane; i < c0; i += 32) x[i] = Sc<T>::zero();
#pragma unroll
        for (int t = 0; t < NC; t++) {
            const int i = c0 + lane + 32 * t;
            if (i < s) x[i] = SCALED ? mul(a[r][t], rd[i]) : a[r][t];
        }
    }
}

constexpr int kTriThreads = 128;
constexpr int kTriR = 2;                                      // rows per warp
constexpr int kTriCols = kTriR * kTriThreads / 32;            // columns of an inverse per CTA

template <typename T, bool SCALED>
__device__ __forceinline__ void tri_inverse(const T *Ls, const T *rd, T *X, int64_t ldx, int s, int j0) {
    const int nc = (s + 31) / 32 - j0 / 32;
    if (nc == 1) tri_inverse_cols<T, 1, kTriR, SCALED>(Ls, rd, X, ldx, s, j0);
    else if (nc == 2) tri_inverse_cols<T, 2, kTriR, SCALED>(Ls, rd, X, ldx, s, j0);
    else if (nc == 3) tri_inverse_cols<T, 3, kTriR, SCALED>(Ls, rd, X, ldx, s, j0);
    else tri_inverse_cols<T, 4, kTriR, SCALED>(Ls, rd, X, ldx, s, j0);
}

}  // namespace selinv
