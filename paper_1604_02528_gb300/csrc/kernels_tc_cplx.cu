// Complex symmetric selected inversion on the tensor cores: the operands of
// the real digit contractions for A = A^T with complex values (Sec. II-C:
// plain transposes), and the finisher of the complex diagonal block.
//
// A complex product sum_q X(q, j) Y(q, i) is one real contraction over the
// 2c-long index k' = 2q + part:
//   rows j     of the left operand: (Re X(q, j), -Im X(q, j)) at k' = 2q, 2q + 1
//   rows s + j of the left operand: (Im X(q, j),  Re X(q, j))
//   right operand:                  (Re Y(q, i),  Im Y(q, i))
// so that row j gives Re(X^T Y)(j, i) and row s + j gives Im(X^T Y)(j, i).
// With X = Lhat this left operand serves both A^{-1}_{C,K} = -A^{-1}_{C,C}
// Lhat (k_selinv_tcw, the right operand being the gathered A^{-1}_{C,C}, which
// is symmetric) and the diagonal product Lhat^T A^{-1}_{C,K} (k_diag_tc).
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"
#include "fixedpoint.cuh"
#include "launch.h"
#include "diag_fin.cuh"
#include "tile_gemm.cuh"

namespace selinv {


// ---------------------------------------------------------------------------
// k_digits_z: the left operand above for X = Lhat (complex), or (LINV) for
// X = L_KK^{-1} over its s rows, the operand of Lhat_{C,K} = L_{C,K} L_KK^{-1} on
// tcgen05, as fp16 digit planes in the tcgen05 operand layout: per 16-step
// of k' and plane (the 7 planes of a step one after the other) a block of
// roundup(2s, 64) rows x 16, K-major 8 x 8 core matrices.  One exponent per
// column j of X over both parts (shared by rows j and s + j); L_KK^{-1} is
// balanced by D and rounded to its grid.  One CTA per 8 columns: a warp finds a column's
// exponent, then each thread cuts 4 entries of one column -- 8 consecutive k'
// of both rows, whose digits differ in order and sign only -- and stores 16
// bytes per plane and row (2-byte stores of one k' at a time: 542 us for the
// 64-column supernodes of a 1024-atom sheet).
// work = (problem, (K << 8) | block of 8 columns).
// ---------------------------------------------------------------------------
template <bool LINV>
__global__ void __launch_bounds__(256) k_digits_z(const ProbDesc *__restrict__ descs, const int2 *__restrict__ work,
                                                  int nwork) {
    grid_dep_wait();
    __shared__ int colE[8];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int w = blockIdx.x;
    if (w >= nwork) return;
    const ProbDesc &P = descs[work[w].x];
    const int K = work[w].y >> 8;
    const int jb = work[w].y & 0xFF;
    const int fc = P.super_ptr[K];
    const int s = P.super_ptr[K + 1] - fc;
    const int64_t ld = P.rowptr[K + 1] - P.rowptr[K];
    const int len = LINV ? s : (int)(ld - s);               // entries of a column
    const int64_t ldx = LINV ? s : ld;
    const double2 *X = LINV ? static_cast<const double2 *>(P.Linv) + P.linv_off[K]
                            : static_cast<const double2 *>(P.LD) + P.panel_off[K] + s;
    // L_KK^{-1}'s rows k are balanced against L's columns (k_balance)
    const zd *D = static_cast<const zd *>(P.D) + fc;
    auto add = [&](int q) { return LINV ? 2 * kBalBias - k_balance(bexp(D[q])) : 0; };
    {
        const int j = jb * 8 + warp;
        int E = 0;
        if (j < s)
            for (int q = lane; q < len; q += 32) {
                const double2 v = X[(int64_t)j * ldx + q];
                const int ev = max(bexp(v.x), bexp(v.y));
                E = max(E, LINV ? bal_exp(ev, add(q)) : ev);
            }
#pragma unroll
        for (int o = 16; o; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
        if (lane == 0) {
            colE[warp] = E;
            if (j < s) (LINV ? P.linvexp : P.colexp)[fc + j] = E;
        }
    }
    __syncthreads();
    const int64_t s64 = (2 * s + 63) / 64 * 64;
    const int k16 = (2 * len + 15) / 16 * 16;
    uint16_t *pu = LINV ? P.linvd + P.linvd_off[K] : P.lhsu + P.lhsu_off[K];
    for (int e = threadIdx.x; e < k16; e += 256) {            // (column, 8 k' = 4 entries)
        const int jj = e % 8, k8 = e / 8, j = jb * 8 + jj, E = colE[jj];
        if (j >= s) continue;
        uint32_t h1[kDig][4], h2[kDig][4];                     // rows j and s + j, a (2q, 2q + 1) pair per word
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int q = 4 * k8 + u;
            const double2 v = q < len ? X[(int64_t)j * ldx + q] : make_double2(0.0, 0.0);
            int dr[kDig], di[kDig];
            const int sh = q < len ? add(q) : 0;
            digits7<LINV>(v.x, E, dr, sh);
            digits7<LINV>(v.y, E, di, sh);
#pragma unroll
            for (int i = 0; i < kDig; i++) {
                const uint32_t r = f16_of_int(dr[i]), m = f16_of_int(di[i]);
                h1[i][u] = r | ((m ^ 0x8000u) << 16);          // (Re, -Im)
                h2[i][u] = m | (r << 16);                      // (Im,  Re)
            }
        }
        const int64_t base = (int64_t)(k8 / 2) * kDig * s64 * 16 + (k8 % 2) * 64;
        const int r2 = s + j;
        const int64_t o1 = base + (j / 8) * 128 + (j % 8) * 8, o2 = base + (r2 / 8) * 128 + (r2 % 8) * 8;
#pragma unroll
        for (int i = 0; i < kDig; i++) {
            *reinterpret_cast<uint4 *>(pu + i * s64 * 16 + o1) = make_uint4(h1[i][0], h1[i][1], h1[i][2], h1[i][3]);
            *reinterpret_cast<uint4 *>(pu + i * s64 * 16 + o2) = make_uint4(h2[i][0], h2[i][1], h2[i][2], h2[i][3]);
        }
    }
}

// ---------------------------------------------------------------------------
// k_diag_fin_z: A^{-1}_KK = Dinv_K - Lhat^T A^{-1}_{C,K} (complex) from the
// exact sums of k_diag_tc, symmetrized with the plain transpose (Sec. II-C);
// Hermitian: Dinv_K - Lhat^H A^{-1}_{C,K}, symmetrized as (X + X^H) / 2
// (diag_fin_pair).  One CTA per (K, 2 columns).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_diag_fin_z(const ProbDesc *__restrict__ descs,
                                                    const Item *__restrict__ items, int nitems) {
    grid_dep_wait();
    const int w = blockIdx.x;
    if (w >= nitems) return;
    const Item it = items[w];
    diag_fin_pair<true>(descs[it.prob], it.K, 2 * it.tile, 1);
}

cudaError_t launch_digits_z(int linv, const ProbDesc *d, const int2 *work, int nwork, cudaStream_t st) {
    if (nwork <= 0) return cudaSuccess;
    if (linv) k_digits_z<true><<<nwork, 256, 0, st>>>(d, work, nwork);
    else k_digits_z<false><<<nwork, 256, 0, st>>>(d, work, nwork);
    return cudaGetLastError();
}

cudaError_t launch_diag_fin_z(const ProbDesc *d, const Item *items, int n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_diag_fin_z<<<n, 256, 0, st>>>(d, items, n);
    return cudaGetLastError();
}

}  // namespace selinv
