// Digit planes of the rows of a panel product's left operand, as the SYRK
// modes of the transposed tcgen05 kernel read them.
#pragma once

#include "common.cuh"
#include "fixedpoint.cuh"
#include "tile_gemm.cuh"

namespace selinv {

// Rows 32 b .. 32 b + 31 of x (c rows, kw columns), cut by one CTA of 256
// threads: per block of 128 rows, per 16-step of k the 7 planes of 128 x 16
// one after the other (K-major 8 x 8 core matrices), one exponent per row
// (exps[row]).  A warp per 4 rows finds their exponents, then each thread
// cuts 8 consecutive k of one row, a 16-byte store per plane.
// ROUND: to the nearest point of the row's grid instead of toward zero, the
// columns' exponents shifted by add(k) (balanced rows; else add gives 0).
template <bool ROUND, class X, class S>
__device__ __forceinline__ void digit_rows(const X &x, const S &add, int kw, int c, int b, uint16_t *base, int *exps) {
    __shared__ int rowE[32];
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int k16 = (kw + 15) / 16 * 16, nst = k16 / 16;
    for (int rr = 0; rr < 4; rr++) {
        const int r = warp * 4 + rr, p = b * 32 + r;
        int E = 0;
        if (p < c)
            for (int k = lane; k < kw; k += 32) E = max(E, ROUND ? bal_exp(bexp(x(p, k)), add(k)) : bexp(x(p, k)));
#pragma unroll
        for (int o = 16; o; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
        if (lane == 0) {
            rowE[r] = E;
            if (p < c) exps[p] = E;
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 32 * (k16 / 8); e += 256) {
        const int r = e % 32, k0 = (e / 32) * 8, p = b * 32 + r;
        if (p >= c) continue;
        uint32_t h[kDig][4];
#pragma unroll
        for (int t = 0; t < 8; t += 2) {
            int d0[kDig], d1[kDig];
            digits7<ROUND>(k0 + t < kw ? x(p, k0 + t) : 0.0, rowE[r], d0, k0 + t < kw ? add(k0 + t) : 0);
            digits7<ROUND>(k0 + t + 1 < kw ? x(p, k0 + t + 1) : 0.0, rowE[r], d1, k0 + t + 1 < kw ? add(k0 + t + 1) : 0);
#pragma unroll
            for (int i = 0; i < kDig; i++) h[i][t / 2] = f16_of_int(d0[i]) | (f16_of_int(d1[i]) << 16);
        }
        const int t1 = p / 128, r128 = p % 128, st = k0 / 16;
        const int64_t ub = ((int64_t)(t1 * nst + st) * kDig) * 128 * 16 + (r128 / 8) * 128 + ((k0 % 16) / 8) * 64 + (r128 % 8) * 8;
#pragma unroll
        for (int i = 0; i < kDig; i++)
            *reinterpret_cast<uint4 *>(base + ub + (int64_t)i * 128 * 16) = make_uint4(h[i][0], h[i][1], h[i][2], h[i][3]);
    }
}

}  // namespace selinv
