// Exact fixed-point helpers shared by the tensor-core kernels.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

namespace selinv {

constexpr int kDig = 7;          // digits per FP64 operand of the tensor-core products

// fp16 bit pattern of a small integer v (|v| <= 128): exact via an fp32
// round trip through the magic constant 1.5 * 2^23, then an exact narrowing.
__device__ __forceinline__ uint32_t f16_of_int(int v) {
    const float f = __int_as_float(0x4B400000 + v) - 12582912.0f;
    return (uint32_t)__half_as_ushort(__float2half_rn(f));
}

// Balanced operands of a product over the columns k of a supernode, sum_k
// X(p, k) Y(k, j) with X(p, k) growing like 1 / sqrt(D_k) and Y like sqrt(D_k)
// (rows of L against rows of L D, or against columns of L_KK^{-1}): in a badly
// scaled matrix D spans many decades within one supernode, and digits on one
// grid per row would lose what the grid's largest entry hides.  With e_k half
// of D_k's exponent, X 2^{e_k} and Y 2^{-e_k} have rows of even size and the
// same product, exactly.  k_balance(D_k) is e_k + kBalBias, the shift of X's
// exponents; 2 kBalBias - k_balance that of Y's; exponents on the biased scale
// stay positive, and kBalBad marks an infinity or a NaN.
constexpr int kBalBias = 1024, kBalBad = 1 << 20;
__device__ __forceinline__ int k_balance(int dexp) {   // dexp: biased exponent of D_k (its larger part)
    return ((dexp - 1023) >> 1) + kBalBias;
}
__device__ __forceinline__ int bal_exp(int e, int add) { return e == 0x7FF ? kBalBad : (e ? e + add : 0); }

// 7 balanced base-256 digits (most significant first) of x on the grid of
// biased exponent E (E >= exponent of x): x ~= sum_i d_i 2^(E-1022-7-8i), cut
// toward zero (ROUND: to nearest, half away from zero); add: x taken as
// x 2^add (E on that scale).
template <bool ROUND = false>
__device__ __forceinline__ void digits7(double x, int E, int d[kDig], int add = 0) {
    const long long b = __double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7FF);
    unsigned long long mant = ex ? ((b & 0xFFFFFFFFFFFFFull) | (1ull << 52)) : 0ull;
    const int sh = E - (ex + add) - 2;               // M = mant * 2^(2 - (E - ex)) < 2^55
    if (ROUND && sh > 0 && sh < 55) mant += 1ull << (sh - 1);
    unsigned long long M = sh < 0 ? (mant << (-sh)) : (sh < 64 ? (mant >> sh) : 0ull);
#pragma unroll
    for (int i = kDig - 1; i >= 1; i--) {
        int v = (int)(M & 0xFFull);
        M >>= 8;
        if (v >= 128) { v -= 256; M += 1; }
        d[i] = v;
    }
    d[0] = (int)M;                                   // <= 128
    if (b < 0) {
#pragma unroll
        for (int i = 0; i < kDig; i++) d[i] = -d[i];
    }
}


// (hi * 2^32 + lo) * 2^(sc - 48) as a double, rounded once to nearest even,
// with integer operations only (the FP64 pipe is GB300's scarcest unit) and
// shifts of 64-bit words (with 128-bit shifts by a variable the 8192
// conversions at the end of a factorization update's tile took 10 us of its
// 27, 7 of 23 so).
__device__ __forceinline__ double fixed_to_double(long long hi, long long lo, int sc) {
    const __int128 n = ((__int128)hi << 32) + (__int128)lo;
    const unsigned long long sgn = n < 0 ? 0x8000000000000000ull : 0ull;
    const unsigned __int128 m = n < 0 ? (unsigned __int128)(-n) : (unsigned __int128)n;
    unsigned long long mh = (unsigned long long)(m >> 64), ml = (unsigned long long)m;
    int e2 = sc - 48 + 75;                              // value = q * 2^e2 below, q = the top 53 bits
    if (mh == 0) {
        mh = ml;
        ml = 0;
        e2 -= 64;
    }
    if (mh == 0) return 0.0;
    const int lz = __clzll((long long)mh);              // leading bit to bit 63 of mh
    mh = (mh << lz) | ((ml >> 1) >> (63 - lz));
    ml <<= lz;
    e2 -= lz;
    unsigned long long q = mh >> 11;
    const uint32_t cut = (uint32_t)mh & 0x7FFu;         // what is below q's last bit, with any bit of ml
    if (cut > 0x400u || (cut == 0x400u && (ml != 0 || (q & 1ull)))) q++;
    if (q >> 53) {
        q >>= 1;
        e2++;
    }
    const int be = e2 + 52 + 1023;                      // q in [2^52, 2^53)
    if (be <= 0 || be >= 2047) {                        // outside the normal range
        const double v = ldexp((double)q, e2);
        return sgn ? -v : v;
    }
    return __longlong_as_double((long long)(sgn | ((unsigned long long)be << 52) | (q & 0xFFFFFFFFFFFFFull)));
}

// The same for a low word of 32 bits (96-bit sums): three 32-bit words, half the
// instructions.  Issue slots bound the conversions at the end of a tensor-core
// tile (18 warps, 8192 of them).
__device__ __forceinline__ double fixed96_to_double(long long hi, uint32_t lo, int sc) {
    const bool neg = hi < 0;
    uint32_t w0 = neg ? 0u - lo : lo;
    const unsigned long long h = neg ? ~(unsigned long long)hi + (lo == 0u ? 1ull : 0ull) : (unsigned long long)hi;
    uint32_t w2 = (uint32_t)(h >> 32), w1 = (uint32_t)h;
    int be = sc - 48 + 95 + 1023;                       // biased exponent of bit 95
    if (w2 == 0u) {
        w2 = w1;
        w1 = w0;
        w0 = 0u;
        be -= 32;
        if (w2 == 0u) {
            w2 = w1;
            w1 = 0u;
            be -= 32;
            if (w2 == 0u) return 0.0;
        }
    }
    const int lz = __clz((int)w2);                      // leading bit to bit 31 of w2
    w2 = __funnelshift_l(w1, w2, lz);
    w1 = __funnelshift_l(w0, w1, lz);
    w0 <<= lz;
    be -= lz;
    if (be <= 0 || be >= 2046) return fixed_to_double(hi, (long long)lo, sc);   // outside the normal range, or next to it
    // the top 53 bits; the bit below with all that follows rounds them, and a
    // carry out of the mantissa is one more in the exponent
    const uint32_t cut = w1 & 0x7FFu;
    unsigned long long q = ((unsigned long long)w2 << 21) | (w1 >> 11);
    q += cut > 0x400u || (cut == 0x400u && (w0 != 0u || (q & 1ull))) ? 1ull : 0ull;
    q += (unsigned long long)(uint32_t)(be - 1) << 52;
    return __longlong_as_double((long long)(q | (neg ? 0x8000000000000000ull : 0ull)));
}

}  // namespace selinv
