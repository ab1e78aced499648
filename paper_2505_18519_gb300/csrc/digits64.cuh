// Error-free splitting of FP64 values into integer digits, for matrix products of
// FP64 accuracy on the tensor cores as sums of exact FP16 digit products (Ozaki,
// Ogita, Oishi and Rump, error-free transformation of a matrix product into sums
// of products of low-precision matrices, Numer. Algorithms 59, 2012).
//
// A group of values sharing an exponent e becomes integers F = rint(x 2^e), the
// largest |F| at most 0.99 2^(TOT - 1), and F = sum_q d_q 2^(BITS (D - 1 - q)) with
// D balanced digits d_q in [-2^(BITS-1), 2^(BITS-1)): integers, so exact in FP16.  The
// products d_i d_j of one order s = i + j accumulate in one FP32 accumulator; the
// orders 0 .. D - 1 are kept.  Every partial sum is an integer of magnitude at
// most (number of products) 2^(2 BITS - 2) <= 2^24, so the tensor cores add exactly:
//   BITS 8, D 8: 36 digit products, up to 128 terms (8 * 128 * 2^14 = 2^24);
//   BITS 7, D 9: 45 digit products, up to 455 terms (9 * 455 * 2^12 < 2^24).
// The dropped orders are below 2^-63 (2^-62) of the two groups' largest entries
// per term, so a product's error is that of one rounding of each operand to 63
// (62) bits and of the result where the caller rounds it.
#pragma once
#include <cuda_fp16.h>
#include <math.h>
#include <stdint.h>

namespace afq {

template <int BITS>
struct Dg64 {
    static_assert(BITS == 8 || BITS == 7, "digit width");
    static constexpr int D = BITS == 8 ? 8 : 9;         // digits per value, and orders kept
    static constexpr int TOT = BITS * D;                // 64, 63
    static constexpr int MAXK = BITS == 8 ? 128 : 455;  // terms of an exact product
    // sum_q 2^(BITS - 1) 2^(BITS q): added to F it makes every digit's field non-negative
    static constexpr uint64_t BIAS = BITS == 8 ? 0x8080808080808080ull : 0x4081020408102040ull;
    // F_A F_B summed = (combined accumulators, see dg64_sum) 2^UNIT
    static constexpr int UNIT = BITS == 8 ? 72 : 70;
    static constexpr int XTRA = BITS == 8 ? 3 : 1;      // extra low bits of dg64_sum_fine
};

constexpr int DG64_NAN = INT32_MIN / 4;   // exponent of a group with a non-finite entry

// Exponent e of a group whose largest |entry| is m: m 2^e <= 0.99 2^(TOT - 1).
template <int BITS>
__device__ __forceinline__ int dg64_exp(double m) {
    if (!(m <= 1.7976931348623157e308)) return DG64_NAN;
    if (m == 0.0) return 0;
    return Dg64<BITS>::TOT - 2 - ilogb(m * 0.5 * 1.0102) - 1;
}

// rint(x 2^e) as an integer (|x 2^e| < 2^63), halves away from zero.
__device__ __forceinline__ long long dg64_fix(double x, int e) {
    const long long u = __double_as_longlong(x);
    const int ex = (int)((u >> 52) & 0x7ff);
    if (ex == 0) return 0;
    unsigned long long m = ((unsigned long long)u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
    const int sh = ex - 1075 + e;
    if (sh >= 0) m <<= sh;
    else if (sh >= -53) m = (m + (1ull << (-sh - 1))) >> (-sh);
    else m = 0;
    return u < 0 ? -(long long)m : (long long)m;
}

// The digits of eight values as FP16: put(q, eight K elements of 16 bits) for digit q.
template <int BITS, class Put>
__device__ __forceinline__ void dg64_unit(const long long (&F)[8], Put put) {
    constexpr int D = Dg64<BITS>::D;
    uint32_t lo[8], hi[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const uint64_t u = (uint64_t)F[t] + Dg64<BITS>::BIAS;
        lo[t] = (uint32_t)u;
        hi[t] = (uint32_t)(u >> 32);
    }
    // 1024 + 2^(BITS - 1) in FP16: a field f below it as the half 1024 + f is one byte merge
    const uint32_t b2 = BITS == 8 ? 0x64806480u : 0x64406440u;
    const __half2 bias = *reinterpret_cast<const __half2*>(&b2);
#pragma unroll
    for (int q = 0; q < D; ++q) {
        uint32_t w[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            uint32_t v;
            if constexpr (BITS == 8) {
                const int b = D - 1 - q, bb = b & 3;
                const uint32_t x = b >= 4 ? hi[2 * t] : lo[2 * t], y = b >= 4 ? hi[2 * t + 1] : lo[2 * t + 1];
                v = (__byte_perm(x, y, (uint32_t)(bb | (bb << 4) | ((4 + bb) << 8) | ((4 + bb) << 12))) & 0x00FF00FFu) |
                    0x64006400u;
            } else {
                const int k = BITS * (D - 1 - q);
                const uint32_t x = k >= 32 ? hi[2 * t] >> (k - 32) : __funnelshift_r(lo[2 * t], hi[2 * t], k);
                const uint32_t y = k >= 32 ? hi[2 * t + 1] >> (k - 32) : __funnelshift_r(lo[2 * t + 1], hi[2 * t + 1], k);
                v = (x & 127u) | ((y & 127u) << 16) | 0x64006400u;
            }
            const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&v), bias);
            w[t] = *reinterpret_cast<const uint32_t*>(&d);
        }
        put(q, make_uint4(w[0], w[1], w[2], w[3]));
    }
}

// The accumulators of the orders as one integer in units of 2^UNIT of F_A F_B
// (rounded there), plus rnd (a small integer); |result| <= (sum |x| of a row / largest |x|) 2^54 + rnd.
template <int BITS>
__device__ __forceinline__ long long dg64_sum(const float (&a)[Dg64<BITS>::D], float rnd) {
    if constexpr (BITS == 8) {
        const int h01 = __float2int_rn(a[0]) * 256 + __float2int_rn(a[1]);
        const int h23 = __float2int_rn(a[2]) * 256 + __float2int_rn(a[3]);
        const int i5 = __float2int_rn(fmaf(a[7], 0x1p-16f, fmaf(a[6], 0x1p-8f, a[5] + rnd)));
        const long long H = (long long)h01 * 65536 + h23;
        const long long L = (long long)__float2int_rn(a[4]) * 256 + i5;
        return H * 65536 + L;
    } else {
        const int h01 = __float2int_rn(a[0]) * 128 + __float2int_rn(a[1]);
        const int h23 = __float2int_rn(a[2]) * 128 + __float2int_rn(a[3]);
        const int h45 = __float2int_rn(a[4]) * 128 + __float2int_rn(a[5]);
        const int i6 = __float2int_rn(fmaf(a[8], 0x1p-14f, fmaf(a[7], 0x1p-7f, a[6] + rnd)));
        const long long H = (long long)h01 * 16384 + h23;
        const long long L = (long long)h45 * 128 + i6;
        return H * 2097152 + L;
    }
}

// The same with XTRA more low bits (units of 2^(UNIT - XTRA)), for at most MAXK / 2 terms.
template <int BITS>
__device__ __forceinline__ long long dg64_sum_fine(const float (&a)[Dg64<BITS>::D]) {
    if constexpr (BITS == 8) {
        const int h01 = __float2int_rn(a[0]) * 256 + __float2int_rn(a[1]);
        const int h23 = __float2int_rn(a[2]) * 256 + __float2int_rn(a[3]);
        const long long H = (long long)h01 * 65536 + h23;
        const long long L = (long long)__float2int_rn(a[4]) * 256 + __float2int_rn(a[5]);
        return (H * 65536 + L) * 8 + __float2int_rn(fmaf(a[7], 0x1p-13f, a[6] * 0x1p-5f));
    } else {
        const int h01 = __float2int_rn(a[0]) * 128 + __float2int_rn(a[1]);
        const int h23 = __float2int_rn(a[2]) * 128 + __float2int_rn(a[3]);
        const int h45 = __float2int_rn(a[4]) * 128 + __float2int_rn(a[5]);
        const long long H = (long long)h01 * 16384 + h23;
        const long long L = (long long)h45 * 128 + __float2int_rn(a[6]);
        return (H * 2097152 + L) * 2 + __float2int_rn(fmaf(a[8], 0x1p-13f, a[7] * 0x1p-6f));
    }
}

}  // namespace afq
