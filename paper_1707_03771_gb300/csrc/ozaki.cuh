// Ozaki error-free splitting shared by the split-precision kernels: a value v of a row (or column)
// whose power of two is e (|v 2^-e| < 1) is written as sum_s d_s 2^{-7s} 2^e + r, |r| <= 2^{-7S-1} 2^e,
// with integer digits d_1 in [-128, 128] and d_{s>1} in [-64, 63], each exact in BF16.
#pragma once
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>

namespace dfhf {

// Longest exact chunk of a product of S-slice operands, in contraction terms (a multiple of 64). The pairs
// (s, t) with s + t = L + 2 meet in level L; per term the top level S - 1 is the largest, at most
// 2 * 128 * 64 (d_1 with d_S, twice) + (S - 2) * 64 * 64 (the inner pairs) = 2^14 + (S - 2) 2^12. A chunk
// of K terms keeps every level sum an integer of magnitude <= K * that <= 2^24, exact in FP32 whatever
// the order of the tensor-core additions: 1024, 768, 640, 576 and 448 terms for S = 2, 3, 4, 5 and 7.
template <int S>
constexpr int exact_chunk() {
    return ((1 << 24) / ((1 << 14) + (S > 2 ? S - 2 : 0) * (1 << 12))) / 64 * 64;
}
static_assert(exact_chunk<3>() == 768 && exact_chunk<5>() == 576 && exact_chunk<7>() == 448, "exact chunks");

// 2^e as a double, -1022 <= e <= 1023
__device__ __forceinline__ double pow2d(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }

// v 2^e for any e the slices produce (two exact power-of-two factors keep each in the normal range)
__device__ __forceinline__ double scale_pow2(double v, int e) {
    const int a = e / 2;
    return (v * pow2d(a)) * pow2d(e - a);
}

// rint(v 2^k), ties to even, from the bits of v: for a normal v = m 2^{be-1075} (m the 53-bit significand)
// the scaled value is m 2^{-d} with d = 1075 - be - k, rounded by an integer shift. Exact, as the scaling by
// a power of two is; no FP64 instruction on this path (the FP64 pipe, not HBM, bounded the slicing kernels
// when the scaling and the conversion ran there). Zero gives 0; a subnormal v, or a scaled value of 2^52 or
// more, takes the FP64 route (rint of the exactly scaled value), which the slices never need.
__host__ __device__ __forceinline__ long long rint_pow2(double v, int k) {
    unsigned long long b;
    memcpy(&b, &v, sizeof b);
    if ((b << 1) == 0) return 0;
    const int be = (int)((b >> 52) & 0x7ff);
    const int d = 1075 - be - k;
    if (be == 0 || d <= 0) {
        const int a = k / 2;
        return (long long)rint(ldexp(ldexp(v, a), k - a));
    }
    if (d >= 54) return 0;                            // |v 2^k| < 2^53 2^-54 = 1/2
    // ties to even by an addition before the shift: half less one, plus the lowest kept bit
    const unsigned long long m = (b & 0xfffffffffffffULL) | 0x10000000000000ULL;
    const long long q = (long long)((m + ((1ULL << (d - 1)) - 1) + ((m >> d) & 1)) >> d);
    return (b >> 63) ? -q : q;
}

// float(d) for |d| < 2^22 by an addition: int-to-float conversions run at an eighth of its rate
__device__ __forceinline__ unsigned small_float_bits(int d) {
    return __float_as_uint(__int_as_float(0x4B400000 + d) - 12582912.f);
}

// the two values' high halves (exact BF16 of the digits) as one word, a first
__device__ __forceinline__ unsigned pack_bf16(unsigned a, unsigned b) { return __byte_perm(a, b, 0x7632); }

// The digits come from one integer: T = rint(v 2^{7S-e}) (|T| <= 2^{7S}) peeled into balanced base-128
// digits from the least significant end (d_S..d_2 in [-64, 63], d_1 the remaining quotient), as the bits of
// floats. Integer arithmetic throughout, 64 bits wide only while T needs it.
template <int S>
__device__ __forceinline__ void split_digits(double v, int e, unsigned (&f)[S]) {
    long long T = rint_pow2(v, 7 * S - e);
    int t = 0;
#pragma unroll
    for (int s = S - 1; s >= 1; --s) {
        if (7 * (s + 1) + 1 > 31) {                   // T still has more than 31 bits
            const long long u = T + 64;
            f[s] = small_float_bits((int)(u & 127) - 64);
            T = u >> 7;
            t = (int)T;
        } else {
            if (s == S - 1) t = (int)T;
            const int u = t + 64;
            f[s] = small_float_bits((u & 127) - 64);
            t = u >> 7;
        }
    }
    f[0] = small_float_bits(S == 1 ? (int)T : t);
}

// slices of one value, and of two values that are neighbours in every slice (out 4-byte aligned)
template <int S>
__device__ __forceinline__ void split_pow2(double v, int e, __nv_bfloat16* out, long long stride) {
    unsigned f[S];
    split_digits<S>(v, e, f);
#pragma unroll
    for (int s = 0; s < S; ++s) out[s * stride] = __ushort_as_bfloat16((unsigned short)(f[s] >> 16));
}
template <int S>
__device__ __forceinline__ void split_pow2_pair(double a, int ea, double b, int eb, __nv_bfloat16* out, long long stride) {
    unsigned f[S], g[S];
    split_digits<S>(a, ea, f);
    split_digits<S>(b, eb, g);
#pragma unroll
    for (int s = 0; s < S; ++s) *reinterpret_cast<unsigned*>(out + s * stride) = pack_bf16(f[s], g[s]);
}

// |v| as the bits of a non-negative double, which order as their values do (a NaN counts as zero): maxima in
// integer arithmetic, off the FP64 pipe
__device__ __forceinline__ unsigned long long abs_bits(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
    return b > 0x7ff0000000000000ull ? 0 : b;
}

}  // namespace dfhf
