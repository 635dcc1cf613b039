// sep.cuh -- the separable fixed-point dictionary of the exact correlation.
//
// Each 1-D basis row (DCT-II and Haar, Section 2.1 Eq. (1)-(2), Section 2.3)
// enters in fixed point, Bf = round(B 2^48), an integer below 2^47.5 in
// magnitude (|B| <= sqrt(2/b) <= 2^-0.5).  The 2-D atom (p, q) of a family is
// the outer product of rows p and q (Section 2.1; its pixel (i, m) sits at
// v = m b + i, Appendix A), so with this dictionary the correlation of a
// block y is the exact integer
//
//     T[p][q] = sum_m Bf[q][m] Z[p][m],    Z[p][m] = sum_i Bf[p][i] y[i][m],
//
// i.e. B Y B^T in integers, and c = T 2^-96 rounded once into a double-float.
// With centred pixels y~ = y - 128 the kernels form Z~ = Bf y~ and T~ = Bf^T Z~
// and add the exact centring term 128 R[p] R[q], R[p] = sum_i Bf[p][i].
// Magnitudes: |Z~| < 128 sqrt(b) 2^47.5 <= 2^59, |T| < 2^112 (b <= 128).
//
// Against the exact dictionary the fixed-point entry errs by at most
// 2^-49 (|B[p][i]| + |B[q][m]|) + 2^-97; the rounding into the double-float
// adds 2^-48 |c| at most.
#pragma once
#include <cstdint>

#include "df.cuh"

namespace aqmp {

constexpr int kSepFixBits = 48;                 // Bf = round(B 2^kSepFixBits)

// Normalise a nonzero 128-bit magnitude (ahi:alo) so that bit 127 is set and
// round its top 24 bits to nearest, ties to even: m (<= 2^24), e the index of
// the leading bit, lz the normalising shift, and the signed remainder in
// normalised units, (rhi:rlo) = n - m 2^104 with |rhi| <= 2^39.
__device__ __forceinline__ void round24(unsigned long long ahi, unsigned long long alo, unsigned long long &m,
                                        int &e, int &lz, long long &rhi, unsigned long long &rlo) {
    lz = ahi ? __clzll((long long)ahi) : 64 + __clzll((long long)alo);
    unsigned long long nhi, nlo;
    if (lz == 0) {
        nhi = ahi;
        nlo = alo;
    } else if (lz < 64) {
        nhi = (ahi << lz) | (alo >> (64 - lz));
        nlo = alo << lz;
    } else {
        nhi = alo << (lz - 64);
        nlo = 0ull;
    }
    e = 127 - lz;
    m = nhi >> 40;
    const unsigned long long r = nhi & ((1ull << 40) - 1), half = 1ull << 39;
    if (r > half || (r == half && (nlo != 0ull || (m & 1ull)))) ++m;
    rhi = (long long)(nhi - (m << 40));      // exact modulo 2^64, and in range
    rlo = nlo;
}

// m 2^k as a float for 2^23 <= m <= 2^24 and a normal result.
__device__ __forceinline__ float pow2_float(unsigned long long m, int k) {
    return __int_as_float(((k + 23 + 127) << 23) + (int)(m - (1ull << 23)));
}

// T 2^-96 as the double-float (RN(T), RN(T - RN(T))) scaled by 2^-96, ties to
// even: a function of T alone, ~2^-48 relative.  |T| < 2^112.  The general
// form, on the integer pipes: about 130 instructions, most of them variable
// 64-bit shifts.
static __device__ __noinline__ df int128_to_df_any(__int128 T) {
    if (T == 0) return df{0.0f, 0.0f};
    const bool neg = T < 0;
    const unsigned __int128 a = neg ? (unsigned __int128)(-T) : (unsigned __int128)T;
    const unsigned long long ahi = (unsigned long long)(a >> 64), alo = (unsigned long long)a;
    const int s96 = -2 * kSepFixBits;
    float hi, lo = 0.0f;
    if (ahi == 0ull && alo < (1ull << 24)) {
        hi = __fmul_rn((float)(unsigned)alo, __int_as_float((127 + s96) << 23));      // exact
    } else {
        unsigned long long m;
        int e, lz;
        long long rhi;
        unsigned long long rlo;
        round24(ahi, alo, m, e, lz, rhi, rlo);
        hi = pow2_float(m, e - 23 + s96);
        if (rhi != 0 || rlo != 0ull) {
            // |remainder| in normalised units, then rounded the same way and
            // scaled back by 2^-lz
            const bool rneg = rhi < 0;
            unsigned long long bhi = (unsigned long long)rhi, blo = rlo;
            if (rneg) {
                blo = ~rlo + 1ull;
                bhi = ~(unsigned long long)rhi + (blo == 0ull ? 1ull : 0ull);
            }
            unsigned long long m2;
            int e2, lz2;
            long long r2hi;
            unsigned long long r2lo;
            round24(bhi, blo, m2, e2, lz2, r2hi, r2lo);
            lo = pow2_float(m2, e2 - 23 - lz + s96);
            if (rneg) lo = -lo;
        }
    }
    return neg ? df{-hi, -lo} : df{hi, lo};
}

// s + e = a + b exactly, for |a| >= |b| or a = 0.
__device__ __forceinline__ float fast_sum(float a, float b, float &e) {
    const float s = __fadd_rn(a, b);
    e = __fadd_rn(b, -__fadd_rn(s, -a));
    return s;
}

// The same double-float, bit for bit, on the FP32 pipe: about 60 instructions.
// T is cut into five balanced 23-bit digits F_k (exact floats; a nonzero F_k
// exceeds the sum of those below it), which two sweeps of error-free sums
// turn into T = hi + lo + r + ge + (the error of q), hi and lo each the
// rounding of what it stands for.  That is certified: |lo| strictly below half
// a unit of hi, and so r with what is below it for lo (the comparisons widen
// them); or r alone, which rounds to even by itself when nothing is below it.
// Other values, near a tie, take the general form: none in 10^7 random
// integers above 2^65 (|c| > 2^-31), up to a fifth at 50 to 56 bits.
// Side 64, 50 910 leaves: the Haar family's kernel takes 0.85 ms with it and
// 1.50 with the general form alone.
constexpr unsigned long long kDigitBiasLo = (1ull << 22) | (1ull << 45);      // half a unit of each of the four
constexpr unsigned long long kDigitBiasHi = (1ull << 4) | (1ull << 27);       // lower digits, as 128 bits

// ... from the words of T + the digits' bias.
__device__ __forceinline__ df biased_to_df(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3) {
    static_assert(2 * kSepFixBits == 96, "digit weights");
    constexpr float kMid = 12582912.0f;             // 2^23 + 2^22: the digit 0 in the low mantissa bits
    auto digit = [&](uint32_t bits, float unit) {
        return __fmaf_rn(__uint_as_float((bits & 0x7fffffu) | 0x4B000000u), unit, -kMid * unit);
    };
    const float f0 = digit(w0, 0x1p-96f);
    const float f1 = digit(__funnelshift_r(w0, w1, 23), 0x1p-73f);
    const float f2 = digit(__funnelshift_r(w1, w2, 14), 0x1p-50f);
    const float f3 = digit(__funnelshift_r(w2, w3, 5), 0x1p-27f);
    const float f4 = __fmaf_rn(__uint_as_float(__funnelshift_r(w2, w3, 28) + 0x4B400000u), 0x1p-4f, -kMid * 0x1p-4f);
    float e0, e1, e2, e3, g0, g1, g2, ge, l1, r;
    const float a = fast_sum(f4, fast_sum(f3, fast_sum(f2, fast_sum(f1, f0, e0), e1), e2), e3);
    const float b = fast_sum(e3, fast_sum(e2, fast_sum(e1, e0, g0), g1), g2);
    const float q = __fadd_rn(g1, g0);
    const float G = fast_sum(g2, q, ge);
    const float hi = fast_sum(a, b, l1);
    float lo = fast_sum(l1, G, r);
    const float x = __fmaf_rn(fabsf(r), q == 0.0f ? 1.0f : 1.0f + 0x1p-18f, __fmaf_rn(fabsf(q), 0x1p-22f, fabsf(ge)));
    if (__builtin_expect(!(__fadd_rn(lo, x) == lo && __fadd_rn(lo, -x) == lo && __fmaf_rn(lo, 1.0f + 0x1p-20f, hi) == hi), 0)) {
        const unsigned long long tl = ((unsigned long long)w1 << 32) | w0, th = ((unsigned long long)w3 << 32) | w2;
        return int128_to_df_any((__int128)((((unsigned __int128)th << 64) | tl) -
                                           (((unsigned __int128)kDigitBiasHi << 64) | kDigitBiasLo)));
    }
    if (lo == 0.0f) lo = copysignf(0.0f, hi);       // as the general form
    return df{hi, lo};
}

__device__ __forceinline__ df int128_to_df(__int128 T) {
    const unsigned __int128 t = (unsigned __int128)T + (((unsigned __int128)kDigitBiasHi << 64) | kDigitBiasLo);
    return biased_to_df((uint32_t)t, (uint32_t)(t >> 32), (uint32_t)(t >> 64), (uint32_t)(t >> 96));
}

}  // namespace aqmp
