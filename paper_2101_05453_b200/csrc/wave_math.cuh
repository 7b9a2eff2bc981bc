// The wavefront kernels' own exact arithmetic: layer-norm statistics and quotients, and the piecewise-linear tables' lookup.  Host and
// device, like qmath.cuh, so that it is checked on a CPU against Python integers.
#pragma once
#include "qmath.cuh"

namespace ql {

// value of input x from its table entry e (act_table.cuh)
QL_HD int32_t act_line_value(int32_t e, int32_t x, int sh, int k)
{
    return (e + (((e & 1023) * (x & ((1 << sh) - 1))) << k)) >> 16;
}

// Layer-norm constants of one (row, gate).  The quotient q' = round(2^10 (2^10 q - mean) / sigma), ties away from zero, is
// floor(d M + 1/2) with d = 2^10 q - mean and M the next multiple of 2^-63 above 2^10 / sigma: strictly above, so that ties go
// outwards on both sides, and by so little (|d| < 2^26: 2^-37) that no other quotient, 1 / (2 sigma) > 2^-27 away from a tie, is
// moved across it.  M in two 31-bit limbs makes that two 32 x 32 + 64 multiply-adds whose high word is q': half the
// instructions of an estimate with a remainder test.  (fp64 would take one: but it shares its unit with the tensor core and
// took five times as long while MMAs ran.)
struct alignas(16) WvLnRow {
    int32_t m_hi, m_lo;            // 2^32 M = m_hi + 2^-31 m_lo
    int32_t mean;
    uint32_t sigma;                // top bit: quotients of this row may leave the fast range
};
constexpr uint32_t WV_LN_SLOW = 0x80000000u;

QL_HD int32_t floor_s32(float v)
{
#if defined(__CUDA_ARCH__)
    return __float2int_rd(v);
#else
    return (int32_t)__builtin_floorf(v);
#endif
}

// Estimates of the hardware.  On a CPU they are exact and are made as wrong as the hardware's may be (skew, relative).
#if !defined(__CUDA_ARCH__)
inline float &wv_skew() { static float v = 0.0f; return v; }
#endif
QL_HD float wv_rcp_est(float x)
{
#if defined(__CUDA_ARCH__)
    return rcp_est(x);
#else
    return 1.0f / x * (1.0f + wv_skew());
#endif
}
QL_HD float wv_sqrt_est(float x)
{
#if defined(__CUDA_ARCH__)
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return __builtin_sqrtf(x) * (1.0f + wv_skew());
#endif
}

QL_HD float wv_to_float(uint64_t v)                 // relative error 2^-23: two 32-bit conversions side by side, where one of 64 bits is several
{
    return fma_rn((float)(uint32_t)(v >> 32), 4294967296.0f, (float)(uint32_t)v);
}

// M for a sigma s >= 2^20 (see sigma_min), in two limbs: 2^42 / s and 2^31 times its remainder / s, plus one.
QL_HD void wv_limbs(uint32_t s, int32_t &m_hi, int32_t &m_lo)
{
    // x is the reciprocal within 2^-22: the first quotient is within 2, its remainder fits 32 bits (2^42 = 0 modulo 2^32)
    const float x = wv_rcp_est((float)s);
    uint32_t hi = (uint32_t)(4398046511104.0f * x);
    int32_t rem = (int32_t)(0u - hi * s);
    for (int i = 0; i < 2; ++i)
        if (rem < 0) { --hi; rem += (int32_t)s; }
    for (int i = 0; i < 2; ++i)
        if (rem >= (int32_t)s) { ++hi; rem -= (int32_t)s; }
    // the second within 2^10 at first; what is left is below 2^37 in magnitude, and 2^-8 of it within 32 bits
    uint32_t lo = (uint32_t)((float)rem * 2147483648.0f * x);
    const int64_t left = ((int64_t)rem << 31) - (int64_t)lo * s;
    const int32_t c = floor_s32((float)(int32_t)(left >> 8) * 256.0f * x);
    lo += (uint32_t)c;
    const int32_t last = (int32_t)((uint32_t)left - (uint32_t)c * s);
    if (last < 0) --lo;
    else if (last >= (int32_t)s) ++lo;
    ++lo;
    m_hi = (int32_t)(hi + (lo >> 31));
    m_lo = (int32_t)(lo & 0x7fffffffu);
}

// Statistics as ln_stats_fast (qmath.cuh) with a shorter chain: one thread per (row, gate) computes them while a group waits (alone in a
// warp 1350 cycles with 64-bit conversions and divisions throughout, 850 like this).
QL_HD WvLnRow wv_make_ln(int64_t sum, int64_t sumsq, const DivMagic &dn, uint32_t sigma_min)
{
    const uint64_t half = dn.n >> 1;
    const int32_t am = (int32_t)div_by_magic((uint64_t)(sum < 0 ? -sum : sum) * 1024u + half, dn);
    const int32_t mean = sum < 0 ? -am : am;
    const uint64_t q1 = div_by_magic((uint64_t)sumsq, dn);
    const uint64_t r1 = (uint64_t)sumsq - q1 * dn.n;
    int64_t var = (int64_t)((q1 << 20) + div_by_magic((r1 << 20) + half, dn)) - (int64_t)mean * mean;
    if (var < 0) var = 0;
    // integer root of var < 2^50: fp32 estimate s (relative error 2^-21: within 2^4), one Newton step s + floor(e / 2 s) with the exact
    // e = var - s^2 (|e| < 2^31).  The root is s + e / 2 s - k with 0 <= k < 1 (k < 2^7 / s; below s = 2^7 the estimate is within 1),
    // so that the step is within 1 of it.
    uint32_t s = (uint32_t)wv_sqrt_est(wv_to_float((uint64_t)var));
    const int32_t e = (int32_t)(var - (int64_t)s * s);
    if (s) s += (uint32_t)floor_s32(0.5f * (float)e * wv_rcp_est((float)s));
    const int64_t rest = var - (int64_t)s * s;
    if (rest < 0) --s;
    else if (rest > 2 * (int64_t)s) ++s;
    WvLnRow r;
    r.mean = mean; r.sigma = s; r.m_hi = 0; r.m_lo = 0;        // sigma = 0: the quotient is 0
    if (s >= sigma_min) {
        wv_limbs(s, r.m_hi, r.m_lo);
    } else if (s) {
        r.sigma |= WV_LN_SLOW;
    }
    return r;
}

QL_HD int32_t wv_ln_quotient(int32_t q, int32_t m_hi, int32_t m_lo, int32_t mean)
{
    const int32_t d = 1024 * q - mean;
    // the added 2^63 makes the low product's high word non-negative and is the 1/2 of the sum
    const uint64_t lo = (uint64_t)((int64_t)(2 * d) * m_lo) + 0x8000000000000000ull;
    return (int32_t)(((int64_t)d * m_hi + (int64_t)(lo >> 32)) >> 32);
}

}  // namespace ql
