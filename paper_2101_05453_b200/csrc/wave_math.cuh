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

// floor(n / d) for n < 2^57, d < 2^26 and a quotient below 2^31; x: reciprocal estimate of d (relative error 2^-21 at most)
QL_HD uint32_t wv_div(uint64_t n, uint32_t d, float x)
{
    uint32_t q = (uint32_t)((float)n * x);                     // within 2^11
    int64_t r = (int64_t)(n - (uint64_t)q * d);
    const int32_t c = floor_s32((float)r * x);                 // then within 1 (rounded towards zero, a negative one could be 2 off)
    q += (uint32_t)c;
    r -= (int64_t)c * d;
    if (r < 0) { --q; r += d; }
    if (r >= (int64_t)d) ++q;
    return q;
}

QL_HD float wv_sqrt_est(float x)
{
#if defined(__CUDA_ARCH__)
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return __builtin_sqrtf(x);
#endif
}

// Statistics as ln_stats_fast (qmath.cuh) with a shorter chain: one thread per (row, gate) computes them while a group waits.
QL_HD WvLnRow wv_make_ln(int64_t sum, int64_t sumsq, const DivMagic &dn, uint32_t sigma_min)
{
    const uint64_t half = dn.n >> 1;
    const int32_t am = (int32_t)div_by_magic((uint64_t)(sum < 0 ? -sum : sum) * 1024u + half, dn);
    const int32_t mean = sum < 0 ? -am : am;
    const uint64_t q1 = div_by_magic((uint64_t)sumsq, dn);
    const uint64_t r1 = (uint64_t)sumsq - q1 * dn.n;
    int64_t var = (int64_t)((q1 << 20) + div_by_magic((r1 << 20) + half, dn)) - (int64_t)mean * mean;
    if (var < 0) var = 0;
    // integer root: fp32 estimate (within 2^4), one Newton step, exact correction
    uint32_t s = (uint32_t)wv_sqrt_est((float)var);
    const int64_t e = var - (int64_t)s * s;
    if (s) s += (uint32_t)(int32_t)(0.5f * (float)e * rcp_est((float)s));
    for (int i = 0; i < 2; ++i)
        if ((int64_t)s * s > var) --s;
    for (int i = 0; i < 2; ++i)
        if ((int64_t)(s + 1u) * (s + 1u) <= var) ++s;
    WvLnRow r;
    r.mean = mean; r.sigma = s; r.m_hi = 0; r.m_lo = 0;        // sigma = 0: the quotient is 0
    if (s >= sigma_min) {
        const float x = rcp_est((float)s);
        const uint32_t hi = wv_div((uint64_t)1 << 42, s, x);
        const uint32_t lo = wv_div((uint64_t)((1ull << 42) - (uint64_t)hi * s) << 31, s, x) + 1u;
        r.m_hi = (int32_t)(hi + (lo >> 31)); r.m_lo = (int32_t)(lo & 0x7fffffffu);
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
