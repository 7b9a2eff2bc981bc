// Host build of the kernels' fixed-point arithmetic (qmath.cuh, wave_math.cuh) so that CPU-only tests can sweep it
// exhaustively.  Not part of libqlstm.so and not used by any product path.
#include "../qmath.cuh"
#include "../wave_math.cuh"

extern "C" {
int32_t qmh_mbqm(int32_t x, int32_t mult, int32_t shift) { return ql::mbqm(x, ql::Scale{mult, shift}); }
void qmh_mbqm_many(const int32_t *x, int n, int32_t mult, int32_t shift, int32_t *out)
{
    for (int i = 0; i < n; ++i) out[i] = ql::mbqm(x[i], ql::Scale{mult, shift});
}
void qmh_fast_rescale_many(const int32_t *x, int n, int32_t mult, int32_t shift, int32_t *out)
{
    ql::FastScale f = ql::make_fast_scale(ql::Scale{mult, shift});
    for (int i = 0; i < n; ++i) out[i] = ql::fast_rescale(x[i], f);
}
void qmh_sigmoid_fast_all(int m, int32_t *out) { for (int x = -32768; x < 32768; ++x) out[x + 32768] = ql::sigmoid_q_fast(x, m); }
void qmh_tanh_fast_all(int m, int32_t *out) { for (int x = -32768; x < 32768; ++x) out[x + 32768] = ql::tanh_q_fast(x, m); }
void qmh_layernorm_row_fast(const int16_t *q, int n, const int16_t *L, const int32_t *b, int32_t mult, int32_t shift, int16_t *out)
{
    int64_t s = 0, s2 = 0;
    for (int i = 0; i < n; ++i) { s += q[i]; s2 += (int64_t)q[i] * q[i]; }
    ql::LnRow r = ql::make_ln_row(ql::ln_stats(s, s2, n));
    ql::Scale sc{mult, shift};
    ql::FastScale f = ql::make_fast_scale(sc);
    for (int i = 0; i < n; ++i) out[i] = (int16_t)ql::ln_apply_fast(q[i], r, L[i], b[i], sc, f);
}
// the quotient alone, with hand-picked statistics (tiny sigma against large deviations)
int64_t qmh_ln_quotient_fast(int32_t q, int64_t mean, int64_t sigma)
{
    ql::LnStats st{mean, sigma};
    return ql::ln_quotient_fast(q, ql::make_ln_row(st));
}
int32_t qmh_cell_update_fast(int32_t i, int32_t z, int32_t f, int32_t c, int m) { return ql::cell_update_fast(i, z, f, c, m); }
int32_t qmh_hidden_fast(int32_t o, int32_t c, int m, int32_t mult, int32_t shift, int32_t zp)
{
    ql::Scale sc{mult, shift};
    return ql::hidden_q_fast(o, c, m, sc, ql::make_fast_scale(sc), zp);
}
uint64_t qmh_isqrt(uint64_t v) { return ql::isqrt64(v); }
uint64_t qmh_isqrt_from_f32(uint64_t v) { return ql::isqrt_from_f32(v); }
uint64_t qmh_div_by_magic(uint64_t x, uint32_t n) { return ql::div_by_magic(x, ql::make_div_magic(n)); }
void qmh_ln_stats(int64_t sum, int64_t sumsq, int n, int fast, int64_t *mean_sigma)
{
    ql::LnStats s = fast ? ql::ln_stats_fast(sum, sumsq, ql::make_div_magic((uint32_t)n)) : ql::ln_stats(sum, sumsq, n);
    mean_sigma[0] = s.mean; mean_sigma[1] = s.sigma;
}
// statistics of a row as the wavefront kernels form them: mean, sigma, whether the quotients need the division, and the limbs
void qmh_wave_ln(int64_t sum, int64_t sumsq, int n, uint32_t sigma_min, int64_t *out5)
{
    const ql::WvLnRow r = ql::wv_make_ln(sum, sumsq, ql::make_div_magic((uint32_t)n), sigma_min);
    out5[0] = r.mean; out5[1] = r.sigma & ~ql::WV_LN_SLOW; out5[2] = (r.sigma & ql::WV_LN_SLOW) != 0; out5[3] = r.m_hi; out5[4] = r.m_lo;
}
// quotients of many inputs with the limbs that wv_make_ln forms for a given sigma
void qmh_wave_quotients(const int32_t *q, int count, int32_t mean, uint32_t sigma, int32_t *out)
{
    int32_t hi, lo;
    ql::wv_limbs(sigma, hi, lo);
    for (int i = 0; i < count; ++i) out[i] = ql::wv_ln_quotient(q[i], hi, lo, mean);
}
void qmh_wave_limbs(uint32_t sigma, int32_t *out2) { ql::wv_limbs(sigma, out2[0], out2[1]); }
void qmh_wave_skew(float v) { ql::wv_skew() = v; }
int32_t qmh_line_value(int32_t e, int32_t x, int sh, int k) { return ql::act_line_value(e, x, sh, k); }
}
