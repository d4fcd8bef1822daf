// physics.cuh -- per-particle device functions of the QED substep (templated on
// float / double): quantum parameters (§2), 1-D rate lookups (§3.1, §3.2),
// 2-D inverse-CDF sampling (§3.1, §3.2) and the optical-depth reset.
#pragma once

#include "common.cuh"
#include "fp64_math.cuh"

namespace qed {

__device__ __forceinline__ float d_log(float x) { return logf(x); }
__device__ __forceinline__ double d_log(double x) { return log(x); }
__device__ __forceinline__ float d_exp(float x) { return expf(x); }
__device__ __forceinline__ double d_exp(double x) { return exp(x); }
__device__ __forceinline__ float d_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double d_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float d_fma(float a, float b, float c) { return fmaf(a, b, c); }
// ln x on the integers (fixed64.cuh) for x in [2^-86, 2^86]; Tang's beyond
__device__ __forceinline__ double log_int(double x)
{
    const int hi = __double2hiint(x);
    if ((unsigned)(hi - (937 << 20)) >= (172u << 20)) return log_tang(x);  // (also zero, negative, NaN)
    const uint64_t m = (uint64_t)((hi & 0x000fffff) | 0x00100000) << 32 | (uint32_t)__double2loint(x);
    return fix_ln(m << 11, (hi >> 20) - 1023 - 63);
}

// e^x on the integers for |x| < 690 (one rounding of x to 2^-53, one of the result); Tang's beyond
__device__ __forceinline__ double exp_int(double x)
{
    if ((__double2hiint(x) & 0x7fffffff) >= 0x40859000) return exp_tang(x);  // (also infinite, NaN)
    int k;
    const int64_t m = fix_exp(fix_from_ln(x), k, kFixExp);
    return fix_to_double(m, k - 62);
}

// logarithm and exponential of the 1-D rate lookups: in FP32 the hardware's
// approximate forms (__logf: absolute error ~2^-21 near 1; __expf: ~2 + 1.2 |x|
// ulp), whose ~1e-6 relative effect on a rate is far below the tables'
// interpolation error; in FP64 (the form behind the integer one of fixed64.cuh) the
// integer logarithm and exponential, so that a particle that the integers gave up
// costs no more than it did before there were any
__device__ __forceinline__ float r_log(float x) { return __logf(x); }
__device__ __forceinline__ double r_log(double x) { return log_int(x); }
__device__ __forceinline__ float r_exp(float x) { return __expf(x); }
__device__ __forceinline__ double r_exp(double x) { return exp_int(x); }
__device__ __forceinline__ double d_fma(double a, double b, double c) { return fma(a, b, c); }
// square root, reciprocal square root and quotient of the event kernels: FP32 as
// they are; FP64 on the integers (fixed64.cuh) where the arguments are ordinary (an
// FP64 square root or division is ~10 FP64 instructions of 76 issue slots
// each), within 2^-58 before the last rounding, so that now and then the last
// bit differs from the IEEE operation's
__device__ __forceinline__ float e_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double e_sqrt(double x) { return fix_plain(x) ? fix_sqrt_double(x) : sqrt(x); }
__device__ __forceinline__ float e_div(float a, float b) { return a / b; }
__device__ __forceinline__ double e_div(double a, double b)
{
    return fix_plain(__longlong_as_double(__double_as_longlong(a) & 0x7fffffffffffffffll)) && fix_plain(b) ? fix_div(a, b)
                                                                                                          : a / b;
}
// |p| and 1/|p| (0 for p = 0) from p^2
__device__ __forceinline__ void e_norm(float p2, float &p, float &inv)
{
    p = sqrtf(p2);
    inv = p > 0.0f ? 1.0f / p : 0.0f;
}
__device__ __forceinline__ void e_norm(double p2, double &p, double &inv)
{
    if (fix_plain(p2)) {
        fix_sqrt_double(p2, p, inv);
    } else {
        p = sqrt(p2);
        inv = p2 > 0.0 ? rsqrt(p2) : 0.0;
    }
}

// logarithm and exponential of the 2-D inverse-CDF sampling: FP32 the library
// forms; the general FP64 forms the integer logarithm (ln chi and ln r are
// interpolation coordinates, where its 2^-62 absolute error near 1 is far below
// the tables' spacing) and Tang's exponential
__device__ __forceinline__ float s_log(float x) { return logf(x); }
__device__ __forceinline__ double s_log(double x) { return log_int(x); }
// and of the draw r itself: near r = 1, where ln r is small and decides the hardest
// photons' xi, by the series that the optical-depth resets take
static __device__ __noinline__ double neg_log1p_series(double u);
__device__ __forceinline__ float s_log_draw(float r) { return logf(r); }
__device__ __forceinline__ double s_log_draw(double r)
{
    return __double_as_longlong(r) > __double_as_longlong(1.0 - 0x1p-8) ? -neg_log1p_series(r) : log_int(r);
}
__device__ __forceinline__ float s_exp(float x) { return expf(x); }
__device__ __forceinline__ double s_exp(double x) { return exp_tang(x); }

// leading asymptotes of T outside the table (Eq. (t_func), read in the paper's
// chi_gamma convention): T ~ 3 sqrt(3) / (16 sqrt(2)) exp(-8 / (3 chi)) for
// small chi, T ~ C chi^{-1/3} with C = 15 3^{2/3} Gamma(2/3)^3 / (14 pi sqrt(3)
// Gamma(1/3)) for large chi.
constexpr double kTSmall = 0.22963966338592293;
constexpr double kTLarge = 0.37961230854357125;
constexpr double kLnTSmall = -1.4712438795175893;  // ln kTSmall
constexpr double kLnTLarge = -0.9686047877362934;  // ln kTLarge

// chi of a lepton, §2: chi^2 = (gamma E + p x B)^2 - (p.E)^2 in these units.
// FP32: with n = p/|p| and E_perp = E - (n.E) n the same quantity is the sum of
// squares |gamma E_perp + p x B|^2 + (n.E)^2 (expand gamma^2 = 1 + p^2 and use
// p x B perpendicular to n), which avoids the cancellation of the difference
// form when chi is small against gamma |E| + |p| |B|; a particle at rest has
// chi = |E|.  FP64 keeps the difference form: its cancellation error, 1e-16
// (S/chi)^2 relative, is below the FP64 tolerance, and it saves the FP64
// square root and division of n (as does the integer form that runs first,
// fixed64.cuh).
// The rate multiplies by 1/gamma.  FP64 takes gamma and 1/gamma from one
// reciprocal square root (within 1 ulp); FP32 keeps IEEE square roots and
// divisions here (with reciprocal square roots the HBM-bound evolution kernel
// measured ~1.5 % slower; photons, below, take them).
// Returns chi, gamma and 1/gamma; NaN inputs give NaN.
__device__ __forceinline__ float chi_lepton(float px, float py, float pz, float ex, float ey, float ez, float bx,
                                            float by, float bz, float &gamma, float &inv_gamma)
{
    const float p2 = px * px + py * py + pz * pz;
    gamma = sqrtf(1.0f + p2);
    inv_gamma = 1.0f / gamma;
    const float pm = sqrtf(p2);
    const float inv = pm > 0.0f ? 1.0f / pm : 0.0f;
    const float nx = px * inv, ny = py * inv, nz = pz * inv;
    const float ne = nx * ex + ny * ey + nz * ez;
    const float fx = gamma * (ex - ne * nx) + (py * bz - pz * by);
    const float fy = gamma * (ey - ne * ny) + (pz * bx - px * bz);
    const float fz = gamma * (ez - ne * nz) + (px * by - py * bx);
    const float s = fx * fx + fy * fy + fz * fz + (p2 > 0.0f ? ne * ne : ex * ex + ey * ey + ez * ez);
    return sqrtf(s);
}

__device__ __forceinline__ double chi_lepton(double px, double py, double pz, double ex, double ey, double ez,
                                             double bx, double by, double bz, double &gamma, double &inv_gamma)
{
    const double g2 = 1.0 + (px * px + py * py + pz * pz);
    inv_gamma = rsqrt(g2);
    gamma = g2 * inv_gamma;
    const double fx = gamma * ex + (py * bz - pz * by);
    const double fy = gamma * ey + (pz * bx - px * bz);
    const double fz = gamma * ez + (px * by - py * bx);
    const double pe = px * ex + py * ey + pz * ez;
    const double s = fx * fx + fy * fy + fz * fz - pe * pe;
    return sqrt(s < 0.0 ? 0.0 : s);  // (NaN stays NaN)
}

// chi_gamma of a photon, §2 (gamma -> |p|, v -> c n).  FP32: | |p| E_perp + p x B |,
// the perpendicular part of |p| E + p x B; FP64: the difference form.  Returns
// chi, |p| and 1/|p| (0 for p = 0), from a reciprocal square root (rsqrtf within
// 2 ulp, FP64 rsqrt within 1 ulp).
__device__ __forceinline__ float chi_photon(float px, float py, float pz, float ex, float ey, float ez, float bx,
                                            float by, float bz, float &pm, float &inv_pm)
{
    const float p2 = px * px + py * py + pz * pz;
    inv_pm = p2 > 0.0f ? rsqrtf(p2) : 0.0f;
    pm = p2 * inv_pm;
    const float nx = px * inv_pm, ny = py * inv_pm, nz = pz * inv_pm;
    const float ne = nx * ex + ny * ey + nz * ez;
    const float fx = pm * (ex - ne * nx) + (py * bz - pz * by);
    const float fy = pm * (ey - ne * ny) + (pz * bx - px * bz);
    const float fz = pm * (ez - ne * nz) + (px * by - py * bx);
    return sqrtf(fx * fx + fy * fy + fz * fz);
}

__device__ __forceinline__ double chi_photon(double px, double py, double pz, double ex, double ey, double ez,
                                             double bx, double by, double bz, double &pm, double &inv_pm)
{
    const double p2 = px * px + py * py + pz * pz;
    inv_pm = p2 > 0.0 ? rsqrt(p2) : 0.0;
    pm = p2 * inv_pm;
    const double fx = pm * ex + (py * bz - pz * by);
    const double fy = pm * ey + (pz * bx - px * bz);
    const double fz = pm * ez + (px * by - py * bx);
    const double pe = px * ex + py * ey + pz * ez;
    const double s = fx * fx + fy * fy + fz * fz - pe * pe;
    return sqrt(s < 0.0 ? 0.0 : s);
}

// The same in fields with only Ey and Bz (a linearly polarised wave along x), the
// terms with a zero factor left out (the compiler may not do that by itself): a
// product of a finite number and zero added to another number changes nothing
// but the sign of a zero, and every sum below is squared, so a finite
// particle's chi has the same bits, with the roundings as the full forms
// contract; a momentum component that is not finite still gives a chi that is not.
__device__ __forceinline__ float chi_lepton_yz(float px, float py, float pz, float ey, float bz, float &gamma,
                                               float &inv_gamma)
{
    const float p2 = px * px + py * py + pz * pz;
    gamma = sqrtf(1.0f + p2);
    inv_gamma = 1.0f / gamma;
    const float pm = sqrtf(p2);
    const float inv = pm > 0.0f ? 1.0f / pm : 0.0f;
    const float nx = px * inv, ny = py * inv, nz = pz * inv;
    const float ne = __fmul_rn(ny, ey);
    const float fx = fmaf(gamma, -__fmul_rn(ne, nx), __fmul_rn(py, bz));
    const float fy = fmaf(gamma, fmaf(-ne, ny, ey), -__fmul_rn(px, bz));
    const float fz = __fmul_rn(gamma, -__fmul_rn(ne, nz));
    const float s = fx * fx + fy * fy + fz * fz + (p2 > 0.0f ? ne * ne : ey * ey);
    return sqrtf(s);
}

__device__ __forceinline__ float chi_photon_yz(float px, float py, float pz, float ey, float bz, float &pm, float &inv_pm)
{
    const float p2 = px * px + py * py + pz * pz;
    inv_pm = p2 > 0.0f ? rsqrtf(p2) : 0.0f;
    pm = p2 * inv_pm;
    const float nx = px * inv_pm, ny = py * inv_pm, nz = pz * inv_pm;
    const float ne = __fmul_rn(ny, ey);
    const float fx = fmaf(pm, -__fmul_rn(ne, nx), __fmul_rn(py, bz));
    const float fy = fmaf(pm, fmaf(-ne, ny, ey), -__fmul_rn(px, bz));
    const float fz = __fmul_rn(pm, -__fmul_rn(ne, nz));
    return sqrtf(fx * fx + fy * fy + fz * fz);
}

// log-log interpolation of a 1-D table held in `tab` (shared or global):
// ln f(chi) = ln f_n + (ln chi - ln chi_n) (ln f_{n+1} - ln f_n) / (ln chi_{n+1} - ln chi_n),
// n = clamp(floor((ln chi - ln chi_min) / d), 0, N - 2); chi clamped into the table.
template <typename T>
__device__ __forceinline__ T interp_ln(const T *tab, T lc, T ln_min, T inv_d, int n)
{
    T t = (lc - ln_min) * inv_d;
    t = t < T(0) ? T(0) : (t > T(n - 1) ? T(n - 1) : t);
    int i = (int)t;
    i = i > n - 2 ? n - 2 : i;
    const T f = t - T(i);
    const T a = tab[i], b = tab[i + 1];
    return d_fma(f, b - a, a);
}

// QS rate (Eq. (qs_total_cross)): (2/3) alpha G(chi) / gamma; G clamped to the
// end values outside [chi_min, chi_max] (§3.2); chi == 0 gives 0.
template <typename T>
__device__ __forceinline__ T qs_rate(const T *tab, const Table1D<T> &v, T chi, T, T inv_gamma)
{
    if (!(chi > T(0))) return T(0);
    const T lnG = interp_ln(tab, r_log(chi), v.ln_min, v.inv_d, v.n);
    return T(2.0 / 3.0 * kAlpha) * r_exp(lnG) * inv_gamma;
}

// BW rate (Eq. (bw_cross_tot)): alpha chi T(chi) / gamma_g; the asymptotes of
// Eq. (t_func) outside [chi_min, chi_max] (§3.1).  All three branches give
// ln T, so a warp whose photons straddle the table's ends runs one exponential:
// ln T = ln(kTSmall) - 8 / (3 chi) below, ln(kTLarge) - (ln chi) / 3 above.
template <typename T>
__device__ __forceinline__ T bw_rate(const T *tab, const Table1D<T> &v, T chi, T pm, T inv_pm)
{
    if (!(chi > T(0)) || !(pm > T(0))) return T(0);
    const T lc = r_log(chi);
    T lnT;
    if (chi < v.chi_min)
        lnT = T(kLnTSmall) - T(8.0 / 3.0) / chi;
    else if (chi > v.chi_max)
        lnT = d_fma(lc, T(-1.0 / 3.0), T(kLnTLarge));
    else
        lnT = interp_ln(tab, lc, v.ln_min, v.inv_d, v.n);
    return T(kAlpha) * chi * r_exp(lnT) * inv_pm;
}

// uniform for sampling in the working precision: FP64 as drawn; FP32 rounded
// toward zero so that it stays in (0, 1)
template <typename T>
__device__ __forceinline__ T sample_uniform(double u);
template <>
__device__ __forceinline__ double sample_uniform<double>(double u) { return u; }
// FP32: u rounded toward zero, from the bits (u >= 2^-54 is a normal float;
// the same value as __double2float_rz without an FP64 instruction)
template <>
__device__ __forceinline__ float sample_uniform<float>(double u)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(u);
    return __uint_as_float((unsigned int)((((b >> 52) & 0x7ffu) - 1023u + 127u) << 23) |
                           (unsigned int)((b >> 29) & 0x7fffffu));
}

// 1 - u rounded toward zero to FP32 for a draw u in [1/2, 1] (the BW fold):
// 1 - u = (2^53 - M) 2^-53 exactly, M the 53-bit significand of u, then the
// top 24 bits of that integer
__device__ __forceinline__ float one_minus_rz(double u)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(u);
    if (b >= 0x3ff0000000000000ull) return 0.0f;                        // u = 1
    const unsigned long long n = (1ull << 53) - ((b & 0xfffffffffffffull) | (1ull << 52));  // u in [1/2, 1)
    const int len = 64 - __clzll((long long)n);                          // 1 .. 52
    const unsigned int mant = (unsigned int)(len > 24 ? n >> (len - 24) : n << (24 - len)) & 0x7fffffu;
    return __uint_as_float(((unsigned int)(len - 1 - 53 + 127) << 23) | mant);
}

// interpolated row value of a 2-D table at column m: v_n,m + w (v_{n+1},m - v_n,m)
template <typename T>
__device__ __forceinline__ T row_val(const T *r0, const T *r1, T w, int m)
{
    const T a = __ldg(r0 + m), b = __ldg(r1 + m);
    return d_fma(w, b - a, a);
}

// locate the chi interval of a 2-D table (chi clamped into the table, §3.1/§3.2);
// r0, r1 are the two rows, off their offset (for the difference table)
template <typename T>
__device__ __forceinline__ void locate_2d(const Table2D<T> &tb, T chi, const T *&r0, const T *&r1, T &w,
                                          size_t &off, int &row)
{
    T c = chi < tb.chi_min ? tb.chi_min : (chi > tb.chi_max ? tb.chi_max : chi);
    T t = (s_log(c) - tb.ln_min) * tb.inv_d;
    t = t < T(0) ? T(0) : (t > T(tb.n_chi - 1) ? T(tb.n_chi - 1) : t);
    int n = (int)t;
    n = n > tb.n_chi - 2 ? tb.n_chi - 2 : n;
    w = t - T(n);
    row = n;
    off = (size_t)n * tb.pitch;
    r0 = tb.v + off;
    r1 = r0 + tb.pitch;
}

// where the search of a row starts: the bracket that the guide tables of the two
// rows give for bin b of the draw (both rows' answers, hence the interpolated
// row's, lie between their guides at b and b + 1), widened by one entry on each
// side against rounding at the edges.  Invariant: P_lo <= x (or lo == 0), P_hi > x
// (hi == M: sentinel).
__device__ __forceinline__ void search_bracket(const int32_t *g0, const int32_t *g1, int b, int M, int &lo, int &hi)
{
    const int a0 = __ldg(g0 + b), a1 = __ldg(g1 + b), c0 = __ldg(g0 + b + 1), c1 = __ldg(g1 + b + 1);
    lo = (a0 < a1 ? a0 : a1) - 1, hi = (c0 > c1 ? c0 : c1) + 2;
    lo = lo < 0 ? 0 : lo;
    hi = hi > M ? M : hi;
}

// largest m in [0, M-1] with P_m <= x on the interpolated row (binary search;
// the row is non-decreasing), then clamped to [0, M-2]; m = 0 when x < P_0.
template <typename T>
__device__ __forceinline__ int search_row(const T *r0, const T *r1, T w, int M, T x, const int32_t *g0,
                                          const int32_t *g1, int b)
{
    int lo, hi;
    search_bracket(g0, g1, b, M, lo, hi);
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (row_val(r0, r1, w, mid) <= x)
            lo = mid;
        else
            hi = mid;
    }
    return lo > M - 2 ? M - 2 : lo;
}

// ---------------------------------------------------------------------------
// The FP64 inverse CDFs on 64-bit integers: chi's interval as in the rates, the
// draw and the row's values in one unit (BW: P and r in 2^-62; QS: ln P and ln r in
// 2^-58 to 2^-63), the quotient to 2^-58.  The general forms below take ~55 FP64 instructions
// of 76 issue slots each for an event, these none (2e6 photons all decaying, with the
// caller's ordering of the products: 727 -> 613 us).
// They return false, for the general forms: chi outside [2^-86, 2^86], a table that
// the units cannot hold, a draw off its row's ends or on a flat stretch, and small
// draws -- BW r < 2^-9 (1 in 256), where FP64 holds more than the unit does, QS
// r < 2^-20 --, QS r above 1 - 2^-15, where ln P and ln r are small and FP64 holds more of
// them (its error stays at 1e-15 with ln r by its series, the integers' is 1e-11 at 1 - 2^-30), and QS
// xi above e^(-1/8).
// ---------------------------------------------------------------------------
struct UnitBW {  // a value in [0, 1], rounded down; anything else: ok = false
    static __device__ __forceinline__ int64_t of(double x, int, bool &ok)
    {
        const uint32_t hi = (uint32_t)__double2hiint(x);
        ok = ok && hi <= 0x3ff00000u;  // (1 + a fraction below 2^-20 passes, and stays below 2^63)
        const uint64_t m = (uint64_t)((hi & 0x000fffffu) | 0x00100000u) << 32 | (uint32_t)__double2loint(x);
        return (int64_t)fix_shr(m << 10, 1023 - (int)(hi >> 20));  // (zero and subnormal values: 0)
    }
};
struct UnitQS {  // in 2^-(58 + s), +-2^(4 - s) for values beyond (ok = false)
    static __device__ __forceinline__ int64_t of(double x, int s, bool &ok)
    {
        const int hi = __double2hiint(x), d = 1026 - s - ((hi >> 20) & 0x7ff);
        const uint64_t m = (uint64_t)((hi & 0x000fffff) | 0x00100000) << 32 | (uint32_t)__double2loint(x);
        ok = ok && d >= 0;
        const int64_t v = d >= 0 ? (int64_t)fix_shr(m << 9, d) : (1ll << 62) - 1;
        return hi < 0 ? -v : v;
    }
};

template <typename U>
__device__ __forceinline__ int64_t fix_row(const double *r0, const double *r1, const Fix &w, int m, int s, bool &ok)
{
    const int64_t a = U::of(__ldg(r0 + m), s, ok), b = U::of(__ldg(r1 + m), s, ok);
    return a + mul_q62(w, fix_limbs(b - a));
}

// the column m of draw x (guide bin b) on the row at chi, and (x - P_m) / (P_{m+1} - P_m)
// in 2^-61.  Entries beyond the unit compare as its ends; rows do not decrease, so
// that they matter only where the columns at m hold one.
template <typename U>
__device__ __forceinline__ bool fix_column(const Table2D<double> &tb, double chi, int64_t x, int s, int b, int &m,
                                           int64_t &f)
{
    const int hi = __double2hiint(chi);
    bool ok = tb.fix.ok && (unsigned)(hi - (937 << 20)) < (172u << 20);
    if (!ok) return false;
    const uint64_t mc = (uint64_t)((hi & 0x000fffff) | 0x00100000) << 32 | (uint32_t)__double2loint(chi);
    int unit, row;
    const int64_t lc = fix_ln_value(mc << 11, (hi >> 20) - 1023 - 63, unit);
    const Fix w = fix_locate(tb.fix, unit == -63 ? (lc + 512) >> 10 : (lc + 8) >> 4, row);
    const double *r0 = tb.v + (size_t)row * tb.pitch, *r1 = r0 + tb.pitch;
    const int32_t *g0 = tb.guide + (size_t)row * (kGuideBins + 1), *g1 = g0 + kGuideBins + 1;
    b = b > kGuideBins - 1 ? kGuideBins - 1 : b;
    int hi_m;
    search_bracket(g0, g1, b, tb.n_xi, m, hi_m);
    bool any = true;
    while (hi_m - m > 1) {
        const int mid = (m + hi_m) >> 1;
        if (fix_row<U>(r0, r1, w, mid, s, any) <= x)
            m = mid;
        else
            hi_m = mid;
    }
    m = m > tb.n_xi - 2 ? tb.n_xi - 2 : m;
    const int64_t p0 = fix_row<U>(r0, r1, w, m, s, ok), dp = fix_row<U>(r0, r1, w, m + 1, s, ok) - p0, d = x - p0;
    if (!ok || d < 0 || d >= dp) return false;
    const int z = __clzll(dp) - 1;
    f = (int64_t)__umul64hi((uint64_t)d << z, fix_recip((uint64_t)dp << z));
    return true;
}

__device__ __forceinline__ bool bw_sample_fixed(const Table2D<double> &tb, double chi, double u, double &x)
{
    bool ok = true;
    int64_t r = UnitBW::of(u, 0, ok), f;
    r = r > (1ll << 61) ? (1ll << 62) - r : r;
    int m;
    if (!ok || r < (1ll << 53) || !fix_column<UnitBW>(tb, chi, r, 0, (int)(r >> 55), m, f)) return false;
    // (m + f) dx, rounded once
    const int k = 32 - __clz(m);
    const int64_t c = ((int64_t)m << (61 - k)) + (f >> k);
    if (c == 0) return false;
    const int z = __clzll(c) - 2;
    x = fix_to_double(mul_q62(fix_limbs(c << z), tb.dx_fix), 1 + k - z - tb.dx_shift);
    if (__double_as_longlong(x) > __double_as_longlong(0.5)) x = 0.5;
    return true;
}

__device__ __forceinline__ bool qs_sample_fixed(const Table2D<double> &tb, double chi, double r, double &xi)
{
    const int hi = __double2hiint(r);
    bool ok = true;
    const int64_t v = UnitBW::of(r, 0, ok);
    if (!ok || hi < 0x3eb00000 || hi >= 0x3fefffc0 || !tb.dx_shift) return false;  // 2^-20 <= r < 1 - 2^-15
    const uint64_t mr = (uint64_t)((hi & 0x000fffff) | 0x00100000) << 32 | (uint32_t)__double2loint(r);
    int unit, m, k;
    int64_t f;
    const int64_t lr = fix_ln_value(mr << 11, (hi >> 20) - 1023 - 63, unit);
    // the unit with |ln r|: 2^-58 below r = 1/2, up to 2^-63, so that it is finer than
    // FP64's roundings of ln P until the logarithm's own error is all there is
    const int z = __clzll(-lr), s = unit == -63 ? (z < 5 ? z : 5) : 0;
    if (!fix_column<UnitQS>(tb, chi, unit == -63 ? lr >> (5 - s) : 2 * lr, s, (int)(v >> 56), m, f)) return false;
    // ln xi = -(n - 1 - m - f) dx, 2^-53
    const int64_t c = ((int64_t)(tb.n_xi - 1 - m) << 52) - ((f + 256) >> 9);
    const int sh = tb.dx_shift - 63;
    const int64_t y = (mul_q62(fix_limbs(c), tb.dx_fix) + ((1ll << sh) >> 1)) >> sh;
    // near xi = 1 the lepton keeps gamma (1 - xi), a rounding of xi over 1 - xi: as before
    if (y < (1ll << 50)) return false;
    const int64_t e = fix_exp(-y, k, kFixExp);  // (its own statement: it sets k)
    xi = fix_to_double(e, k - 62);
    return true;
}
static_assert(kGuideBins == 64, "the guide's bin is the top 6 bits of r");

// QS inverse CDF (§3.2): ln P interpolated in ln chi, binary search on ln r, then
// ln xi = ln xi_m + (ln r - ln P_m)(ln xi_{m+1} - ln xi_m)/(ln P_{m+1} - ln P_m).
// The denominator is interpolated from the FP64-formed column differences, so
// that it keeps its relative accuracy in the FP32 tables (where two neighbouring
// entries share most of their digits); the same holds below xi_min, where the
// first segment is extrapolated.
template <typename T>
__device__ __forceinline__ T qs_sample_row(const Table2D<T> &tb, T chi, T r)
{
    const T *r0, *r1;
    T w;
    size_t off;
    int row;
    locate_2d(tb, chi, r0, r1, w, off, row);
    const T lr = s_log_draw(r);
    const int *g0 = tb.guide + (size_t)row * (kGuideBins + 1);
    int b = (int)(r * T(kGuideBins));
    b = b > kGuideBins - 1 ? kGuideBins - 1 : (b < 0 ? 0 : b);
    const int m = search_row(r0, r1, w, tb.n_xi, lr, g0, g0 + kGuideBins + 1, b);
    const T p0 = row_val(r0, r1, w, m);
    const T dp = row_val(tb.dv + off, tb.dv + off + tb.pitch, w, m);  // P_{m+1} - P_m
    const T x0 = tb.x0 + T(m) * tb.dx;
    const T x1 = (m + 1 == tb.n_xi - 1) ? T(0) : tb.x0 + T(m + 1) * tb.dx;
    if (!(dp > T(0))) return s_exp(x0);
    T lx = x0 + e_div((lr - p0) * (x1 - x0), dp);
    lx = lx > T(0) ? T(0) : lx;
    return s_exp(lx);
}

// (out of line: the few draws that the integer forms leave)
static __device__ __noinline__ double qs_sample_fp64(const Table2D<double> &tb, double chi, double r)
{
    return qs_sample_row<double>(tb, chi, r);
}

template <typename T>
__device__ __forceinline__ T qs_sample_xi(const Table2D<T> &tb, T chi, T r)
{
    if constexpr (sizeof(T) == 8) {
        double xi;
        return qs_sample_fixed(tb, chi, r, xi) ? xi : qs_sample_fp64(tb, chi, r);
    } else {
        return qs_sample_row<T>(tb, chi, r);
    }
}


// BW inverse CDF (§3.1): r <= 1/2 samples the electron, otherwise the positron
// with r -> 1 - r; P interpolated in ln chi_g, binary search on r, linear in xi
// (denominator from the column differences, as for QS).
template <typename T>
__device__ __forceinline__ T bw_sample_row(const Table2D<T> &tb, T chi, T r)
{
    const T *r0, *r1;
    T w;
    size_t off;
    int row;
    locate_2d(tb, chi, r0, r1, w, off, row);
    const int *g0 = tb.guide + (size_t)row * (kGuideBins + 1);
    int b = (int)(r * T(2 * kGuideBins));
    b = b > kGuideBins - 1 ? kGuideBins - 1 : (b < 0 ? 0 : b);
    const int m = search_row(r0, r1, w, tb.n_xi, r, g0, g0 + kGuideBins + 1, b);
    const T p0 = row_val(r0, r1, w, m);
    const T dp = row_val(tb.dv + off, tb.dv + off + tb.pitch, w, m);
    const T x0 = T(m) * tb.dx;
    const T x1 = (m + 1 == tb.n_xi - 1) ? T(0.5) : T(m + 1) * tb.dx;
    if (!(dp > T(0))) return x0;
    T x = x0 + e_div((r - p0) * (x1 - x0), dp);
    return x > T(0.5) ? T(0.5) : (x < T(0) ? T(0) : x);
}

static __device__ __noinline__ double bw_sample_fp64(const Table2D<double> &tb, double chi, double r)
{
    return bw_sample_row<double>(tb, chi, r);
}

template <typename T>
__device__ __forceinline__ T bw_sample_xi(const Table2D<T> &tb, T chi, double u, bool &electron)
{
    // split on the FP64 draw, then round the folded value (keeps 1 - u accurate)
    electron = __double_as_longlong(u) <= __double_as_longlong(0.5);  // u <= 1/2 (u > 0: the bits order as the values)
    if constexpr (sizeof(T) == 4) {
        return bw_sample_row<T>(tb, chi, electron ? sample_uniform<T>(u) : one_minus_rz(u));
    } else {
        double x;
        if (bw_sample_fixed(tb, chi, u, x)) return x;
        return bw_sample_fp64(tb, chi, electron ? u : 1.0 - u);
    }
}


// store an FP64 optical depth: FP64 as is; FP32 as (tau, tau_c) with tau_c the
// rounding residual (the optical depth is tau - tau_c)
template <typename T>
__device__ __forceinline__ void store_tau(T *tau, T *tau_c, int64_t i, double x);
template <>
__device__ __forceinline__ void store_tau<double>(double *tau, double *, int64_t i, double x) { tau[i] = x; }
// (h, c) = (fl32(x), fl32(h - x)), both rounded to nearest even.  Where both are
// normal floats (2^-74 <= |x| < 2^127) from the bits of x with integer
// operations, without an FP64 instruction (GB300's FP64 pipe bounds the event
// kernels when many particles fire): h keeps the top 24 of x's 53 significant
// bits, rounded; h - x is the rounding residual, an integer of at most 29 bits
// times 2^(e - 52), exact in FP64, rounded once by the integer-to-float
// conversion and scaled exactly.  Elsewhere (0, tiny, huge, infinite, NaN) by
// FP64 conversions, with the same results.
static __device__ __noinline__ float2 split_f32_pair_fp64(double x)  // (out of line: never predicated into the others)
{
    const float h = __double2float_rn(x);
    return make_float2(h, __double2float_rn((double)h - x));
}

__device__ __forceinline__ void split_f32_pair(double x, float &h, float &c)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7ffu) - 1023;
    if (e < -74 || e > 126) {
        const float2 p = split_f32_pair_fp64(x);
        h = p.x, c = p.y;
        return;
    }
    const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;  // 53 significant bits
    unsigned int keep = (unsigned int)(m >> 29);                                  // the top 24
    const unsigned int rem = (unsigned int)(m & 0x1fffffffu);                     // the other 29
    const bool up = rem > 0x10000000u || (rem == 0x10000000u && (keep & 1u));
    int diff = up ? (int)(0x20000000u - rem) : -(int)rem;  // (|h| - |x|) / 2^(e - 52)
    keep += up ? 1u : 0u;
    int eh = e;
    if (keep == 0x1000000u) {  // rounded up into the next binade
        keep >>= 1;
        ++eh;
    }
    const bool neg = (b >> 63) != 0;
    h = __uint_as_float((neg ? 0x80000000u : 0u) | ((unsigned int)(eh + 127) << 23) | (keep & 0x7fffffu));
    if (neg) diff = -diff;
    c = __int2float_rn(diff) * __uint_as_float((unsigned int)(e - 52 + 127) << 23);  // exact scaling by 2^(e - 52)
}

template <>
__device__ __forceinline__ void store_tau<float>(float *tau, float *tau_c, int64_t i, double x)
{
    float h, c;
    split_f32_pair(x, h, c);
    tau[i] = h;
    tau_c[i] = c;
}

// -ln U to FP64 for U in [2^-54, 1]: the integer logarithm (fixed64.cuh); above
// 1 - 2^-8, where ln U is small and that logarithm's error no longer shrinks
// with it, the Taylor series of log1p(d) with d = U - 1 (exact: U >= 1/2), whose
// remainder d^8/8 is below 2^-59 of the result.  The optical-depth resets were
// the event kernels' largest FP64 cost, and GB300's FP64 pipe their bound when
// many particles fire.
static __device__ __noinline__ double neg_log1p_series(double u)
{
    const double d = u - 1.0;
    double q = fma(d, -1.0 / 7, 1.0 / 6);
    q = fma(d, q, -0.2);
    q = fma(d, q, 0.25);
    q = fma(d, q, -1.0 / 3);
    q = fma(d, q, 0.5);
    return fma(d * d, q, -d);  // -(d - d^2/2 + d^3/3 - ... - d^7/7)
}

// -ln U = v 2^unit for the 53-bit uniform U of the words (uniform53: M 2^-k, M from
// the words' bits), without assembling U; false: U above 1 - 2^-8, by the series
template <bool F64>
__device__ __forceinline__ bool neg_log_words(const U4 &w, int64_t &v, int &unit)
{
    const uint64_t d = (((uint64_t)w.y << 32) | w.x) >> 11;
    const bool big = d >= (1ull << 52);
    const uint64_t m = big ? d + (d & 1ull) : 2ull * d + 1ull;
    const int lz = __clzll((long long)m), e = (big ? -53 : -54) - lz;
    const uint64_t n = m << lz;  // U = n 2^e
    if (e >= -64 && (e > -64 || (n >> 56) == 255)) return false;
    v = -(F64 ? fix_ln_value(n, e, unit) : fix_ln_48(n, e, unit));
    return true;
}

// tau = -ln U, U the 53-bit uniform of (seed, (id, step, purpose)), to FP64 (§3)
__device__ __forceinline__ double tau_draw(uint64_t seed, uint64_t id, int64_t step, uint32_t purpose)
{
    const U4 w = draw(seed, id, step, purpose);
    int64_t v;
    int unit;
    if (!neg_log_words<true>(w, v, unit)) return neg_log1p_series(uniform53(w.x, w.y));
    return fix_to_double(v, unit);
}

// (h, c) = (fl32(x), fl32(h - x)) of x = v 2^unit, v > 0 with x far inside the
// normal floats: the top 24 of v's bits, rounded to nearest even, and the residual
// (its upper 31 bits) by one integer-to-float conversion
__device__ __forceinline__ void split_fixed(int64_t v, int unit, float &h, float &c)
{
    const int lz = __clzll((long long)v);
    const uint64_t n = (uint64_t)v << lz, rem = n & 0xffffffffffull;  // the other 40
    unsigned int keep = (unsigned int)(n >> 40);
    const bool up = rem > 0x8000000000ull || (rem == 0x8000000000ull && (keep & 1u));
    const int64_t diff = up ? (int64_t)(0x10000000000ull - rem) : -(int64_t)rem;  // (h - x) / 2^(unit - lz)
    keep += up ? 1u : 0u;  // (2^24 carries into the exponent)
    const int e = unit - lz;
    h = __uint_as_float(((unsigned int)(e + 63 + 126) << 23) + keep);
    c = __int2float_rn((int)(diff >> 9)) * __uint_as_float((unsigned int)(e + 9 + 127) << 23);
}

// store tau = -ln U of (seed, (id, step, purpose)): FP64 as is, FP32 as the float pair
__device__ __forceinline__ void store_draw(double *tau, double *, int64_t i, uint64_t seed, uint64_t id, int64_t step,
                                           uint32_t purpose)
{
    tau[i] = tau_draw(seed, id, step, purpose);
}
__device__ __forceinline__ void store_draw(float *tau, float *tau_c, int64_t i, uint64_t seed, uint64_t id,
                                           int64_t step, uint32_t purpose)
{
    const U4 w = draw(seed, id, step, purpose);
    int64_t v;
    int unit;
    float h, c;
    if (neg_log_words<false>(w, v, unit))
        split_fixed(v, unit, h, c);
    else
        split_f32_pair(neg_log1p_series(uniform53(w.x, w.y)), h, c);
    tau[i] = h;
    tau_c[i] = c;
}

}  // namespace qed
