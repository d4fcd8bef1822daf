// fixed64.cuh -- the FP64 evolution's chi and rate in 64-bit integer arithmetic.
//
// GB300 does two FP64 instructions per SM and clock (measured 1.68), 64 integer
// multiply-adds: a warp's FP64 instruction holds the pipe for as long as 76
// issue slots.  A 64 x 64-bit product takes three wide integer multiply-adds, so
// the quantum parameter, the logarithm, the table lookup and the exponential
// are done here on block-scaled 62-bit integers, and only the last
// multiply-add into the optical depth is an FP64 instruction.
//
// Accuracy: the force gamma E + p x B is formed to 2^-57 (typically 2^-59) of the
// blocks' scale |p| |F|, its squares to 2^-58, where FP64 rounds each term and
// each sum to 2^-53; the logarithms and the table values are held to 2^-53
// absolute, the exponential to 2^-58 relative.  What a block scale cannot hold
// -- a force more than 2^5 below |p| |F| where FP64 could hold it (fix_particle),
// subnormal blocks, infinities, NaN -- and values within rounding of a branch (the
// ends of a table, a cut-off) are left to the FP64 path by the caller.  Against
// extended precision chi and the rate are no less exact than the FP64 path's (the host
// tests of this file): in rms 1 to 3 times closer for beams across a field, 10 to 60 times
// closer for broad distributions and where the force nearly cancels.
//
// A block-scaled value is v 2^e, |v| < 2^62, as two signed limbs of v/4:
// v/4 = h 2^30 + l, |h| < 2^30, |l| < 2^30, so that products of limbs and sums
// of six of them stay inside a signed 64-bit accumulator.
#pragma once

#include <stdint.h>

#include "fixed_tables.h"

namespace qed {

struct Fix {
    int h, l;
};

// limbs of v/4 for |v| < 2^62 (floor: l >= 0)
__host__ __device__ __forceinline__ Fix fix_limbs(int64_t v)
{
    return Fix{(int)(v >> 32), (int)((uint32_t)v >> 2)};
}

// v >> d, 0 for d >= 64 (PTX clamps the amount)
__device__ __forceinline__ uint64_t fix_shr(uint64_t v, int d)
{
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(d));
    return r;
#else
    return d > 63 ? 0 : v >> d;
#endif
}

// a double on the block exponent eb (biased, the largest of its block): v 2^(eb - 1084);
// top: eb in the exponent's place with ones below it
__device__ __forceinline__ Fix fix_from(double x, int top)
{
    const int hi = __double2hiint(x);
    const uint32_t lo = (uint32_t)__double2loint(x);
    const int d = (top - (hi & 0x7fffffff)) >> 20;  // eb - the exponent
    const uint32_t mh = ((uint32_t)hi & 0x000fffffu) | 0x00100000u;
    // 53 bits << 9 (a zero or subnormal among larger values is shifted out: eb >= 128)
    const uint64_t v = fix_shr((uint64_t)__funnelshift_l(lo, mh, 9) << 32 | (lo << 9), d);
    const int s = (hi >> 31) | 1;
    return Fix{(int)(v >> 32) * s, (int)((uint32_t)v >> 2) * s};
}

__device__ __forceinline__ int64_t wide(int a, int b) { return (int64_t)a * b; }
__device__ __forceinline__ uint64_t uwide(uint32_t a, uint32_t b) { return (uint64_t)a * b; }

// sums of products (v/4)(w/4): h h' 2^60 + (h l' + l h') 2^30; l l' (below 2^60) is left out
struct Acc {
    int64_t hh, m;
};
__device__ __forceinline__ void mac(Acc &a, const Fix &x, const Fix &y)
{
    a.hh += wide(x.h, y.h);
    a.m += wide(x.h, y.l) + wide(x.l, y.h);
}
__device__ __forceinline__ void msc(Acc &a, const Fix &x, const Fix &y)
{
    const int h = -x.h, l = -x.l;
    a.hh += wide(h, y.h);
    a.m += wide(h, y.l) + wide(l, y.h);
}
// the sum in units of 2^60
__device__ __forceinline__ int64_t acc_value(const Acc &a) { return a.hh + (a.m >> 30); }

// x y / 2^62 for |x|, |y| < 2^62 with two guard bits (x y / 2^64 times 4)
__device__ __forceinline__ int64_t mul_q62(const Fix &x, const Fix &y)
{
    return 4 * wide(x.h, y.h) + ((wide(x.h, y.l) + wide(x.l, y.h)) >> 28);
}

// ---------------------------------------------------------------------------
// ln(n 2^e) / 2 in units of 2^-53 for n in [2^63, 2^64): (63 + e) ln2/2 + (ln m)/2,
// m = n / 2^63 in [1, 2).  u = m r_j - 1 with r_j ~ 1/c_j of 16 bits, c_j the
// centre of m's interval of width 1/256: exact to 2^-63, |u| < 2^-8.9; ln m =
// -ln r_j + u - u^2/2 + u^3/3 - ... - u^6/6 (the rest below 2^-64); the cubic
// tail is below 2^-28, its 28 bits leave 2^-56.  (Table-driven reduction after
// P. T. P. Tang, ACM TOMS 16 (1990) 378.)
// ---------------------------------------------------------------------------
__device__ __forceinline__ int64_t fix_half_ln(uint64_t n, int e, const int *tab_r, const long long *tab_ln)
{
    const int j = (int)(n >> 55) & 255;
    const uint32_t r = (uint32_t)tab_r[j];
    const int64_t u = (int64_t)((uwide((uint32_t)(n >> 32), r) << 17) + (uwide((uint32_t)n, r) >> 15));  // 2^-64
    const int a = (int)(u >> 25);                  // 2^-39
    const int b = (int)((uint32_t)u & 0x1ffffffu);  // 2^-64
    const int64_t h2 = (wide(a, a) + (wide(a, b) >> 24)) >> 15;  // u^2/2, 2^-64
    // t = 1/3 - u/4 + u^2/5 - u^3/6, 2^-31
    int t = 429496730 - (__mulhi(a, 357913941) >> 7);
    t = 536870912 - (__mulhi(a, t) >> 7);
    t = 715827883 - (__mulhi(a, t) >> 7);
    const int64_t c3 = wide((int)(h2 >> 16), __mulhi(a, t)) >> 21;  // u^3 t, 2^-64
    const int64_t l = tab_ln[j] + ((u - h2 + c3) >> 1);             // ln m, 2^-63
    const int k = 63 + e;
    return (wide(k, (int)(kHalfLn2 >> 32)) << 22) +
           ((wide(k, (int)((uint32_t)kHalfLn2 >> 1)) + (l >> 2) + 256) >> 9);  // one rounding (2^-62 to 2^-53)
}

// e^x = m 2^k for x in units of 2^-53, |x| < 800: m in [2^62, 2^63) but for its
// last bits.  x = (256 k + j) ln2/256 + r, |r| < 2^-9.4; e^r - 1 by its Taylor
// polynomial (r^6/720 < 2^-66).  (After Tang, ACM TOMS 15 (1989) 144.)
__device__ __forceinline__ int64_t fix_exp(int64_t x, int &k, const long long *tab)
{
    // n = round(x 256/ln2): the high word of x in 2^-21, kExpSteps in 2^-21; rounded at 2^-42
    const int n = (int)((wide((int)(x >> 32), kExpSteps) + (1ll << 41)) >> 42);
    const uint64_t nk = ((uint64_t)wide(n, (int)(kExpStep >> 32)) << 32) +
                        (uint64_t)((int64_t)n * (int64_t)(uint32_t)kExpStep) +
                        (uint64_t)(int64_t)(__mulhi(n, (int)(kExpStepLo >> 1)) * 2);
    const int64_t r = (int64_t)(((uint64_t)x << 11) - nk);  // 2^-64 (modulo 2^64)
    k = n >> 8;
    const int a = (int)(r >> 24);                   // 2^-40
    const int b = (int)((uint32_t)r & 0xffffffu);
    const int64_t h2 = (wide(a, a) + (wide(a, b) >> 23)) >> 17;  // r^2/2, 2^-64
    // t = 1/3 + r/12 + r^2/60, 2^-31
    int t = 178956971 + (__mulhi(a, 35791394) >> 8);
    t = 715827883 + (__mulhi(a, t) >> 8);
    const int64_t c3 = wide((int)(h2 >> 16), __mulhi(a, t)) >> 23;  // (r^2/2)(r t)
    const int64_t e1 = r + h2 + c3;                                  // e^r - 1, 2^-64, below 2^55
    const int64_t tj = tab[n & 255];
    const Fix ft{(int)(tj >> 32), (int)((uint32_t)tj >> 2)}, fe = fix_limbs(e1 << 6);
    return tj + ((wide(ft.h, fe.h) + ((wide(ft.h, fe.l) + wide(ft.l, fe.h)) >> 30)) >> 6);
}

// x in units of 2^-53 (to nearest) from its bits, |x| < 700
__device__ __forceinline__ int64_t fix_from_ln(double x)
{
    const int hi = __double2hiint(x), sh = 1032 - ((hi >> 20) & 0x7ff);  // the 53 bits << 11 have the unit 2^-63 at 2^9
    uint64_t m = ((uint64_t)((hi & 0x000fffff) | 0x00100000) << 32 | (uint32_t)__double2loint(x)) << 11;
    m = sh > 63 ? 0 : ((m >> sh) + 1) >> 1;
    return hi < 0 ? -(int64_t)m : (int64_t)m;
}

// sq = sqrt(g2 2^60) for g2 in [2^58, 2^62 - 2^58], to 1, and its reciprocal:
// 1/sqrt(g2 2^60) = inv 2^inv_e, inv in [2^62, 2^63], to 2^-59.  Newton steps on
// the integers from the 22-bit reciprocal square root.
__device__ __forceinline__ void fix_sqrt(uint64_t g2, int64_t &sq, uint64_t &inv, int &inv_e)
{
    const int s = (__clzll((long long)g2) & ~1) - 2;
    const uint64_t n = g2 << s;  // [2^60, 2^62): g and its estimates stay below 2^63
    const float nf = (float)(uint32_t)(n >> 32) * 0x1p-30f;
    const float y = rsqrtf(nf);
    const uint32_t g0 = (uint32_t)(nf * y * 0x1p31f);
    const int y0 = (int)fminf(y * 0x1p30f, 2147483520.0f);  // 2^-30, [1, 2)
    // g = sqrt(n) 2^32: the residuals n 2^64 - g^2, times y0/2
    const int64_t d0 = (int64_t)(n - uwide(g0, g0));
    const uint64_t g1 = ((uint64_t)g0 << 32) + (uint64_t)(wide((int)(d0 >> 11), y0) >> 19);
    const uint32_t gh = (uint32_t)(g1 >> 32), gl = (uint32_t)g1;
    const int64_t d1 = (int64_t)(((n - uwide(gh, gh)) << 32) - 2 * uwide(gh, gl) - (uwide(gl, gl) >> 32));
    const uint64_t g = g1 + (uint64_t)(wide((int)(d1 >> 22), y0) >> 40);  // [2^62, 2^63)
    sq = (int64_t)(g >> (s / 2 + 2));
    // 1/g: y (1 + e), e = 1 - g y (unit 2^-61, then 2^-93)
    const uint32_t fh = (uint32_t)(g >> 32), fl = (uint32_t)g;
    const int64_t e0 = (int64_t)((1ull << 61) - uwide(fh, (uint32_t)y0) - (uwide(fl, (uint32_t)y0) >> 32));
    const uint64_t y1 = ((uint64_t)y0 << 32) + (uint64_t)(wide(y0, (int)(e0 >> 10)) >> 19);  // 2^-62
    const uint32_t yh = (uint32_t)(y1 >> 32), yl = (uint32_t)y1;
    const int64_t e1 = -(int64_t)((uwide(fh, yh) << 32) + uwide(fh, yl) + uwide(fl, yh) + (uwide(fl, yl) >> 32));
    inv = y1 + (uint64_t)(wide((int)yh, (int)(e1 >> 21)) >> 40);
    inv_e = s / 2 + 2 - 125;  // 1/(g 2^-(s/2+2)) = (y 2^-62 2^-63) 2^(s/2+2)
}

// the double nearest to v 2^e for |v| < 2^63 (normal results; 0 for v = 0)
__device__ __forceinline__ double fix_to_double(int64_t v, int e)
{
    const uint64_t a = v < 0 ? 0 - (uint64_t)v : (uint64_t)v;
    if (a == 0) return 0.0;
    const int lz = __clzll((long long)a);
    const uint64_t n = a << lz;
    uint64_t t = n >> 11;
    const uint32_t rest = (uint32_t)n & 0x7ffu;
    t += rest > 0x400u || (rest == 0x400u && (t & 1)) ? 1 : 0;  // to nearest, ties to even (2^53 carries into the exponent)
    const uint64_t bits = ((uint64_t)(unsigned)(e - lz + 11 + 52 + 1022) << 52) + t;
    return __hiloint2double((int)(bits >> 32) | (v < 0 ? (int)0x80000000 : 0), (int)(uint32_t)bits);
}

// x = g 2^e with e even, g in [2^59, 2^61), for a positive normal x
__device__ __forceinline__ uint64_t fix_even(double x, int &e)
{
    const int hi = __double2hiint(x), be = hi >> 20;
    const uint64_t m = (uint64_t)((hi & 0x000fffff) | 0x00100000) << 32 | (uint32_t)__double2loint(x);
    const int s = be & 1 ? 8 : 7;  // be - 1075 - s is even
    e = be - 1075 - s;
    return m << s;
}

// whether x is positive, normal and within 2^+-500 (the integer forms below)
__device__ __forceinline__ bool fix_plain(double x)
{
    return (unsigned)(__double2hiint(x) - (523 << 20)) < (1000u << 20);
}

// sqrt(x) and 1/sqrt(x) for fix_plain(x): within 2^-59 before the rounding to FP64
__device__ __forceinline__ void fix_sqrt_double(double x, double &root, double &inv_root)
{
    int e, ie;
    const uint64_t g = fix_even(x, e);
    int64_t sq;
    uint64_t inv;
    fix_sqrt(g, sq, inv, ie);
    const int h = e / 2 - 30;  // sqrt(x) = sq 2^h
    root = fix_to_double(sq, h);
    inv_root = fix_to_double((int64_t)(inv >> 1), ie + 1 - h);  // (inv may be 2^63)
}

__device__ __forceinline__ double fix_sqrt_double(double x)
{
    double r, i;
    fix_sqrt_double(x, r, i);
    return r;
}

// 1/(g 2^-63) in 2^-62 for g in [2^62, 2^63), within 2^-58: two Newton steps from
// the 22-bit reciprocal (as in fix_sqrt)
__device__ __forceinline__ uint64_t fix_recip(uint64_t g)
{
    const uint32_t fh = (uint32_t)(g >> 32), fl = (uint32_t)g;
    const float y = __frcp_rn((float)fh * 0x1p-31f);
    const int y0 = (int)fminf(y * 0x1p30f, 2147483520.0f);  // 2^-30, [1, 2)
    const int64_t e0 = (int64_t)((1ull << 61) - uwide(fh, (uint32_t)y0) - (uwide(fl, (uint32_t)y0) >> 32));
    const uint64_t y1 = ((uint64_t)y0 << 32) + (uint64_t)(wide(y0, (int)(e0 >> 10)) >> 19);  // 2^-62
    const uint32_t yh = (uint32_t)(y1 >> 32), yl = (uint32_t)y1;
    const int64_t e1 = -(int64_t)((uwide(fh, yh) << 32) + uwide(fh, yl) + uwide(fl, yh) + (uwide(fl, yl) >> 32));
    return y1 + (uint64_t)(wide((int)yh, (int)(e1 >> 21)) >> 40);
}

// a / b for fix_plain(|a|), fix_plain(b): within 2^-58 before the rounding to
// FP64 (the reciprocal of b's significand times a's)
__device__ __forceinline__ double fix_div(double a, double b)
{
    const int ha = __double2hiint(a), hb = __double2hiint(b);
    const uint64_t ma = (uint64_t)((ha & 0x000fffff) | 0x00100000) << 32 | (uint32_t)__double2loint(a);
    const uint64_t mb = (uint64_t)((hb & 0x000fffff) | 0x00100000) << 32 | (uint32_t)__double2loint(b);
    const uint64_t inv = fix_recip(mb << 10);       // 1/(mb 2^-53), 2^-62
    const uint64_t p = __umul64hi(ma << 10, inv);  // (ma 2^-53)(2^53/mb) 2^61
    const int64_t q = (ha ^ hb) < 0 ? -(int64_t)p : (int64_t)p;
    return fix_to_double(q, ((ha >> 20) & 0x7ff) - ((hb >> 20) & 0x7ff) - 61);
}

// ln(n 2^e) = v 2^unit for n in [2^63, 2^64), |ln| < 62: the reduction of
// fix_half_ln over intervals of 1/1024 (|u| < 2^-10.9, so that the cubic tail's 30
// bits leave 2^-64): within 2^-62 absolute for arguments in [1/2, 2), where ln is
// small, and 2^-57, less than a sixteenth of an ulp of FP64, beyond.  No FP64
// instruction: one costs as much as 76 issue slots, this function ~60.
__device__ __forceinline__ int64_t fix_ln_value(uint64_t n, int e, int &unit)
{
    const int j = (int)(n >> 53) & 1023;
    const uint32_t r = __ldg(&kFineLogR[j]);
    const int64_t u = (int64_t)((uwide((uint32_t)(n >> 32), r) << 17) + ((uwide((uint32_t)n, r) + 16384) >> 15));  // 2^-64
    const int a = (int)(u >> 24);                   // 2^-40
    const int b = (int)((uint32_t)u & 0xffffffu);    // 2^-64
    const int64_t h2 = (wide(a, a) + (wide(a, b) >> 23)) >> 17;  // u^2/2, 2^-64
    int t = 536870912 - (__mulhi(a, 429496730) >> 8);            // 1/4 - u/5, 2^-31
    t = 1431655765 - (__mulhi(a, t) >> 7);                       // 1/3 - u/4 + u^2/5, 2^-32
    const int64_t c3 = wide((int)(h2 >> 11), (int)(wide(a, t) >> 29)) >> 31;  // u^3 t, 2^-64
    const int64_t l = __ldg(&kFineLog[j]) + ((u - h2 + c3 + 1) >> 1);         // ln m, 2^-63
    const int k = 63 + e;
    // k ln 2 + ln m in 2^-57, or in 2^-63 where k is 0 or -1
    const bool fine = k == 0 || k == -1;
    const int64_t kl = (wide(k, (int)(kHalfLn2 >> 32)) << 27) + (wide(k, (int)((uint32_t)kHalfLn2 >> 1)) >> 4);
    unit = fine ? -63 : -57;
    return fine ? (k ? l - kLn2 : l) : kl + ((l + 32) >> 6);
}

// The same over the 256 intervals of fix_half_ln, within 2^-57 absolute at every argument:
// of the FP32 path's optical depths, whose float pair holds 2^-48 (a pair's low word
// is a rounding residual, and a last-bit change of the logarithm can move it by 2^-12
// of itself a step later, so this form stays as it is).
__device__ __forceinline__ int64_t fix_ln_48(uint64_t n, int e, int &unit)
{
    const int j = (int)(n >> 55) & 255;
    const uint32_t r = (uint32_t)__ldg(&kFixLogR[j]);
    const int64_t u = (int64_t)((uwide((uint32_t)(n >> 32), r) << 17) + (uwide((uint32_t)n, r) >> 15));  // 2^-64
    const int a = (int)(u >> 25);                  // 2^-39
    const int b = (int)((uint32_t)u & 0x1ffffffu);  // 2^-64
    const int64_t h2 = (wide(a, a) + (wide(a, b) >> 24)) >> 15;  // u^2/2, 2^-64
    int t = 429496730 - (__mulhi(a, 357913941) >> 7);            // 1/3 - u/4 + u^2/5 - u^3/6, 2^-31
    t = 536870912 - (__mulhi(a, t) >> 7);
    t = 715827883 - (__mulhi(a, t) >> 7);
    const int64_t c3 = wide((int)(h2 >> 15), (int)(wide(a, t) >> 29)) >> 25;  // u^3 t, 2^-64
    const int64_t l = __ldg(&kFixLog[j]) + ((u - h2 + c3) >> 1);              // ln m, 2^-63
    const int k = 63 + e;
    // k ln 2 + ln m in 2^-57, or in 2^-63 where k is 0 or -1
    const bool fine = k == 0 || k == -1;
    const int64_t kl = (wide(k, (int)(kHalfLn2 >> 32)) << 27) + (wide(k, (int)((uint32_t)kHalfLn2 >> 1)) >> 4);
    unit = fine ? -63 : -57;
    return fine ? (k ? l - 2 * kHalfLn2 : l) : kl + (l >> 6);
}

__device__ __forceinline__ double fix_ln(uint64_t n, int e)
{
    int unit;
    const int64_t v = fix_ln_value(n, e, unit);
    return fix_to_double(v, unit);
}

// ---------------------------------------------------------------------------
// One process's 1-D rate table on the integers (filled by the host when the
// tables are made): logarithms in units of 2^-53.  ok: the axis fits.
// ---------------------------------------------------------------------------
struct FixAxis {
    long long ln_min, ln_max;  // of chi
    Fix scale;                 // (n - 1) / (ln_max - ln_min) of the shifted difference, see fix_table
    int shift, frac;           // of that difference; fraction bits of the table coordinate
    int n, ok;
};

constexpr long long kFixLnTSmall = -13251786775133077ll;  // ln of T's asymptotes (kLnTSmall, kLnTLarge), 2^-53
constexpr long long kFixLnTLarge = -8724416322236899ll;

// the interval of the axis at ln chi = lc (clamped into it) and the fraction of it, 2^-62
__device__ __forceinline__ Fix fix_locate(const FixAxis &ax, int64_t lc, int &i)
{
    int64_t d = lc - ax.ln_min;
    const int64_t dmax = ax.ln_max - ax.ln_min;
    d = d < 0 ? 0 : (d > dmax ? dmax : d);
    // t = d (n - 1) / dmax in units of 2^-frac (below 2^60): the difference shifted below 2^62 times the scale
    const int64_t t = mul_q62(fix_limbs(d << ax.shift), ax.scale);
    i = (int)(t >> ax.frac);
    i = i > ax.n - 2 ? ax.n - 2 : i;
    return fix_limbs((t - ((int64_t)i << ax.frac)) << (62 - ax.frac));
}

// the table's logarithms at ln chi = lc (clamped into the axis): ln f_i + f (ln f_{i+1} - ln f_i)
__device__ __forceinline__ int64_t fix_table(const FixAxis &ax, const long long *tab, int64_t lc)
{
    int i;
    const Fix f = fix_locate(ax, lc, i);
    const int64_t a = tab[i];
    return a + mul_q62(f, fix_limbs(tab[i + 1] - a));
}

// A chi cut-off on the integers: ln cut in units of 2^-53 (a particle's ln chi on the
// integers is within 333, 2^61.4 units); -2^62 where no particle is below it (no
// cut-off, or below e^-499), 2^62 where every one is (above e^499, infinite).
constexpr long long kFixFar = 1ll << 62;

__device__ __forceinline__ int64_t fix_ln_cut(double cut, const int *tab_r, const long long *tab_ln)
{
    const int hi = __double2hiint(cut);
    if (hi < (1023 - 720) << 20) return -kFixFar;  // (also negative)
    if (hi >= (1023 + 720) << 20) return kFixFar;
    const uint64_t m = (uint64_t)((hi & 0x000fffff) | 0x00100000) << 32 | (uint32_t)__double2loint(cut);
    return 2 * fix_half_ln(m << 11, (hi >> 20) - 1023 - 63, tab_r, tab_ln);
}

// ln chi against a cut-off: below: no evolution; near: within rounding of it, for the FP64 form to decide.
// (With every particle under a cut-off left to that form, 4e6 leptons took 705 us instead of 158,
// photons 748 instead of 164.)
struct FixCut {
    bool below, near;
};

__device__ __forceinline__ FixCut fix_cut(int64_t ln_chi, int64_t ln_cut)
{
    const int64_t d = ln_chi - ln_cut;
    return FixCut{d < 0, (uint64_t)(d + 1024) <= 2048ull};
}

struct FixOut {
    double rate;     // rate / coef: G(chi)/gamma, chi T(chi)/|p|
    int64_t ln_chi;  // 2^-53
    int64_t s;       // chi^2 = s 2^s_e
    int s_e;
};

// chi and the rate of one particle (§2, §3.1, §3.2; the difference form of
// chi^2, as the FP64 path).  false: the caller takes the FP64 path (the header).
__device__ __forceinline__ bool fix_particle(bool qs, double px, double py, double pz, double ex, double ey, double ez,
                                             double bx, double by, double bz, const FixAxis &ax, const long long *tab,
                                             const int *tab_r, const long long *tab_ln, const long long *tab_ex,
                                             FixOut &o)
{
    const auto mag_hi = [](double x) { return __double2hiint(x) & 0x7fffffff; };
    const auto imax = [](int a, int b) { return a > b ? a : b; };
    int ep = imax(imax(mag_hi(px), mag_hi(py)), mag_hi(pz)) >> 20;
    const int me = imax(imax(mag_hi(ex), mag_hi(ey)), mag_hi(ez));
    const int mf = imax(imax(me, mag_hi(bx)), imax(mag_hi(by), mag_hi(bz))), ef = mf >> 20;
    if (qs) ep = imax(ep, 1023);  // gamma^2 = 1 + p^2 on one scale
    // blocks within 2^+-400 (no infinity, NaN or subnormal, and no overflow that FP64 would see; a lepton's
    // momentum may be anything below 1, at rest too)
    bool ok = ax.ok && (unsigned)(ep - 623) <= 800u && (unsigned)(ef - 623) <= 800u;
    const int tp = ep << 20 | 0xfffff, tf = ef << 20 | 0xfffff;
    const Fix x = fix_from(px, tp), y = fix_from(py, tp), z = fix_from(pz, tp);
    Acc a{wide(x.h, x.h) + wide(y.h, y.h) + wide(z.h, z.h), wide(x.h, x.l) + wide(y.h, y.l) + wide(z.h, z.l)};
    uint64_t g2 = (uint64_t)(a.hh + (a.m >> 29));
    const int sh = 58 - 2 * (ep - 1023);
    if (qs && sh >= 0) g2 += 1ull << sh;
    g2 = ok ? g2 : 1ull << 60;
    int64_t sq;
    uint64_t inv;
    int inv_e;
    fix_sqrt(g2, sq, inv, inv_e);
    const Fix g{(int)(sq >> 30), (int)(sq & 0x3fffffff)};
    const Fix e0 = fix_from(ex, tf), e1 = fix_from(ey, tf), e2 = fix_from(ez, tf);
    const Fix b0 = fix_from(bx, tf), b1 = fix_from(by, tf), b2 = fix_from(bz, tf);
    Acc f0{0, 0}, f1{0, 0}, f2{0, 0}, pe{0, 0};
    mac(f0, g, e0), mac(f0, y, b2), msc(f0, z, b1);
    mac(f1, g, e1), mac(f1, z, b0), msc(f1, x, b2);
    mac(f2, g, e2), mac(f2, x, b1), msc(f2, y, b0);
    mac(pe, x, e0), mac(pe, y, e1), mac(pe, z, e2);
    const int64_t v0 = acc_value(f0), v1 = acc_value(f1), v2 = acc_value(f2), ve = acc_value(pe);
    const auto mag = [](int64_t v) { return (unsigned)((int)(v >> 32) ^ (int)(v >> 63)); };
    const unsigned top = mag(v0) | mag(v1) | mag(v2) | mag(ve);
    // The largest at least 2^-5 of the blocks' scale; 2^-26 where E is within 2^2 of the
    // largest field: there gamma E, whose rounding of gamma FP64 carries into the force
    // (2^-54.3 of the scale in rms), cancels against p x B in FP64 too.  (Without that
    // exception 4e6 leptons within 0.3 of a wave's direction paid both forms, 715 us
    // instead of 156, photons 815 instead of 183.)
    ok = ok && top >= (me >= mf - (2 << 20) ? 1u << 2 : 1u << 23);
    const int k = __clz((int)(top | 1u)) - 2;
    const Fix q0 = fix_limbs(v0 << k), q1 = fix_limbs(v1 << k), q2 = fix_limbs(v2 << k), qe = fix_limbs(ve << k);
    const int64_t s = wide(q0.h, q0.h) + wide(q1.h, q1.h) + wide(q2.h, q2.h) - wide(qe.h, qe.h) +
                      ((wide(q0.h, q0.l) + wide(q1.h, q1.l) + wide(q2.h, q2.l) - wide(qe.h, qe.l)) >> 29);
    ok = ok && s >= (1ll << 26);
    const uint64_t sp = s > 0 ? (uint64_t)s : 1ull;
    o.s = s;
    o.s_e = 2 * (ep + ef - k) - 4144;
    const int lz = __clzll((long long)sp);
    ok = ok && (unsigned)(o.s_e + 960) <= 1860u;  // chi^2 well inside the range of FP64
    const int64_t lc = fix_half_ln(sp << lz, o.s_e - lz, tab_r, tab_ln);
    o.ln_chi = lc;
    int64_t v;
    bool none = false;
    if (qs) {
        v = fix_table(ax, tab, lc);
    } else {
        // the ends of the table, where T jumps to its asymptotes, are decided by the FP64 path
        const auto close = [](int64_t d) { return (uint64_t)(d + 1024) <= 2048ull; };
        ok = ok && !close(lc - ax.ln_min) && !close(lc - ax.ln_max);
        if (lc < ax.ln_min) {
            int ke;
            const int64_t m = fix_exp(lc < -(700ll << 53) ? 700ll << 53 : -lc, ke, tab_ex) / 3;  // 1/(3 chi)
            none = ke > 7;  // 8/(3 chi) above 683: T below 1e-296
            v = lc + kFixLnTSmall - (none ? 0 : (ke >= 6 ? m << (ke - 6) : m >> (6 - ke > 63 ? 63 : 6 - ke)));
        } else if (lc > ax.ln_max) {
            v = lc + kFixLnTLarge - lc / 3;
        } else {
            v = lc + fix_table(ax, tab, lc);
        }
    }
    int ke;
    const int64_t m = fix_exp(v, ke, tab_ex);
    const uint64_t pr = __umul64hi((unsigned long long)m, inv);  // [2^59, 2^62]
    const int lr = __clzll((long long)pr);
    // the double nearest to pr 2^(64 + ke - 62 + inv_e) 2^-(ep - 1082)
    const int be = 64 + ke - 62 + inv_e - (ep - 1082) - lr + 11 + 52 + 1023;
    ok = ok && (none || (unsigned)(be - 2) <= 2040u);
    const uint64_t t = (((pr << lr) >> 10) + 1) >> 1;  // 53 bits, rounded (2^53: the carry moves into the exponent)
    const uint64_t bits = ((uint64_t)(unsigned)(be - 1) << 52) + t;
    o.rate = none ? 0.0 : __hiloint2double((int)(bits >> 32), (int)(uint32_t)bits);
    return ok;
}

}  // namespace qed
