// The integer evolution arithmetic (csrc/fixed64.cuh) compiled for the host, with
// the CUDA intrinsics that it uses written out, for tests/test_fixed_host.py.
#include <math.h>
#include <stdint.h>
#include <string.h>

#define __device__
#define __host__
#define __forceinline__ inline
static inline int __double2hiint(double x) { uint64_t b; memcpy(&b, &x, 8); return (int)(b >> 32); }
static inline int __double2loint(double x) { uint64_t b; memcpy(&b, &x, 8); return (int)(uint32_t)b; }
static inline double __hiloint2double(int h, int l)
{
    const uint64_t b = (uint64_t)(uint32_t)h << 32 | (uint32_t)l;
    double x;
    memcpy(&x, &b, 8);
    return x;
}
static inline uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, int s) { return (uint32_t)((((uint64_t)hi << 32 | lo) << s) >> 32); }
static inline int __mulhi(int a, int b) { return (int)(((int64_t)a * b) >> 32); }
static inline int __clz(int v) { return __builtin_clz((unsigned)v); }
static inline int __clzll(long long v) { return __builtin_clzll((unsigned long long)v); }
static inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b)
{
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
}
static inline float __frcp_rn(float x) { return 1.0f / x; }
template <class T> static inline T __ldg(const T *p) { return *p; }
static int g_skew;  // rsqrtf on the GPU is within 2 ulp: skewed either way here
static inline float rsqrtf(float x) { return (1.0f / sqrtf(x)) * (1.0f + 1.2e-7f * (float)(g_skew++ % 3 - 1)); }

#include "fixed64.cuh"

extern "C" void fixed_roots(int64_t n, const double *a, const double *b, double *root, double *inv, double *quot, int *ok)
{
    for (int64_t i = 0; i < n; ++i) {
        ok[i] = qed::fix_plain(b[i]);
        if (!ok[i]) continue;
        qed::fix_sqrt_double(b[i], root[i], inv[i]);
        quot[i] = qed::fix_div(a[i], b[i]);
    }
}

extern "C" void fixed_ln(int64_t n, const uint64_t *m, const int *e, double *out)
{
    for (int64_t i = 0; i < n; ++i) out[i] = qed::fix_ln(m[i], e[i]);
}

// n particles (rows px py pz ex ey ez bx by bz of p); the table of n_tab values on [chi_min, chi_max]
extern "C" void fixed_rates(int qs, int64_t n, const double *p, double chi_min, double chi_max, int n_tab,
                            const long long *ln_f, double *rate, double *ln_chi, double *chi,
                            int *ok)
{
    qed::FixAxis ax;
    const long double one = 9007199254740992.0L, l0 = logl(chi_min), l1 = logl(chi_max);
    ax.n = n_tab, ax.ok = 1, ax.shift = 0;
    ax.ln_min = (long long)rintl(l0 * one), ax.ln_max = (long long)rintl(l1 * one);
    const uint64_t d = (uint64_t)(ax.ln_max - ax.ln_min);
    int bits = 0;
    while ((n_tab - 1) >> bits) ++bits;
    while ((d << (ax.shift + 1)) < (1ull << 62)) ++ax.shift;
    ax.frac = 60 - bits;
    ax.scale = qed::fix_limbs(
        (int64_t)rintl((long double)(n_tab - 1) / ldexpl((long double)d, ax.shift) * ldexpl(1.0L, ax.frac + 62)));
    for (int64_t i = 0; i < n; ++i) {
        qed::FixOut o;
        ok[i] = qed::fix_particle(qs != 0, p[i], p[n + i], p[2 * n + i], p[3 * n + i], p[4 * n + i], p[5 * n + i],
                                  p[6 * n + i], p[7 * n + i], p[8 * n + i], ax, ln_f, kFixLogR, kFixLog,
                                  kFixExp, o);
        rate[i] = o.rate;
        ln_chi[i] = (double)o.ln_chi * 0x1p-53;
        chi[i] = sqrt(ldexp((double)o.s, o.s_e));
    }
}
