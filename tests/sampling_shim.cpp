// The FP64 sampling, the optical-depth draws (csrc/physics.cuh) and the chi cut-offs (csrc/fixed64.cuh) compiled for the
// host, for tests/test_sampling_host.py and tests/test_cut_host.py.
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "device_shim.h"

#include "physics.cuh"

namespace qed {
int register_err_word(ErrWordIO) { return 0; }
}  // namespace qed

using namespace qed;

// as the library forms them from a table's parameters and entries (csrc/tables.cu)
static FixAxis axis(double lo, double hi, int n)
{
    FixAxis f;
    const long double one = 9007199254740992.0L;
    f.n = n, f.ok = 1, f.shift = 0;
    f.ln_min = (long long)rintl(logl(lo) * one), f.ln_max = (long long)rintl(logl(hi) * one);
    const uint64_t d = (uint64_t)(f.ln_max - f.ln_min);
    int bits = 0;
    while ((n - 1) >> bits) ++bits;
    while ((d << (f.shift + 1)) < (1ull << 62)) ++f.shift;
    f.frac = 60 - bits;
    f.scale = fix_limbs(
        (int64_t)rintl((long double)(n - 1) / ldexpl((long double)d, f.shift) * ldexpl(1.0L, f.frac + 62)));
    return f;
}

struct HostTable {
    std::vector<double> dv;
    std::vector<int32_t> guide;
    Table2D<double> t;
    HostTable(bool qs, int n_chi, int n_xi, double lo, double hi, double xi_min, const double *v)
        : dv((size_t)n_chi * n_xi), guide((size_t)n_chi * (kGuideBins + 1))
    {
        for (int i = 0; i < n_chi; ++i) {
            const double *row = v + (size_t)i * n_xi;
            for (int m = 0; m < n_xi; ++m) dv[(size_t)i * n_xi + m] = m + 1 < n_xi ? row[m + 1] - row[m] : 0.0;
            for (int e = 0; e <= kGuideBins; ++e) {
                const double x = qs ? std::log((double)e / kGuideBins) : (double)e / (2 * kGuideBins);
                const int m = (int)(std::upper_bound(row, row + n_xi, x) - row) - 1;
                guide[(size_t)i * (kGuideBins + 1) + e] = e == 0 ? 0 : e == kGuideBins ? n_xi - 1 : std::max(m, 0);
            }
        }
        t.v = v, t.dv = dv.data(), t.guide = guide.data();
        t.ln_min = std::log(lo), t.inv_d = (n_chi - 1) / (std::log(hi) - std::log(lo));
        t.chi_min = lo, t.chi_max = hi, t.n_chi = n_chi, t.n_xi = n_xi, t.pitch = n_xi;
        const double dx = qs ? -std::log(xi_min) / (n_xi - 1) : 0.5 / (n_xi - 1);
        t.x0 = qs ? std::log(xi_min) : 0.0, t.dx = dx;
        t.fix = axis(lo, hi, n_chi);
        t.dx_shift = 61 - std::ilogb(dx);
        t.dx_fix = fix_limbs((int64_t)std::ldexp(dx, t.dx_shift));
    }
};

// the photon's xi: by the integers (ok[i]: they took the draw), by the general form,
// and by the general form with the table-driven FP64 logarithm throughout
extern "C" void host_qs(int n_chi, int n_xi, double lo, double hi, double xi_min, const double *v, int64_t n,
                        const double *chi, const double *r, double *fixed, int *ok, double *general, double *tang)
{
    const HostTable h(true, n_chi, n_xi, lo, hi, xi_min, v);
    const Table2D<double> &t = h.t;
    for (int64_t i = 0; i < n; ++i) {
        fixed[i] = NAN;
        ok[i] = qs_sample_fixed(t, chi[i], r[i], fixed[i]);
        general[i] = qs_sample_row<double>(t, chi[i], r[i]);
        const double c = std::min(std::max(chi[i], lo), hi);
        const double p = std::min(std::max((log_tang(c) - t.ln_min) * t.inv_d, 0.0), n_chi - 1.0);
        const int k = std::min((int)p, n_chi - 2);
        const double w = p - k, lr = log_tang(r[i]), *r0 = v + (size_t)k * n_xi, *r1 = r0 + n_xi;
        const double *d0 = t.dv + (size_t)k * n_xi, *d1 = d0 + n_xi;
        int m = search_row(r0, r1, w, n_xi, lr, t.guide + (size_t)k * (kGuideBins + 1),
                           t.guide + (size_t)(k + 1) * (kGuideBins + 1),
                           std::min((int)(r[i] * kGuideBins), kGuideBins - 1));
        const double dp = row_val(d0, d1, w, m), x0 = t.x0 + m * t.dx, x1 = m + 1 == n_xi - 1 ? 0.0 : t.x0 + (m + 1) * t.dx;
        tang[i] = dp > 0.0 ? exp_tang(std::min(x0 + (lr - row_val(r0, r1, w, m)) * (x1 - x0) / dp, 0.0)) : exp_tang(x0);
    }
}

// -ln U of the Philox words (lo, hi): the draw, and the table-driven FP64 logarithm
extern "C" void host_draw(int64_t n, const uint32_t *lo, const uint32_t *hi, double *u, double *draw, double *tang)
{
    for (int64_t i = 0; i < n; ++i) {
        int64_t v;
        int unit;
        u[i] = uniform53(lo[i], hi[i]);
        draw[i] = neg_log_words<true>(U4{lo[i], hi[i], 0, 0}, v, unit) ? fix_to_double(v, unit) : neg_log1p_series(u[i]);
        tang[i] = u[i] > 1.0 - 0x1p-8 ? neg_log1p_series(u[i]) : -log_tang_core(u[i], 0);
    }
}

// ln cut in units of 2^-53, and ln chi values of those units against it (1 below, 2 near, 3 both)
extern "C" void host_cut(double cut, int64_t n, const int64_t *ln_chi, int64_t *ln_cut, int *side)
{
    *ln_cut = fix_ln_cut(cut, kFixLogR, kFixLog);
    for (int64_t i = 0; i < n; ++i) {
        const FixCut c = fix_cut(ln_chi[i], *ln_cut);
        side[i] = (c.below ? 1 : 0) + (c.near ? 2 : 0);
    }
}

// e^x and ln x of the rate lookups' FP64 form, and their table-driven forms
extern "C" void host_logexp(int64_t n, const double *x, double *e, double *e64, double *l, double *l64)
{
    for (int64_t i = 0; i < n; ++i) e[i] = r_exp(x[i]), e64[i] = exp_tang(x[i]), l[i] = r_log(x[i]), l64[i] = log_tang(x[i]);
}
