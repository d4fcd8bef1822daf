// evolve_core.cuh -- the per-particle optical-depth evolution (chi, rate
// lookup, decrement, warp-ballot compaction of the firing particles) on values
// already in registers, and the 16-byte vector loads/stores of the particle
// arrays; shared by the evolution kernels and the fused push + evolution.
#pragma once

#include "evolve.cuh"
#include "physics.cuh"

namespace qed {

template <typename T, int VEC>
struct Vec;
template <>
struct Vec<float, 4> {
    using type = float4;
};
template <>
struct Vec<float, 2> {
    using type = float2;
};
template <>
struct Vec<double, 2> {
    using type = double2;
};

template <typename T, int VEC>
__device__ __forceinline__ void load_vec(const T *p, int64_t i, T (&out)[VEC])
{
    if constexpr (VEC == 1) {
        out[0] = __ldcs(p + i);
    } else {
        using V = typename Vec<T, VEC>::type;
        const V v = __ldcs(reinterpret_cast<const V *>(p + i));
        if constexpr (VEC == 4) {
            out[0] = v.x, out[1] = v.y, out[2] = v.z, out[3] = v.w;
        } else {
            out[0] = v.x, out[1] = v.y;
        }
    }
}

template <typename T, int VEC>
__device__ __forceinline__ void store_vec(T *p, int64_t i, const T (&in)[VEC])
{
    if constexpr (VEC == 1) {
        __stcs(p + i, in[0]);
    } else {
        using V = typename Vec<T, VEC>::type;
        V v;
        if constexpr (VEC == 4) {
            v.x = in[0], v.y = in[1], v.z = in[2], v.w = in[3];
        } else {
            v.x = in[0], v.y = in[1];
        }
        __stcs(reinterpret_cast<V *>(p + i), v);
    }
}

// The 1-D rate tables of both processes in shared memory: FP32 as they are, FP64
// as 64-bit integers (units of 2^-53) with the tables of the integer logarithm
// and exponential (fixed64.cuh).
template <typename T>
struct RateSmem;
template <>
struct RateSmem<float> {
    float qs[QED_MAX_TABLE_N], bw[QED_MAX_TABLE_N];
};
template <>
struct RateSmem<double> {
    long long qs[QED_MAX_TABLE_N], bw[QED_MAX_TABLE_N];
    long long ln[256], ex[256];
    int r[256];
    int off[2];  // per process: nonzero if a value or a step of its table does not fit the integers
    double coef_dt[2];  // per process: the rate's constant factor times dt
    long long ln_cut[2];  // per process: its chi cut-off (fix_ln_cut)
};

__device__ __forceinline__ void stage_rates(RateSmem<float> &s, const TablesView<float> &tab, float, float, float,
                                            int threads)
{
    for (int i = threadIdx.x; i < tab.qs_G.n; i += threads) s.qs[i] = tab.qs_G.ln_f[i];
    for (int i = threadIdx.x; i < tab.bw_T.n; i += threads) s.bw[i] = tab.bw_T.ln_f[i];
}

// the table on integers; nonzero where it does not fit: |ln f| < 700, steps below 500
__device__ __forceinline__ int stage_fix(long long *out, const Table1D<double> &t, int threads)
{
    const auto below = [](double x, int hi_limit) { return (__double2hiint(x) & 0x7fffffff) < hi_limit; };
    int off = 0;
    for (int i = threadIdx.x; i < t.n; i += threads) {
        const double x = t.ln_f[i];
        off |= below(x, 0x4085e000) ? 0 : 1;                                  // 700
        if (i + 1 < t.n) off |= below(t.ln_f[i + 1] - x, 0x407f4000) ? 0 : 1;  // 500
        out[i] = fix_from_ln(x);
    }
    return off;
}

// every thread of the CTA; the caller's next barrier publishes it
__device__ __forceinline__ void stage_rates(RateSmem<double> &s, const TablesView<double> &tab, double dt, double cut_qs,
                                            double cut_bw, int threads)
{
    if (threadIdx.x < 2) {
        s.off[threadIdx.x] = 0, s.coef_dt[threadIdx.x] = (threadIdx.x ? kAlpha : 2.0 / 3.0 * kAlpha) * dt;
        s.ln_cut[threadIdx.x] = fix_ln_cut(threadIdx.x ? cut_bw : cut_qs, kFixLogR, kFixLog);
    }
    __syncthreads();
    if (stage_fix(s.qs, tab.qs_G, threads)) s.off[0] = 1;
    if (stage_fix(s.bw, tab.bw_T, threads)) s.off[1] = 1;
    for (int i = threadIdx.x; i < 256; i += threads) s.ln[i] = kFixLog[i], s.ex[i] = kFixExp[i], s.r[i] = kFixLogR[i];
}

// the FP32 decrement of one particle's optical depth by its rate; returns fire
__device__ __forceinline__ bool decrement(float chi, float rate, float dt, float cut, float &tau, float &tc,
                                          float &chi_out, int &bad)
{
    const bool ok = isfinite(chi) && !isnan(tau) && isfinite(rate);
    bad += ok ? 0 : 1;
    if (!ok || chi < cut) rate = 0.0f;  // below the process's chi threshold: no evolution
    chi_out = chi;
    // Kahan-compensated decrement; tau - tc is the optical depth
    if (!isfinite(tau)) return false;  // removed particle (tau = +inf)
    const float y = d_fma(-rate, dt, -tc);
    const float t = tau + y;
    tc = (t - tau) - y;
    tau = t;
    return ok && (t < 0.0f || (t == 0.0f && tc > 0.0f));
}

// one particle in the linearly polarised wave's fields (Ey, Bz)
__device__ __forceinline__ bool evolve_one_yz(int proc, const RateSmem<float> &rs, const TablesView<float> &tv,
                                              float px, float py, float pz, float ey, float bz, float dt, float cut,
                                              float &tau, float &tc, float &chi_out, int &bad)
{
    float chi, rate, en, inv;
    if (proc == QED_PROC_QS) {
        chi = chi_lepton_yz(px, py, pz, ey, bz, en, inv);
        rate = qs_rate(rs.qs, tv.qs_G, chi, en, inv);
    } else {
        chi = chi_photon_yz(px, py, pz, ey, bz, en, inv);
        rate = bw_rate(rs.bw, tv.bw_T, chi, en, inv);
    }
    return decrement(chi, rate, dt, cut, tau, tc, chi_out, bad);
}

// one particle: chi, rate, optical-depth decrement; returns fire
__device__ __forceinline__ bool evolve_one(int proc, const RateSmem<float> &rs, const TablesView<float> &tv, float px,
                                           float py, float pz, float ex, float ey, float ez, float bx, float by,
                                           float bz, float dt, float cut, float &tau, float &tc, float &chi_out,
                                           int &bad)
{
    float chi, rate;
    if (proc == QED_PROC_QS) {
        float gamma, inv;
        chi = chi_lepton(px, py, pz, ex, ey, ez, bx, by, bz, gamma, inv);
        rate = qs_rate(rs.qs, tv.qs_G, chi, gamma, inv);
    } else {
        float pm, inv;
        chi = chi_photon(px, py, pz, ex, ey, ez, bx, by, bz, pm, inv);
        rate = bw_rate(rs.bw, tv.bw_T, chi, pm, inv);
    }
    return decrement(chi, rate, dt, cut, tau, tc, chi_out, bad);
}

struct EvolvedFp64 {
    double tau, chi;
    int fire, bad;
};

// The same with chi and the interpolation in FP64, out of line: the particles that the
// integers of fixed64.cuh leave to it (blocks of subnormal or huge values, infinities,
// NaN, a force far below its terms, chi within rounding of a table's end or of the
// cut-off).  They pay both forms: 4e6 leptons along a static B 526 us, photons 677 (in FP64
// instructions throughout 705 and 838, and 603 and 730 without the integers ahead).
static __device__ __noinline__ EvolvedFp64 evolve_one_fp64(int proc, const Table1D<double> &tb, double px, double py,
                                                           double pz, double ex, double ey, double ez, double bx,
                                                           double by, double bz, double dt, double cut, double tau)
{
    double chi, rate, en, inv;
    if (proc == QED_PROC_QS) {
        chi = chi_lepton(px, py, pz, ex, ey, ez, bx, by, bz, en, inv);
        rate = qs_rate(tb.ln_f, tb, chi, en, inv);
    } else {
        chi = chi_photon(px, py, pz, ex, ey, ez, bx, by, bz, en, inv);
        // (below chi = 0.0035, e^(-8/(3 chi)) is zero in FP64: photons straight along a wave, 4e6 of them
        // 674 us with the logarithm and the exponential of it)
        rate = chi < 0.0035 && chi < tb.chi_min ? 0.0 : bw_rate(tb.ln_f, tb, chi, en, inv);
    }
    const bool ok = isfinite(chi) && !isnan(tau) && isfinite(rate);
    if (!ok || chi < cut) rate = 0.0;  // below the process's chi threshold: no evolution
    tau = tau - rate * dt;
    return EvolvedFp64{tau, chi, ok && tau < 0.0, ok ? 0 : 1};
}

__device__ __forceinline__ bool evolve_one(int proc, const RateSmem<double> &rs, const TablesView<double> &tv,
                                           double px, double py, double pz, double ex, double ey, double ez, double bx,
                                           double by, double bz, double dt, double cut, double &tau, double &,
                                           double &chi_out, int &bad)
{
    const bool qs = proc == QED_PROC_QS;
    const Table1D<double> &tb = qs ? tv.qs_G : tv.bw_T;
    FixOut o;
    bool fast = fix_particle(qs, px, py, pz, ex, ey, ez, bx, by, bz, tb.fix, qs ? rs.qs : rs.bw, rs.r, rs.ln, rs.ex, o);
    // (tau = 0 or NaN: a rate that the integers drop as below 1e-290 could decide)
    const long long tb_bits = __double_as_longlong(tau) & 0x7fffffffffffffffll;
    const FixCut at = fix_cut(o.ln_chi, rs.ln_cut[qs ? 0 : 1]);
    fast = fast && rs.off[qs ? 0 : 1] == 0 && tb_bits != 0 && tb_bits <= 0x7ff0000000000000ll && !at.near;
    if (!fast) {
        const auto mag = [](double x) { return __double_as_longlong(x) & 0x7fffffffffffffffll; };
        const long long inf = 0x7ff0000000000000ll;
        if (!(mag(ex) | mag(ey) | mag(ez) | mag(bx) | mag(by) | mag(bz)) && mag(px) < inf && mag(py) < inf &&
            mag(pz) < inf && tb_bits <= inf) {  // no field: chi = 0, nothing evolves
            chi_out = 0.0;
            return __double_as_longlong(tau) < 0 && tb_bits != 0;
        }
        const EvolvedFp64 r = evolve_one_fp64(proc, tb, px, py, pz, ex, ey, ez, bx, by, bz, dt, cut, tau);
        tau = r.tau, chi_out = r.chi;
        bad += r.bad;
        return r.fire != 0;
    }
    // the only FP64 instruction: tau - (rate / coef) (coef dt)
    tau = fma(at.below ? 0.0 : -o.rate, rs.coef_dt[qs ? 0 : 1], tau);
    const bool fire = __double_as_longlong(tau) < 0 && __double_as_longlong(tau) != (long long)0x8000000000000000ull;
    if (fire) chi_out = sqrt(scalbn((double)o.s, o.s_e));
    return fire;
}

// warp-ballot compaction of the firing particles among [i0, i0 + VEC) (cnt of
// them in this thread) into the segment's firing list: one atomic per warp
template <typename T, int VEC>
__device__ __forceinline__ void compact_fire(const EvolveSeg<T> &sg, int64_t i0, const bool (&fire)[VEC],
                                             const T (&chi)[VEC], int cnt, long long *stats)
{
    if (!__ballot_sync(0xffffffffu, cnt > 0)) return;
    const unsigned lane = threadIdx.x & 31u;
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)lane >= o) incl += v;
    }
    const int wtot = __shfl_sync(0xffffffffu, incl, 31);
    unsigned long long base = 0;
    if (lane == 31) base = atomicAdd(sg.fire_count, (unsigned long long)wtot);
    base = __shfl_sync(0xffffffffu, base, 31);
    long long pos = (long long)base + incl - cnt;
    int over = 0;
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
        if (fire[j]) {
            if (pos < sg.fire_cap) {
                sg.fire_idx[pos] = i0 + j;
                sg.fire_chi[pos] = (double)chi[j];
            } else {
                ++over;
            }
            ++pos;
        }
    }
    warp_count_err(stats ? stats + QED_STAT_FIRE_OVERFLOW : nullptr, over, QED_EW_FIRE_OVERFLOW);
}

// Evaluate, store and compact VEC particles [i0, i0 + VEC) of segment `sg`
// whose inputs are already in registers (full: all VEC are live).  dry != 0
// evaluates everything but stores nothing (used by the launch-shape tuner).
template <typename T, int VEC>
__device__ __forceinline__ void evolve_regs(const EvolveSeg<T> &sg, int64_t n, int64_t i0, bool full,
                                            const T (&px)[VEC], const T (&py)[VEC], const T (&pz)[VEC],
                                            const T (&ex)[VEC], const T (&ey)[VEC], const T (&ez)[VEC],
                                            const T (&bx)[VEC], const T (&by)[VEC], const T (&bz)[VEC], T (&tau)[VEC],
                                            T (&tc)[VEC], const RateSmem<T> &rs, const TablesView<T> &tab,
                                            T dt, T cut, long long *stats, int dry, int &bad)
{
    bool fire[VEC];
    T chi[VEC];
    int cnt = 0;
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
        T c = sizeof(T) == 4 ? tc[j] : T(0);
        fire[j] = evolve_one(sg.proc, rs, tab, px[j], py[j], pz[j], ex[j], ey[j], ez[j], bx[j], by[j],
                                bz[j], dt, cut, tau[j], c, chi[j], bad);
        tc[j] = c;
        fire[j] = fire[j] && (i0 + j < n);
        cnt += fire[j] ? 1 : 0;
    }
    if (dry) return;

    if (full) {
        store_vec<T, VEC>(sg.tau, i0, tau);
        if constexpr (sizeof(T) == 4) store_vec<T, VEC>(sg.tau_c, i0, tc);
    } else {
#pragma unroll
        for (int j = 0; j < VEC; ++j) {
            if (i0 + j < n) {
                sg.tau[i0 + j] = tau[j];
                if constexpr (sizeof(T) == 4) sg.tau_c[i0 + j] = tc[j];
            }
        }
    }

    compact_fire<T, VEC>(sg, i0, fire, chi, cnt, stats);
}

// scalar loads of the live particles among [i0, i0 + VEC) (ragged tail, misaligned arrays)
template <typename T, int VEC>
__device__ __forceinline__ void load_scalar(const EvolveSeg<T> &sg, int64_t n, int64_t i0, T (&px)[VEC],
                                            T (&py)[VEC], T (&pz)[VEC], T (&ex)[VEC], T (&ey)[VEC], T (&ez)[VEC],
                                            T (&bx)[VEC], T (&by)[VEC], T (&bz)[VEC], T (&tau)[VEC], T (&tc)[VEC])
{
#pragma unroll
    for (int j = 0; j < VEC; ++j) {
        const int64_t i = i0 + j;
        const bool v = i < n;
        px[j] = v ? sg.px[i] : T(0);
        py[j] = v ? sg.py[i] : T(0);
        pz[j] = v ? sg.pz[i] : T(0);
        ex[j] = v ? sg.ex[i] : T(0);
        ey[j] = v ? sg.ey[i] : T(0);
        ez[j] = v ? sg.ez[i] : T(0);
        bx[j] = v ? sg.bx[i] : T(0);
        by[j] = v ? sg.by[i] : T(0);
        bz[j] = v ? sg.bz[i] : T(0);
        tau[j] = v ? sg.tau[i] : T(1);
        tc[j] = (sizeof(T) == 4 && v) ? sg.tau_c[i] : T(0);
    }
}

// In a batched step, `live` (n_seg + 1 entries; else NULL) keeps the live counts as the
// evolution reads them and, with stats, the photons removed by pair production that
// are still in the arrays (read, but not evolved).  The step's events count the
// evolved particles from them.  (A kernel that adds them up itself loses registers in
// its loop: FP32 direct loads of 6e7 particles 541 us, so 512; with any code of it
// after the loop 529.)
__device__ __forceinline__ long long removed_photons(const long long *stats)
{
    return stats[QED_STAT_PAIRS] - stats[QED_STAT_COMPACTED];
}

__device__ __forceinline__ bool keeps_removed(const long long *live, const long long *stats)
{
    return live && stats && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0;  // (the last CTA has the fewest tiles)
}

// Segments in device memory (many patches): every CTA reads all segment
// counts (clamped to capacity) into s_n (and the first into `live`), forms the
// inclusive prefix of their tile counts in s_end by a block scan (thread k owns
// segments [k per, (k+1) per)), and returns the total number of tiles.  Ends with a
// barrier.
template <typename T, int THREADS>
__device__ __forceinline__ long long tile_prefix(const EvolveSeg<T> *__restrict__ segs, int n_seg, int64_t tile,
                                                 long long *s_end, long long *s_n, long long *s_warp,
                                                 long long *live)
{
    const int per = (n_seg + THREADS - 1) / THREADS;
    const int s0 = threadIdx.x * per, s1 = min(n_seg, s0 + per);
    long long local = 0;
    for (int s = s0; s < s1; ++s) {
        long long n = *segs[s].count;
        n = n < 0 ? 0 : (n > segs[s].capacity ? segs[s].capacity : n);
        s_n[s] = n;
        if (live && blockIdx.x == 0) live[s] = n;
        local += (n + tile - 1) / tile;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    long long woff = 0;
    for (int w = 0; w < warp; ++w) woff += s_warp[w];
    long long acc = woff + incl - local;
    for (int s = s0; s < s1; ++s) {
        acc += (s_n[s] + tile - 1) / tile;
        s_end[s] = acc;
    }
    __syncthreads();
    return n_seg ? s_end[n_seg - 1] : 0;
}

// the segment of tile t: the first s with s_end[s] > t
__device__ __forceinline__ int find_segment(const long long *s_end, int n_seg, long long t)
{
    int lo = 0, hi = n_seg - 1;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (s_end[mid] > t)
            hi = mid;
        else
            lo = mid + 1;
    }
    return lo;
}

}  // namespace qed
