// pusher.cuh -- descriptors and per-particle arithmetic of the particle push
// (see pusher.cu); the fused push + evolution uses the same functions.
#pragma once

#include "common.cuh"
#include "evolve.cuh"

namespace qed {

struct WaveParams {
    double e0, omega_pi, phase0_pi;  // amplitude; omega / pi and phase0 / pi (phases in half-turns)
    int circular, direction;
};

template <typename T>
struct PushSeg {
    T *x, *y, *z, *px, *py, *pz, *ex, *ey, *ez, *bx, *by, *bz;
    const int64_t *count;
    int64_t cap;
    T q;
};

// sin and cos of pi u (the argument reduction of a half-turn multiple is exact)
__device__ __forceinline__ void d_sincospi(float u, float *s, float *c) { sincospif(u, s, c); }
__device__ __forceinline__ void d_sincospi(double u, double *s, double *c) { sincospi(u, s, c); }

// The wave's parameters, the time and the time step in the working precision.
// The host converts the parameters and the step: a kernel that takes them as
// FP64 arguments converts them again at every use once registers are short (the
// fused cascade kernel held GB300's narrow FP64 pipe 54 % busy with nothing but
// those conversions).  The batched kernels set t from the step counter.
template <typename T>
struct WaveT {
    T omega_pi, phase0_pi, e0, d, t, dt;
    int circular;
};

template <typename T>
inline WaveT<T> wave_in(const WaveParams &w, double dt, double t = 0.0)
{
    return WaveT<T>{(T)w.omega_pi, (T)w.phase0_pi, (T)w.e0, (T)w.direction, (T)t, (T)dt, w.circular};
}

// phase phi = omega (t - d x) + phase0; E = E0 (0, cos phi, [sin phi]); B = d x-hat cross E.
// Evaluated in the working precision, in half-turns (over the cascade's 10
// periods the FP32 phase keeps ~1e-5 rad).
template <typename T>
__device__ __forceinline__ void wave_fields(const WaveT<T> &w, T x, T &ex, T &ey, T &ez, T &bx, T &by, T &bz)
{
    const T u = w.omega_pi * (w.t - w.d * x) + w.phase0_pi;
    T s, c;
    d_sincospi(u, &s, &c);
    ex = T(0);
    ey = w.e0 * c;
    ez = w.circular ? w.e0 * s : T(0);
    bx = T(0);
    by = -w.d * ez;
    bz = w.d * ey;
}

// the linearly polarised wave's fields that are not zero (the sine comes with the cosine and is not used)
template <typename T>
__device__ __forceinline__ void wave_fields_yz(const WaveT<T> &w, T x, T &ey, T &bz)
{
    const T u = w.omega_pi * (w.t - w.d * x) + w.phase0_pi;
    T s, c;
    d_sincospi(u, &s, &c);
    ey = w.e0 * c;
    bz = w.d * ey;
}

// reciprocal square root: FP32 rsqrtf (within 2 ulp), FP64 on the integers (within
// 1 ulp, fixed64.cuh: an FP64 instruction of a warp takes 76 issue slots), and the
// quotient 2/x likewise; the push is not part of the paper's method, and its
// arithmetic budget is the fused cascade kernel's limit
__device__ __forceinline__ float d_rsqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double d_rsqrt(double x)
{
    if (!fix_plain(x)) return rsqrt(x);
    double root, inv;
    fix_sqrt_double(x, root, inv);
    return inv;
}
__device__ __forceinline__ float two_over(float x) { return 2.0f / x; }
__device__ __forceinline__ double two_over(double x) { return fix_plain(x) ? fix_div(2.0, x) : 2.0 / x; }

// products and sums that are not contracted
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return fma(a, b, c); }

// one step of the momentum of a particle of charge q (relativistic Boris
// rotation; q = 0: a photon, unchanged) and the velocity it then moves with
template <typename T>
__device__ __forceinline__ void boris_move(T q, T dt, T ex, T ey, T ez, T bx, T by, T bz, T &px, T &py, T &pz,
                                           T &vx, T &vy, T &vz)
{
    if (q == T(0)) {
        const T p2 = px * px + py * py + pz * pz;
        const T inv = p2 > T(0) ? d_rsqrt(p2) : T(0);
        vx = px * inv, vy = py * inv, vz = pz * inv;
        return;
    }
    const T h = T(0.5) * q * dt;
    const T mx = px + h * ex, my = py + h * ey, mz = pz + h * ez;  // half electric kick
    const T hg = h * d_rsqrt(T(1) + mx * mx + my * my + mz * mz);
    const T tx = hg * bx, ty = hg * by, tz = hg * bz;
    const T f = two_over(T(1) + tx * tx + ty * ty + tz * tz);
    const T sx = f * tx, sy = f * ty, sz = f * tz;
    const T qx = mx + (my * tz - mz * ty), qy = my + (mz * tx - mx * tz), qz = mz + (mx * ty - my * tx);
    px = mx + (qy * sz - qz * sy) + h * ex;
    py = my + (qz * sx - qx * sz) + h * ey;
    pz = mz + (qx * sy - qy * sx) + h * ez;
    const T ig = d_rsqrt(T(1) + px * px + py * py + pz * pz);
    vx = px * ig, vy = py * ig, vz = pz * ig;
}

// the same in fields with only Ey and Bz, the terms with a zero factor left out
// (bit for bit the same for finite momenta, see chi_lepton_yz)
template <typename T>
__device__ __forceinline__ void boris_move_yz(T q, T dt, T ey, T bz, T &px, T &py, T &pz, T &vx, T &vy, T &vz)
{
    if (q == T(0)) {
        const T p2 = px * px + py * py + pz * pz;
        const T inv = p2 > T(0) ? d_rsqrt(p2) : T(0);
        vx = px * inv, vy = py * inv, vz = pz * inv;
        return;
    }
    const T h = T(0.5) * q * dt;
    const T my = fma_rn(h, ey, py);  // half electric kick
    const T hg = h * d_rsqrt(T(1) + px * px + my * my + pz * pz);
    const T tz = mul_rn(hg, bz);
    const T f = two_over(fma_rn(tz, tz, T(1)));
    const T sz = mul_rn(f, tz);
    const T qx = add_rn(px, mul_rn(my, tz)), qy = add_rn(my, -mul_rn(px, tz));
    px = add_rn(px, mul_rn(qy, sz));
    py = fma_rn(h, ey, add_rn(my, -mul_rn(qx, sz)));
    const T ig = d_rsqrt(T(1) + px * px + py * py + pz * pz);
    vx = px * ig, vy = py * ig, vz = pz * ig;
}

template <typename T>
PushSeg<T> push_seg(const qed_species *s, double q);

template <typename T>
qed_status launch_push(const void *d_segs, int n_seg, const WaveParams &w, double t0, double dt,
                       const int64_t *d_step, int64_t step, int64_t capacity, cudaStream_t st);

// the fused push + evolution over segments in device memory (fused.cu): d_push
// holds PushSeg<T>[n_seg] in the order of d_segs; store_fields != 0 also writes
// the fields into the species; vec: every array 16-byte aligned
template <typename T>
qed_status launch_push_evolve(const EvolveSeg<T> *d_segs, const void *d_push, int n_seg, const TablesView<T> &tab,
                              const WaveParams &w, double t0, double dt, const int64_t *d_step, int64_t step,
                              T cut_qs, T cut_bw, long long *stats, int store_fields, bool vec, cudaStream_t st,
                              long long *live);

qed_status check_wave(const qed_plane_wave *w);
WaveParams wave_params(const qed_plane_wave *w);

}  // namespace qed
