// tablegen.cu -- FP64 generation of the four lookup tables on the GPU (§3 says
// the paper's generator needed CPU-only special functions and quadrature; here
// both run on the device).
//
//   Bessel functions: e^x K_nu(x) and e^x int_x^inf K_nu(s) ds from the integral
//   representation K_nu(x) = int_0^inf exp(-x cosh t) cosh(nu t) dt (and the same
//   integrand over cosh t for the tail integral), by the trapezoid rule in t,
//   which converges exponentially for this analytic, even integrand (Trefethen &
//   Weideman, SIAM Review 56 (2014) 385).  Step h = min(1/4, 0.6/sqrt(x)) keeps
//   the discretisation error near exp(-40); both integrals share one pass.
//   The tables need them at millions of arguments but only as functions of one
//   variable, so the trapezoid rule runs at the Chebyshev nodes of 160 pieces of
//   that variable (bessel_pieces_kernel) and the integrands evaluate the pieces'
//   polynomials: 26 FMAs instead of ~25 steps of an exponential, a hyperbolic
//   sine and divisions each.
//   Outer integrals over xi: Gauss-Legendre with 5, 8 or 16 points on the table
//   intervals where the integrand is smooth (gl_points), at nodes that all rows share;
//   tanh-sinh (double-exponential) quadrature (Takahasi & Mori 1974; Bailey,
//   Jeyabalan & Li, Exp. Math. 14 (2005) 317) on the others, which absorbs the
//   steep endpoint behaviour at xi -> 0 and 1.
//   QS (Eq. (qs_g_func)) integrates S(chi, xi) d(ln xi); BW (Eq. (t_func_0))
//   integrates the bracket in xi = chi_- / chi_gamma over [0, 1/2].
//
// One CTA per table row; one thread per Gauss-Legendre interval, one warp per
// tanh-sinh interval, whose sums are reduced by shuffles in a fixed order, so the
// tables are bit-reproducible.
#include <cmath>
#include <vector>

#include "common.cuh"
#include "fp64_math.cuh"

namespace qed {

qed_status check_params(const qed_table_params *p);
qed_status alloc_tables(const qed_table_params *p, qed_tables **out, size_t scratch = 0);
qed_status finish_tables(qed_tables *t, cudaStream_t st);

constexpr double kPi = 3.14159265358979323846;
constexpr double kTsStep = 1.0 / 16.0;  // tanh-sinh step
constexpr int kTsHalf = 52;             // nodes k = -52..52 (|k h| <= 3.25)
constexpr double kQsBelow = 100.0;  // the QS integral below xi_min starts at xi_min e^{-100}

// e^x int_x^inf K_a and e^x K_b, trapezoid rule in t
__device__ void bessel_scaled(double x, double nu_a, double nu_b, double &ia, double &kb)
{
    const double h = fmin(0.25, 0.6 / sqrt(x));
    const double nmax = fmax(nu_a, nu_b);
    double sa = 0.5, sb = 0.5;  // t = 0 terms, weight 1/2
    const double ra = exp(nu_a * h), rb = exp(nu_b * h), r1 = exp(h);
    double pa = 1.0, pb = 1.0, p1 = 1.0;
    for (int k = 1; k < 4000; ++k) {
        const double t = k * h;
        if ((k & 15) == 0) {
            pa = exp(nu_a * t), pb = exp(nu_b * t), p1 = exp(t);
        } else {
            pa *= ra, pb *= rb, p1 *= r1;
        }
        const double s = sinh(0.5 * t);
        const double arg = 2.0 * x * s * s;  // x (cosh t - 1)
        if (arg - nmax * t > 40.0 && arg > 40.0) break;
        const double e = exp(-arg);
        const double cha = 0.5 * (pa + 1.0 / pa), chb = 0.5 * (pb + 1.0 / pb), ch1 = 0.5 * (p1 + 1.0 / p1);
        sa += e * cha / ch1;
        sb += e * chb;
    }
    ia = h * sa;
    kb = h * sb;
}

// BW bracket in xi: int_z K_{1/3} + (xi/(1-xi) + (1-xi)/xi) K_{2/3}(z), z = 2/(3 chi xi (1-xi))
__device__ double bw_integrand(double chi, double xi)
{
    if (!(xi > 0.0) || !(xi < 1.0)) return 0.0;
    const double om = 1.0 - xi;
    const double z = 2.0 / (3.0 * chi * xi * om);
    if (z > 745.0) return 0.0;
    double ia, kb;
    bessel_scaled(z, 1.0 / 3.0, 2.0 / 3.0, ia, kb);
    return exp(-z) * (ia + (xi / om + om / xi) * kb);
}

// ---------------------------------------------------------------------------
// The two scaled functions of a process, e^x int_x^inf K_a and e^x K_b, as
// piecewise polynomials: four pieces per octave of x from 2^-30 to 2^10 (the
// integrands end at x = 745), degree 13.  Both functions are analytic in x but
// for x <= 0; a piece's centre lies at least 9 of its half-widths from 0, so its
// Chebyshev coefficients fall by a factor of 9 + sqrt(80) = 17.9 each and the
// truncation after 14 is below 3e-18.  The piece comes from the bits of x: no
// logarithm.  Below 2^-30 the two leading terms of the power series, whose
// relative remainder is of order x^2 < 2^-60.
// ---------------------------------------------------------------------------
constexpr int kPieceOct = -30, kPieceOcts = 40, kPieces = 4 * kPieceOcts, kPieceCoef = 14;
constexpr int kPieceRow = 2 * kPieceCoef;  // both functions of a piece

// One CTA per piece, both processes (they share K_{2/3}).  The trapezoid rule
// takes the step of the piece's largest argument, so its nodes t_k, and all
// factors but exp(-x (cosh t_k - 1)), are the same for the 14 arguments: the
// threads form them once, then eight threads to an argument each run every
// eighth step of its sum (one exponential and three FMAs).  Bound by FP64
// latency: with the factors formed in every step (~130 FP64 instructions) the
// launch took 362 us, with one warp per piece 148 us.
constexpr int kPieceT = 160;  // trapezoid nodes: (ln(2 (40 + 5/3 t) / 2^-30) / (1/4) = 106 at the lower end
__global__ void __launch_bounds__(128) bessel_pieces_kernel(double *out)
{
    __shared__ double s_c1[kPieceT], s_f[3][kPieceT];  // cosh t - 1; cosh(nu t)/cosh t for nu = 5/3, 1/3; cosh(2t/3)
    __shared__ double s_cos[4 * kPieceCoef], s_part[3][8][16];
    __shared__ int s_live;
    const int piece = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    const double scale = ldexp(1.0, kPieceOct + piece / 4);
    const double hi = scale * (1.0 + (2 * (piece % 4) + 2) / 8.0), lo = scale * (1.0 + (2 * (piece % 4)) / 8.0);
    const double h = fmin(0.25, 0.6 / sqrt(hi));
    if (tid == 0) s_live = 0;
    if (tid < 4 * kPieceCoef) s_cos[tid] = cospi((double)tid / (2 * kPieceCoef));
    __syncthreads();
    for (int k = tid + 1; k <= kPieceT; k += 128) {  // (whole warps)
        const double t = k * h, s = sinh(0.5 * t), c1 = 2.0 * s * s;
        const double e1 = exp(t / 3.0), i1 = 1.0 / e1, e2 = e1 * e1, i2 = i1 * i1;
        const double ch = 1.0 / (e2 * e1 + i2 * i1);  // 1/(2 cosh t)
        s_c1[k - 1] = c1;
        s_f[0][k - 1] = (e2 * e2 * e1 + i2 * i2 * i1) * ch;
        s_f[1][k - 1] = (e1 + i1) * ch;
        s_f[2][k - 1] = 0.5 * (e2 + i2);
        // steps needed: until lo (cosh t - 1) leaves every integrand below e^-40
        const unsigned live = __ballot_sync(0xffffffffu, !(lo * c1 > 40.0 && lo * c1 - 5.0 / 3.0 * t > 40.0));
        if (lane == 0) atomicAdd(&s_live, __popc(live));
    }
    __syncthreads();
    {
        const int i = tid & 15, part = tid >> 4, n = s_live;
        double sum[3] = {0.0, 0.0, 0.0};
        if (i < kPieceCoef) {
            const double x = scale * (1.0 + (2 * (piece % 4) + 1 + s_cos[2 * i + 1]) / 8.0);  // Chebyshev node
            for (int k = part; k < n; k += 8) {
                const double e = exp_tang(fmax(-x * s_c1[k], -700.0));
#pragma unroll
                for (int f = 0; f < 3; ++f) sum[f] = fma(e, s_f[f][k], sum[f]);
            }
        }
#pragma unroll
        for (int f = 0; f < 3; ++f) s_part[f][part][i] = sum[f];
    }
    __syncthreads();
    const int f = tid >> 5;  // a warp per function
    if (f == 3) return;
    double v = 0.0;
    if (lane < kPieceCoef) {
        v = 0.5;  // the term t = 0
#pragma unroll
        for (int p = 0; p < 8; ++p) v += s_part[f][p][lane];
        v *= h;
    }
    // lane i: Chebyshev coefficient i, then the coefficient of x^i by the
    // recurrence T_k = 2 x T_{k-1} - T_{k-2}
    double c = 0.0;
    for (int i = 0; i < kPieceCoef; ++i)  // (the angle in units of pi / (2 kPieceCoef))
        c += __shfl_sync(0xffffffffu, v, i) * s_cos[(2 * i + 1) * lane % (4 * kPieceCoef)];
    c *= (lane ? 2.0 : 1.0) / kPieceCoef;
    double t0 = lane == 0 ? 1.0 : 0.0, t1 = lane == 1 ? 1.0 : 0.0;  // T_0, T_1
    double p = __shfl_sync(0xffffffffu, c, 0) * t0 + __shfl_sync(0xffffffffu, c, 1) * t1;
    for (int i = 2; i < kPieceCoef; ++i) {
        const double up = __shfl_up_sync(0xffffffffu, t1, 1);
        const double t2 = 2.0 * (lane ? up : 0.0) - t0;
        p += __shfl_sync(0xffffffffu, c, i) * t2;
        t0 = t1, t1 = t2;
    }
    if (lane < kPieceCoef) {
        double *qs = out + (size_t)piece * kPieceRow + lane, *bw = qs + (size_t)kPieces * kPieceRow;
        if (f == 0) qs[0] = p;
        if (f == 1) bw[0] = p;
        if (f == 2) qs[kPieceCoef] = bw[kPieceCoef] = p;
    }
}

constexpr double kGamma13 = 2.6789385347077476, kGamma23 = 1.3541179394264004;  // Gamma(1/3), Gamma(2/3)
constexpr double kTwo13 = 1.2599210498948732, kTwo23 = 1.5874010519681994;      // 2^(1/3), 2^(2/3)
constexpr double kPiSqrt3 = 1.8137993642342178;                                  // pi / sqrt(3)

// e^x int_x^inf K_{5/3 or 1/3} and e^x K_{2/3} for 0 < x < 2^10 from the pieces `c` of the process
__device__ __forceinline__ void bessel_at(const double *c, bool qs, double x, double &ia, double &kb)
{
    const int hi = __double2hiint(x);
    const int i = ((hi >> 20) - 1023 - kPieceOct) * 4 + ((hi >> 18) & 3);
    if (i < 0) {
        const double r = cbrt(x), r2 = r * r;
        kb = (1.0 + x) * (0.5 * kGamma23 * kTwo23 / r2 - 0.75 * kGamma13 / kTwo23 * r2);
        ia = (1.0 + x) * (qs ? kGamma23 * kTwo23 / r2 - kPiSqrt3
                             : kPiSqrt3 - 0.75 * kGamma13 * kTwo13 * r2 + 1.125 * kGamma23 / kTwo13 * r2 * r2);
        return;
    }
    const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(x));  // x / 2^e in [1, 2)
    const double t = fma(m, 8.0, -(9.0 + 2 * ((hi >> 18) & 3)));                           // the piece's [-1, 1]
    const double *p = c + min(i, kPieces - 1) * kPieceRow;
    double a = p[kPieceCoef - 1], b = p[2 * kPieceCoef - 1];
#pragma unroll
    for (int k = kPieceCoef - 2; k >= 0; --k) {
        a = fma(a, t, p[k]);
        b = fma(b, t, p[kPieceCoef + k]);
    }
    ia = a, kb = b;
}

// QS integrand in u = ln xi: S(chi, xi) = sqrt(3)/(2 pi) xi [int_Y K_{5/3} + xi^2/(1-xi) K_{2/3}(Y)],
// Y = (2/3) xi / (chi (1 - xi)); BW the bracket in xi.  The integrand is
// e^(-q/chi) [va int(q/chi) + vb K_{2/3}(q/chi)] with q, va, vb functions of xi alone.
constexpr double kQsFactor = 0.27566444771089600;  // sqrt(3) / (2 pi)

__device__ __forceinline__ void node_terms(bool qs, double x, double &q, double &va, double &vb)
{
    if (qs) {
        // xi and om = 1 - xi, each without cancellation, from one exponential
        double xi, om;
        if (x > -0.7) {
            om = -expm1(x);
            xi = 1.0 - om;
        } else {
            xi = exp_tang(x);
            om = 1.0 - xi;
        }
        const double r = xi / om;
        q = (2.0 / 3.0) * r;
        va = kQsFactor * xi;
        vb = va * (xi * r);
    } else {
        const double om = 1.0 - x, r = 1.0 / (x * om);
        q = (2.0 / 3.0) * r;
        va = 1.0;
        vb = (x * x + om * om) * r;  // x/om + om/x
    }
}

__device__ __forceinline__ double row_integrand(const double *c, bool qs, double inv_chi, double q, double va,
                                                double vb)
{
    const double y = q * inv_chi;
    if (!(y <= 745.0)) return 0.0;  // (also 1 - xi = 0, where q is infinite)
    double ia, kb;
    bessel_at(c, qs, y, ia, kb);
    return exp_tang(-y) * fma(vb, kb, va * ia);
}

struct GenArgs {
    double *qs_lnG, *qs_lnP, *bw_lnT, *bw_P;
    double qs_l0, qs_l1, qs_xi_min, qs_ln_xi_min, bw_l0, bw_l1;
    int qs_n_chi, qs_n_xi, bw_n_chi, bw_n_xi;
    int *points;  // [2][n_xi]: the fewest points that an interval's place allows
    double ts_end[kTsHalf + 1], ts_w[kTsHalf + 1];  // tanh-sinh: distance of node k from the nearer end, weight (half-widths)
    double *pieces;  // [2][kPieces][kPieceRow]: the Bessel functions
    double *nodes;   // [2][3][kGlSlots][n_xi]: q, w va, w vb at the Gauss-Legendre nodes of every interval
};

// interval j of a row: QS j = 0 is [xi_min e^-100, xi_min] in ln xi, j >= 1 is
// [xi_{j-1}, xi_j]; BW j >= 1 is [xi_{j-1}, xi_j] on the linear grid, j = 0 empty
__device__ __forceinline__ void row_interval(bool qs, double ln_xi_min, int M, int j, double &lo, double &hi)
{
    if (qs) {
        lo = j == 0 ? ln_xi_min - kQsBelow : ln_xi_min + (j - 1) * (-ln_xi_min) / (M - 1);
        hi = (j == M - 1) ? 0.0 : ln_xi_min + j * (-ln_xi_min) / (M - 1);
    } else {
        lo = 0.5 * (j - 1) / (M - 1);
        hi = (j == M - 1) ? 0.5 : 0.5 * j / (M - 1);
    }
}

// Gauss-Legendre rules (weights and nodes of the reference interval by value).
// What bounds a rule is the place of the integrand's singularity (QS: ln xi = 0,
// where 1 - xi vanishes; BW: xi = 0), c half-widths from the interval's centre
// (the error of n points falls like (c + sqrt(c^2 - 1))^-2n), the interval's
// width in ln xi against the integrand's own scale, and how far e^-Y falls across
// it, e^-f (the error of e^(-f t/2) on [-1, 1]):
//   16 points: c >= 2 (5e-19), f <= 12 (2e-20);
//    8 points: c >= 8 (6e-20), f <= 2 (2e-18);
//    5 points: c >= 40 (9e-20), f <= 0.3 (5e-18).
// QS interval 0, below xi_min, is integrated in w = xi^(1/3), S growing like w
// there: with 16 points if Y(xi_min) <= 1/2 and xi_min <= 1/5 (xi = 1 then lies 2.4
// half-widths from the centre).
constexpr int kGl = 16, kGl8 = 8, kGl5 = 5;
constexpr int kGlSlots = kGl + kGl8 + kGl5;  // the three rules' nodes of an interval, one after the other
struct GaussLegendreRules {
    double x[kGl], w[kGl], x8[kGl8], w8[kGl8], x5[kGl5], w5[kGl5];
};

// the fewest points that the interval's place allows: 16, 8, 5, or 0 (tanh-sinh)
__device__ __forceinline__ int gl_points(bool qs, int j, double lo, double hi)
{
    if (j == 0) return qs && hi <= -1.6095 ? kGl : 0;  // ln(1/5)
    const double c = qs ? -0.5 * (lo + hi) : 0.5 * (lo + hi), h = 0.5 * (hi - lo);
    if (c < 2.0 * h || (qs && h > 0.5)) return 0;
    if (c < 8.0 * h || (qs && h > 0.1)) return kGl;
    return c < 40.0 * h ? kGl8 : kGl5;
}

// the nodes that every row of a process shares: thread = (interval, node), blockIdx.y = process
__global__ void __launch_bounds__(128) row_nodes_kernel(const __grid_constant__ GenArgs a,
                                                         const __grid_constant__ GaussLegendreRules g)
{
    const bool qs = blockIdx.y == 0;
    const int M = qs ? a.qs_n_xi : a.bw_n_xi;
    const int j = blockIdx.x * 4 + threadIdx.x / 32, k = threadIdx.x % 32;
    if (j >= M || k >= kGlSlots) return;
    double lo, hi;
    row_interval(qs, a.qs_ln_xi_min, M, j, lo, hi);
    const int points = gl_points(qs, j, lo, hi);
    if (k == 0) a.points[(qs ? 0 : a.qs_n_xi) + j] = points;
    // (a rule with more points than the place asks for serves the rows where e^-Y falls faster)
    const int n = k < kGl ? kGl : k < kGl + kGl8 ? kGl8 : kGl5;
    if (points == 0 || n < points) return;
    double *out = a.nodes + (qs ? 0 : (size_t)3 * kGlSlots * a.qs_n_xi);
    double x, w;
    if (j == 0) {  // w^3 = xi from 0 to xi_min: S du = (3 S / w) dw
        const double top = cbrt(a.qs_xi_min), v = 0.5 * top * (1.0 + g.x[k]);
        x = 3.0 * log(v);
        w = 0.5 * top * g.w[k] * 3.0 / v;
    } else {
        const double c = 0.5 * (lo + hi), h = 0.5 * (hi - lo);
        x = fma(h, n == kGl ? g.x[k] : n == kGl8 ? g.x8[k - kGl] : g.x5[k - kGl - kGl8], c);
        w = h * (n == kGl ? g.w[k] : n == kGl8 ? g.w8[k - kGl] : g.w5[k - kGl - kGl8]);
    }
    double q, va, vb;
    node_terms(qs, x, q, va, vb);
    out[(size_t)k * M + j] = q;
    out[(size_t)(kGlSlots + k) * M + j] = w * va;
    out[(size_t)(2 * kGlSlots + k) * M + j] = w * vb;
}

// One CTA per row.  Bound by the FP64 pipe: ~60 FP64 instructions per
// Gauss-Legendre node, ~256 x 6 nodes in a row of the 256 x 256 tables, and the
// tanh-sinh intervals (one at the end, and ~4 per row across which e^-Y falls
// steeply), whose nodes and weights on [-1, 1] are shared too.  Shared memory by
// the row's length, so that all 512 rows are resident at once (three to an SM
// left 56 rows for a second wave).
__global__ void __launch_bounds__(256) table_rows_kernel(const __grid_constant__ GenArgs a)
{
    extern __shared__ double s_c[];  // [kPieces][kPieceRow], then acc, tail, cum [M]
    __shared__ short s_hard[QED_MAX_TABLE_N];
    __shared__ int s_n_hard;
    __shared__ double s_chi[2];
    const bool qs = blockIdx.x < (unsigned)a.qs_n_chi;
    const int row = qs ? blockIdx.x : blockIdx.x - a.qs_n_chi;
    const int N = qs ? a.qs_n_chi : a.bw_n_chi;
    const int M = qs ? a.qs_n_xi : a.bw_n_xi;
    double *const acc = s_c + kPieces * kPieceRow, *const tail = acc + M, *const cum = tail + M;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;

    if (threadIdx.x == 0) {
        const double l0 = qs ? a.qs_l0 : a.bw_l0, l1 = qs ? a.qs_l1 : a.bw_l1;
        s_chi[0] = exp(row == N - 1 ? l1 : l0 + row * (l1 - l0) / (N - 1));
        s_chi[1] = 1.0 / s_chi[0];
        s_n_hard = 0;
    }
    const double *pieces = a.pieces + (qs ? 0 : (size_t)kPieces * kPieceRow);
    for (int i = threadIdx.x; i < kPieces * kPieceRow; i += blockDim.x) s_c[i] = pieces[i];
    __syncthreads();
    const double chi = s_chi[0], inv_chi = s_chi[1];

    const double *nodes = a.nodes + (qs ? 0 : (size_t)3 * kGlSlots * a.qs_n_xi);
    const int *allowed = a.points + (qs ? 0 : a.qs_n_xi);
    for (int j = threadIdx.x; j < M; j += blockDim.x) {
        if (!qs && j == 0) {
            acc[0] = 0.0;
            continue;
        }
        int points = allowed[j];
        if (points) {
            // the fall of e^-Y between the outermost nodes of 16, which lie within 1 % of the ends
            const double q0 = nodes[j], q1 = nodes[(size_t)(kGl - 1) * M + j];
            if (fmin(q0, q1) * inv_chi > 800.0 && j > 0) {  // e^-Y is zero on all of it
                acc[j] = 0.0;
                continue;
            }
            const double fall = fabs(q1 - q0) * inv_chi;
            if (points == kGl5 && fall > 0.29) points = kGl8;
            if (points == kGl8 && fall > 1.9) points = kGl;
            if (fall > (j == 0 ? 0.5 : 11.5)) points = 0;
        }
        if (points) {
            const double *p = nodes + (size_t)(points == kGl ? 0 : points == kGl8 ? kGl : kGl + kGl8) * M + j;
            double part = 0.0;
            for (int k = 0; k < points; ++k, p += M)
                part += row_integrand(s_c, qs, inv_chi, p[0], p[(size_t)kGlSlots * M], p[(size_t)2 * kGlSlots * M]);
            acc[j] = part;
        } else {
            s_hard[atomicAdd(&s_n_hard, 1)] = (short)j;
        }
    }
    __syncthreads();
    for (int i = warp; i < s_n_hard; i += nw) {
        const int j = s_hard[i];
        double lo, hi;
        row_interval(qs, a.qs_ln_xi_min, M, j, lo, hi);
        const double r = 0.5 * (hi - lo);
        double part = 0.0;
        for (int k = lane - kTsHalf; k <= kTsHalf; k += 32) {
            const double d = r * a.ts_end[abs(k)];  // offset from the nearer end, exact near the ends
            const double x = k < 0 ? lo + d : (k > 0 ? hi - d : 0.5 * (lo + hi));
            if (!qs && !(x > 0.0)) continue;
            double q, va, vb;
            node_terms(qs, x, q, va, vb);
            part += a.ts_w[abs(k)] * row_integrand(s_c, qs, inv_chi, q, va, vb);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        if (lane == 0) acc[j] = r * part;
    }
    __syncthreads();
    // running sums from both ends, in order (one thread each, in two warps)
    if (threadIdx.x == 0) {
        double c = 0.0;
        for (int m = M - 1; m >= 0; --m) {
            tail[m] = c;  // the sum right of m
            c += acc[m];
        }
    } else if (threadIdx.x == 32) {
        double c = 0.0;
        for (int m = 0; m < M; ++m) {
            c += acc[m];
            cum[m] = c;
        }
    }
    __syncthreads();
    const double tot = cum[M - 1];
    if (qs) {
        // ln P = ln(C/G), except near P = 1 where log1p(-tail/G) keeps the relative accuracy
        double *out = a.qs_lnP + (size_t)row * M;
        for (int m = threadIdx.x; m < M; m += blockDim.x) {
            const double t = tail[m] / tot;
            out[m] = m == M - 1 ? 0.0 : (t < 0.5 ? log1p(-t) : log(cum[m] / tot));
        }
        if (threadIdx.x == 0) a.qs_lnG[row] = log(tot);
    } else {
        double *out = a.bw_P + (size_t)row * M;
        for (int m = threadIdx.x; m < M; m += blockDim.x) {
            double v = tot > 0.0 ? cum[m] / (2.0 * tot) : 0.0;
            if (m == 0) v = 0.0;
            if (m == M - 1 && tot > 0.0) v = 0.5;
            out[m] = v;
        }
        // T = int_0^1 bracket / (pi sqrt(3) chi) = 2 tot / (pi sqrt(3) chi)
        if (threadIdx.x == 0) a.bw_lnT[row] = log(2.0 * tot / (kPi * 1.7320508075688772 * chi));
    }
}

// ---------------------------------------------------------------------------
// Exact inverse CDF, no table (the learned sampler's training targets).  Per chi
// row, the cumulative integral of the spectrum on a fine grid and its density
// at the nodes; per draw, the bracketing interval by binary search, a first
// guess from the cubic Hermite interpolant of the cumulative integral on that
// interval (value and slope at both nodes), then Newton steps on the partial
// integral from the interval's left node (Gauss-Legendre, 8 points).
// Grid variables (both smooth in them over the whole range):
//   QS: v = ln(xi / (1 - xi)) on [ln 1e-12, -ln 1e-12] in kExactIntervals - 1
//       equal intervals, plus [ln 1e-12 - 100, ln 1e-12] below (where P follows
//       its xi^(1/3) law; tanh-sinh there); the density is S(chi, xi) (1 - xi),
//       which resolves both the soft end and the cut-off at 1 - xi ~ 1/chi;
//   BW: v = ln xi on [ln 1e-12, ln 1/2] in kExactIntervals equal intervals,
//       density xi times the bracket of Eq. (t_func_0), normalised to P(1/2) = 1.
// ---------------------------------------------------------------------------
constexpr int kExactIntervals = 1024;
constexpr double kExactLo = -27.631021115928547;  // ln 1e-12

struct GaussLegendre8 {
    double x[8], w[8];  // nodes and weights on [-1, 1]
};

// density in v of the QS photon number spectrum: S(chi, xi) (1 - xi)
__device__ double qs_density_v(double chi, double v)
{
    const double e = exp(-fabs(v));
    const double xi = v >= 0.0 ? 1.0 / (1.0 + e) : e / (1.0 + e);
    const double om = v >= 0.0 ? e / (1.0 + e) : 1.0 / (1.0 + e);  // 1 - xi without cancellation
    if (!(om > 0.0) || !(xi > 0.0)) return 0.0;
    const double Y = (2.0 / 3.0) * xi / (chi * om);
    if (Y > 745.0) return 0.0;
    double ia, kb;
    bessel_scaled(Y, 5.0 / 3.0, 2.0 / 3.0, ia, kb);
    return (0.27566444771089600 /* sqrt(3) / (2 pi) */) * xi * om * exp(-Y) * (ia + xi * xi / om * kb);
}

// density in v = ln xi of the BW split: xi times the bracket
__device__ double bw_density_v(double chi, double v)
{
    const double xi = exp(v);
    return xi * bw_integrand(chi, xi);
}

__device__ __forceinline__ double exact_density(bool qs, double chi, double v)
{
    return qs ? qs_density_v(chi, v) : bw_density_v(chi, v);
}

// node j of the grid (j = 0 .. kExactIntervals)
__device__ __forceinline__ double exact_node(bool qs, int j)
{
    if (qs) {
        if (j == 0) return kExactLo - kQsBelow;
        return kExactLo + (j - 1) * (-2.0 * kExactLo) / (kExactIntervals - 1);
    }
    return kExactLo + j * (-0.6931471805599453 - kExactLo) / kExactIntervals;
}

__device__ double gl8(const GaussLegendre8 &g, bool qs, double chi, double a, double b)
{
    const double c = 0.5 * (a + b), h = 0.5 * (b - a);
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) s += g.w[i] * exact_density(qs, chi, fma(h, g.x[i], c));
    return h * s;
}

// The QS interval below the grid (v from ln 1e-12 - 100 to ln 1e-12): there the
// density grows like e^{v/3} (the xi^(1/3) law of P), so it is integrated in
// w = e^{v/3}, where the integrand 3 density / w is nearly constant (8-point
// Gauss-Legendre on [w(a), w(v)]).
__device__ double gl8_below(const GaussLegendre8 &g, double chi, double a, double v)
{
    const double wa = exp(a / 3.0), wb = exp(v / 3.0);
    const double c = 0.5 * (wa + wb), h = 0.5 * (wb - wa);
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const double w = fma(h, g.x[i], c);
        s += g.w[i] * 3.0 * qs_density_v(chi, 3.0 * log(w)) / w;
    }
    return h * s;
}

constexpr int kExactRowStride = 2 * (kExactIntervals + 1) + 1;  // P[0..M], p[0..M], total

// one CTA per chi row: P at the nodes (P_0 = 0 .. P_M = 1), the density p at
// the nodes divided by the total, then the total
__global__ void __launch_bounds__(256) exact_rows_kernel(int qs, const double *__restrict__ chi_rows,
                                                          double *__restrict__ work, GaussLegendre8 g)
{
    __shared__ double acc[kExactIntervals];
    const double chi = chi_rows[blockIdx.x];
    double *out = work + (size_t)blockIdx.x * kExactRowStride;
    if (qs && threadIdx.x == 0) acc[0] = gl8_below(g, chi, exact_node(true, 0), exact_node(true, 1));
    for (int j = threadIdx.x + (qs ? 1 : 0); j < kExactIntervals; j += blockDim.x)
        acc[j] = gl8(g, qs, chi, exact_node(qs, j), exact_node(qs, j + 1));
    for (int j = threadIdx.x; j <= kExactIntervals; j += blockDim.x)
        out[kExactIntervals + 1 + j] = exact_density(qs, chi, exact_node(qs, j));
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int j = 0; j < kExactIntervals; ++j) tot += acc[j];
        double c = 0.0;
        out[0] = 0.0;
        for (int j = 0; j < kExactIntervals; ++j) {
            c += acc[j];
            out[j + 1] = tot > 0.0 ? c / tot : 0.0;
        }
        out[kExactIntervals] = 1.0;
        out[2 * (kExactIntervals + 1)] = tot;
    }
    __syncthreads();
    const double tot = out[2 * (kExactIntervals + 1)];
    for (int j = threadIdx.x; j <= kExactIntervals; j += blockDim.x)
        out[kExactIntervals + 1 + j] = tot > 0.0 ? out[kExactIntervals + 1 + j] / tot : 0.0;
}

__global__ void __launch_bounds__(128) exact_draw_kernel(int qs, const double *__restrict__ chi_rows,
                                                          const double *__restrict__ work, int64_t m, int64_t k,
                                                          const double *__restrict__ uu, double *__restrict__ xi,
                                                          GaussLegendre8 g)
{
    const int64_t n = m * k;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t row = i / k;
        const double chi = chi_rows[row];
        const double *P = work + (size_t)row * kExactRowStride;
        const double *D = P + kExactIntervals + 1;
        const double tot = P[2 * (kExactIntervals + 1)];
        double u = uu[i];
        u = u < 0.0 ? 0.0 : (u > 1.0 ? 1.0 : u);
        const double r = qs ? u : 2.0 * (u < 1.0 - u ? u : 1.0 - u);
        double v;
        if (!(tot > 0.0) || r >= 1.0) {
            v = qs ? 1e300 : -0.6931471805599453;
        } else if (r <= 0.0) {
            v = -1e300;
        } else {
            int lo = 0, hi = kExactIntervals;  // j: P_j <= r < P_{j+1}
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (P[mid] <= r) lo = mid; else hi = mid;
            }
            const int j = lo;
            const double a = exact_node(qs, j), b = exact_node(qs, j + 1), L = b - a;
            const double P0 = P[j], P1 = P[j + 1];
            if (qs && j == 0) {
                // below the grid: the xi^(1/3) law as the first guess, Newton on ln P
                v = b + 3.0 * (log(r) - log(P1));
                v = v < a ? a : (v > b ? b : v);
                for (int it = 0; it < 8; ++it) {
                    const double F = P0 + gl8_below(g, chi, a, v) / tot;
                    const double f = exact_density(true, chi, v) / tot;
                    if (!(F > 0.0) || !(f > 0.0)) break;
                    double vn = v - (log(F) - log(r)) * F / f;
                    vn = vn < a ? a : (vn > b ? b : vn);
                    const double dv = fabs(vn - v);
                    v = vn;
                    if (dv < 1e-13) break;
                }
            } else {
                // cubic Hermite of P on t in [0, 1]: P(t) = P0 + ... with slopes L p_j, L p_{j+1};
                // its inverse by Newton from the linear guess
                const double m0 = L * D[j], m1 = L * D[j + 1], dP = P1 - P0;
                double t = dP > 0.0 ? (r - P0) / dP : 0.5;
                for (int it = 0; it < 6; ++it) {
                    const double t2 = t * t, t3 = t2 * t;
                    const double h = P0 * (2 * t3 - 3 * t2 + 1) + m0 * (t3 - 2 * t2 + t) + P1 * (-2 * t3 + 3 * t2) +
                                     m1 * (t3 - t2);
                    const double dh = P0 * (6 * t2 - 6 * t) + m0 * (3 * t2 - 4 * t + 1) + P1 * (-6 * t2 + 6 * t) +
                                      m1 * (3 * t2 - 2 * t);
                    if (!(dh > 0.0)) break;
                    double tn = t - (h - r) / dh;
                    tn = tn < 0.0 ? 0.0 : (tn > 1.0 ? 1.0 : tn);
                    t = tn;
                }
                v = a + L * t;
                // Newton on the partial integral (the cumulative integral itself)
                for (int it = 0; it < 4; ++it) {
                    const double F = P0 + gl8(g, qs, chi, a, v) / tot;
                    const double f = exact_density(qs, chi, v) / tot;
                    if (!(f > 0.0)) break;
                    double vn = v - (F - r) / f;
                    vn = vn < a ? a : (vn > b ? b : vn);
                    const double dv = fabs(vn - v);
                    v = vn;
                    if (dv < 1e-7 * L) break;  // the next correction is ~(dv / L)^2 of this one
                }
            }
        }
        double out;
        if (qs) {
            const double e = exp(-fabs(v));
            out = v >= 0.0 ? 1.0 / (1.0 + e) : e / (1.0 + e);
        } else {
            out = exp(v);
            out = out > 0.5 ? 0.5 : out;
            out = (u <= 0.5) ? out : 1.0 - out;
        }
        xi[i] = out;
    }
}

// Gauss-Legendre nodes and weights, n points (Newton's method on the three-term recurrence)
template <int n>
static void gauss_legendre(double (&gx)[n], double (&gw)[n])
{
    for (int i = 0; i < n; ++i) {
        double x = std::cos(kPi * (i + 0.75) / (n + 0.5));
        double dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = x;
            for (int k = 2; k <= n; ++k) {
                const double p2 = ((2.0 * k - 1.0) * x * p1 - (k - 1.0) * p0) / k;
                p0 = p1, p1 = p2;
            }
            dp = n * (x * p1 - p0) / (x * x - 1.0);
            const double dx = p1 / dp;
            x -= dx;
            if (std::fabs(dx) < 1e-16) break;
        }
        gx[i] = x;
        gw[i] = 2.0 / ((1.0 - x * x) * dp * dp);
    }
}

}  // namespace qed

using namespace qed;

extern "C" qed_status qed_exact_sample(qed_process proc, const double *d_chi, int64_t m, const double *d_u,
                                       int64_t k, double *d_xi, double *d_work, int64_t work_capacity, void *stream)
{
    clear_error();
    if (proc != QED_PROC_QS && proc != QED_PROC_BW) QED_FAIL(QED_ERR_INVALID_ARG, "bad process %d", (int)proc);
    if (m < 0 || k < 0) QED_FAIL(QED_ERR_INVALID_ARG, "negative sizes");
    if (m == 0 || k == 0) return QED_OK;
    if (!d_chi || !d_u || !d_xi || !d_work) QED_FAIL(QED_ERR_INVALID_ARG, "a device array is NULL");
    if (m >= (int64_t)1 << 31 || k > ((int64_t)1 << 40) / m) QED_FAIL(QED_ERR_INVALID_ARG, "too many draws");
    if (work_capacity < QED_EXACT_WORK(m))
        QED_FAIL(QED_ERR_INVALID_ARG, "d_work holds %lld doubles, %lld needed", (long long)work_capacity,
                 (long long)QED_EXACT_WORK(m));
    static_assert(QED_EXACT_WORK(1) == kExactRowStride, "work layout");
    static const GaussLegendre8 gl = [] {
        GaussLegendre8 g;
        gauss_legendre<8>(g.x, g.w);
        return g;
    }();
    cudaStream_t st = as_stream(stream);
    const int qs = proc == QED_PROC_QS;
    exact_rows_kernel<<<(unsigned)m, 256, 0, st>>>(qs, d_chi, d_work, gl);
    QED_LAUNCH_CHECK();
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t blocks = (m * k + 127) / 128;
    const int g = (int)(blocks < (int64_t)sms * 8 ? blocks : (int64_t)sms * 8);
    exact_draw_kernel<<<g, 128, 0, st>>>(qs, d_chi, d_work, m, k, d_u, d_xi, gl);
    QED_LAUNCH_CHECK();
    return QED_OK;
}

extern "C" qed_status qed_tables_generate(const qed_table_params *params, qed_tables **out, void *stream)
{
    clear_error();
    if (!out) QED_FAIL(QED_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    qed_status s = check_params(params);
    if (s) return s;
    qed_tables *t = nullptr;
    const size_t scratch =
        ((size_t)2 * kPieces * kPieceRow + (size_t)3 * kGlSlots * (params->qs.n_xi + params->bw.n_xi)) * sizeof(double) +
        (size_t)(params->qs.n_xi + params->bw.n_xi) * sizeof(int);
    if ((s = alloc_tables(params, &t, scratch))) return s;
    cudaStream_t st = as_stream(stream);
    GenArgs a;
    a.qs_lnG = t->d_qs_lnG, a.qs_lnP = t->d_qs_lnP, a.bw_lnT = t->d_bw_lnT, a.bw_P = t->d_bw_P;
    a.qs_l0 = std::log(params->qs.chi_min), a.qs_l1 = std::log(params->qs.chi_max);
    a.qs_xi_min = params->qs.xi_min;
    a.qs_ln_xi_min = std::log(params->qs.xi_min);
    for (int k = 0; k <= kTsHalf; ++k) {
        const double tk = k * kTsStep, sh = 0.5 * kPi * std::sinh(tk), ch = std::cosh(sh);
        a.ts_end[k] = 2.0 / (1.0 + std::exp(2.0 * sh));
        a.ts_w[k] = kTsStep * 0.5 * kPi * std::cosh(tk) / (ch * ch);
    }
    a.bw_l0 = std::log(params->bw.chi_min), a.bw_l1 = std::log(params->bw.chi_max);
    a.qs_n_chi = params->qs.n_chi, a.qs_n_xi = params->qs.n_xi;
    a.bw_n_chi = params->bw.n_chi, a.bw_n_xi = params->bw.n_xi;
    // scratch (the pieces, the shared nodes) in the room of the derived tables, which finish_tables fills afterwards
    a.pieces = (double *)t->derived;
    a.nodes = a.pieces + (size_t)2 * kPieces * kPieceRow;
    a.points = (int *)(a.nodes + (size_t)3 * kGlSlots * (params->qs.n_xi + params->bw.n_xi));
    static const GaussLegendreRules gl = [] {
        GaussLegendreRules g;
        gauss_legendre<kGl>(g.x, g.w);
        gauss_legendre<kGl8>(g.x8, g.w8);
        gauss_legendre<kGl5>(g.x5, g.w5);
        return g;
    }();
    const int m = params->qs.n_xi > params->bw.n_xi ? params->qs.n_xi : params->bw.n_xi;
    const int dyn = (kPieces * kPieceRow + 3 * m) * (int)sizeof(double);
    // (the largest row's size for every call: the attribute is the process's, and a smaller one set by
    // another thread would refuse this launch)
    constexpr int kMaxDyn = (kPieces * kPieceRow + 3 * QED_MAX_TABLE_N) * (int)sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(table_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDyn);
    if (e == cudaSuccess) {
        bessel_pieces_kernel<<<kPieces, 128, 0, st>>>(a.pieces);
        row_nodes_kernel<<<dim3((m + 3) / 4, 2), 128, 0, st>>>(a, gl);
        table_rows_kernel<<<params->qs.n_chi + params->bw.n_chi, 256, dyn, st>>>(a);
        e = cudaGetLastError();
    }
    // every entry must be finite (a chi range whose rates underflow FP64 is
    // rejected): ln G and ln T lie next to each other, one copy
    const size_t n_g = params->qs.n_chi, off_t = t->d_bw_lnT - t->d_qs_lnG, n_one = off_t + params->bw.n_chi;
    std::vector<double> one(n_one);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(one.data(), t->d_qs_lnG, n_one * sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        qed_tables_destroy(t);
        QED_FAIL(QED_ERR_CUDA, "table generation failed: %s", cudaGetErrorString(e));
    }
    for (size_t i = 0; i < n_one; ++i)
        if ((i < n_g || i >= off_t) && !std::isfinite(one[i])) {
            qed_tables_destroy(t);
            QED_FAIL(QED_ERR_NUMERIC, "ln %s is not finite over the requested %s range", i < n_g ? "G" : "T",
                     i < n_g ? "chi" : "chi_gamma");
        }
    if ((s = finish_tables(t, st))) {
        qed_tables_destroy(t);
        return s;
    }
    *out = t;
    return QED_OK;
}
