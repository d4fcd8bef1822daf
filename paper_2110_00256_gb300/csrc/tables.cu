// tables.cu -- the library-owned lookup tables (§3.1, §3.2): creation from host
// arrays, FP32 copies (§3.3: computed in double, stored in single), views for
// kernels, host copies, and a checked binary file format.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "physics.cuh"

namespace qed {

static qed_status check_axis(const qed_table_axis &a, const char *name, bool qs)
{
    if (!(a.chi_min > 0.0) || !(a.chi_max > a.chi_min) || !std::isfinite(a.chi_max))
        QED_FAIL(QED_ERR_INVALID_ARG, "%s: need 0 < chi_min < chi_max (got %g, %g)", name, a.chi_min, a.chi_max);
    if (a.n_chi < 2 || a.n_chi > QED_MAX_TABLE_N || a.n_xi < 2 || a.n_xi > QED_MAX_TABLE_N)
        QED_FAIL(QED_ERR_INVALID_ARG, "%s: n_chi, n_xi must be in [2, %d] (got %d, %d)", name, QED_MAX_TABLE_N, a.n_chi, a.n_xi);
    if (qs && !(a.xi_min > 0.0 && a.xi_min < 1.0))
        QED_FAIL(QED_ERR_INVALID_ARG, "%s: need 0 < xi_min < 1 (got %g)", name, a.xi_min);
    return QED_OK;
}

qed_status alloc_tables(const qed_table_params *p, qed_tables **out, size_t scratch = 0);

qed_status check_params(const qed_table_params *p)
{
    if (p == nullptr) QED_FAIL(QED_ERR_INVALID_ARG, "params is NULL");
    qed_status s = check_axis(p->qs, "qs", true);
    if (s) return s;
    return check_axis(p->bw, "bw", false);
}

// Rows of the FP32 2-D tables lie pitch32() apart: a draw's hot columns (where P is
// large) are one or two of a row's 128-byte lines, and at a power-of-two distance
// the rows' hot lines share a fraction of the cache's sets -- how large a one then
// hangs on where the arrays happen to lie.  5e7 FP32 draws from 256x256 tables, ten
// tables of a process: ln P 941 us wherever they lie (256 floats apart, in separate
// allocations: 931 to 1380, mean 1104).  P, whose hot columns spread over the row, still
// hangs on the place: 1143 to 1553 us, mean 1298 (separate allocations: 1137 to 1676,
// mean 1304); no pad from 0 to 160 floats and no gap up to 1 MB held for every place.
static int pitch32(int n_xi) { return (n_xi + 31) / 32 * 32 + 32; }

// Everything formed entry by entry from the FP64 tables, in one launch: the
// column differences d[n][m] = v[n][m+1] - v[n][m] of both 2-D tables in FP64 (0
// in the last column) and the FP32 copies of all six.  blockIdx.y: process.
struct Derived {
    const double *one[2], *two[2];
    double *diff[2];
    float *f_one[2], *f_two[2], *f_diff[2];
    int n_chi[2], n_xi[2], pitch32[2];
};

__global__ void derive_kernel(const Derived t)
{
    const int p = blockIdx.y, cols = t.n_xi[p];
    const int64_t n = (int64_t)t.n_chi[p] * cols;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double v = t.two[p][i];
        const double d = (int)(i % cols) + 1 < cols ? t.two[p][i + 1] - v : 0.0;
        t.diff[p][i] = d;
        const int64_t k = i / cols * t.pitch32[p] + i % cols;
        t.f_diff[p][k] = __double2float_rn(d);
        t.f_two[p][k] = __double2float_rn(v);
        if (i < t.n_chi[p]) t.f_one[p][i] = __double2float_rn(t.one[p][i]);
    }
}

// Guide table of one 2-D table: for row n and edge e of kGuideBins equal bins
// of the draw r (QS: r in (0, 1], searched as ln r; BW: r in [0, 1/2]), the
// largest m with v[n][m] <= edge (0 if none); edge 0 is -inf, the last +inf.
// A draw in bin b then lies between the rows' guides at b and b + 1.
template <typename T>
__device__ void guide_entry(const T *__restrict__ v, int n_xi, int pitch, bool qs, int32_t *__restrict__ g)
{
    const int n = blockIdx.x, e = threadIdx.x;
    int32_t out;
    if (e == 0) {
        out = 0;
    } else if (e == kGuideBins) {
        out = n_xi - 1;
    } else {
        const T x = qs ? d_log(T(e) / T(kGuideBins)) : T(e) / T(2 * kGuideBins);
        const T *row = v + (size_t)n * pitch;
        int lo = 0, hi = n_xi;  // largest m with row[m] <= x: row[lo] <= x (or lo == 0), row[hi] > x
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (row[mid] <= x)
                lo = mid;
            else
                hi = mid;
        }
        out = lo;
    }
    g[(size_t)n * (kGuideBins + 1) + e] = out;
}

// row blockIdx.x, process blockIdx.y, precision blockIdx.z
__global__ void guide_kernel(const Derived t, int32_t *qs_d, int32_t *bw_d, int32_t *qs_f, int32_t *bw_f)
{
    const int p = blockIdx.y;
    if ((int)blockIdx.x >= t.n_chi[p] || threadIdx.x > kGuideBins) return;
    if (blockIdx.z)
        guide_entry<float>(t.f_two[p], t.n_xi[p], t.pitch32[p], p == 0, p ? bw_f : qs_f);
    else
        guide_entry<double>(t.two[p], t.n_xi[p], t.n_xi[p], p == 0, p ? bw_d : qs_d);
}

static void free_tables(qed_tables *t)
{
    if (!t) return;
    if (t->block) cudaFree(t->block);
    delete t;
}

static size_t n_qs2(const qed_table_params &p) { return (size_t)p.qs.n_chi * p.qs.n_xi; }
static size_t n_bw2(const qed_table_params &p) { return (size_t)p.bw.n_chi * p.bw.n_xi; }

// a 1-D table's axis on integers (fixed64.cuh), in extended precision; a table
// whose logarithms the integers cannot hold (ok = 0) takes the FP64 path
static FixAxis fix_axis(const qed_table_axis &a)
{
    FixAxis f;
    memset(&f, 0, sizeof(f));
    const long double one = 9007199254740992.0L;  // 2^53
    const long double l0 = std::log((long double)a.chi_min), l1 = std::log((long double)a.chi_max);
    f.n = a.n_chi;
    if (!(l0 > -700.0L) || !(l1 < 700.0L)) return f;
    f.ln_min = (long long)rintl(l0 * one);
    f.ln_max = (long long)rintl(l1 * one);
    if (f.ln_max - f.ln_min < 4096) return f;
    const uint64_t d = (uint64_t)(f.ln_max - f.ln_min);
    int bits = 0;
    while ((a.n_chi - 1) >> bits) ++bits;
    while ((d << (f.shift + 1)) < (1ull << 62)) ++f.shift;
    f.frac = 60 - bits;
    f.scale = fix_limbs((int64_t)rintl((long double)(a.n_chi - 1) / ((long double)d * std::ldexp(1.0L, f.shift)) *
                                       std::ldexp(1.0L, f.frac + 62)));
    f.ok = 1;
    return f;
}

qed_status alloc_tables(const qed_table_params *p, qed_tables **out, size_t scratch)
{
    qed_tables *t = new qed_tables();
    memset(t, 0, sizeof(*t));
    t->params = *p;
    t->qs_fix = fix_axis(p->qs);
    t->bw_fix = fix_axis(p->bw);
    cudaGetDevice(&t->device);
    // one allocation (an allocation and a release each for the 16 arrays were
    // most of a table generation's host time): the four FP64 tables, then what is
    // formed from them, with at least `scratch` bytes there
    size_t size = 0;
    const auto place = [&](auto *&ptr, size_t n) {  // offsets first (block == NULL), then addresses
        ptr = (std::remove_reference_t<decltype(ptr)>)((uintptr_t)t->block + size);
        size += (n * sizeof(*ptr) + 255) / 256 * 256;
    };
    const size_t n1[2] = {(size_t)p->qs.n_chi, (size_t)p->bw.n_chi}, n2[2] = {n_qs2(*p), n_bw2(*p)};
    for (int pass = 0; pass < 2; ++pass) {
        size = 0;
        place(t->d_qs_lnG, n1[0]), place(t->d_bw_lnT, n1[1]), place(t->d_qs_lnP, n2[0]), place(t->d_bw_P, n2[1]);
        t->derived = (void *)((uintptr_t)t->block + size);
        const size_t least = size + scratch;
        const size_t f2[2] = {n1[0] * pitch32(p->qs.n_xi), n1[1] * pitch32(p->bw.n_xi)};
        place(t->f_qs_lnG, n1[0]), place(t->f_bw_lnT, n1[1]);
        place(t->f_qs_lnP, f2[0]), place(t->f_qs_dlnP, f2[0]), place(t->f_qs_guide, n1[0] * (kGuideBins + 1));
        place(t->f_bw_P, f2[1]), place(t->f_bw_dP, f2[1]), place(t->f_bw_guide, n1[1] * (kGuideBins + 1));
        place(t->d_qs_dlnP, n2[0]), place(t->d_qs_guide, n1[0] * (kGuideBins + 1));
        place(t->d_bw_dP, n2[1]), place(t->d_bw_guide, n1[1] * (kGuideBins + 1));
        if (size < least) size = least;
        if (pass) break;
        const cudaError_t e = cudaMalloc(&t->block, size);
        if (e != cudaSuccess) {
            delete t;
            QED_FAIL(QED_ERR_CUDA, "table allocation failed: %s", cudaGetErrorString(e));
        }
    }
    *out = t;
    return QED_OK;
}

// round the FP64 tables into the FP32 copies on `stream`, then the guides
qed_status finish_tables(qed_tables *t, cudaStream_t st)
{
    const qed_table_params &p = t->params;
    const Derived d{{t->d_qs_lnG, t->d_bw_lnT}, {t->d_qs_lnP, t->d_bw_P},     {t->d_qs_dlnP, t->d_bw_dP},
                    {t->f_qs_lnG, t->f_bw_lnT}, {t->f_qs_lnP, t->f_bw_P},     {t->f_qs_dlnP, t->f_bw_dP},
                    {p.qs.n_chi, p.bw.n_chi},   {p.qs.n_xi, p.bw.n_xi},
                    {pitch32(p.qs.n_xi), pitch32(p.bw.n_xi)}};
    const size_t most = n_qs2(p) > n_bw2(p) ? n_qs2(p) : n_bw2(p);
    const unsigned blocks = (unsigned)((most + 255) / 256 < 1024 ? (most + 255) / 256 : 1024);
    derive_kernel<<<dim3(blocks, 2), 256, 0, st>>>(d);
    QED_LAUNCH_CHECK();
    const unsigned rows = (unsigned)(p.qs.n_chi > p.bw.n_chi ? p.qs.n_chi : p.bw.n_chi);
    guide_kernel<<<dim3(rows, 2, 2), kGuideBins + 1, 0, st>>>(d, t->d_qs_guide, t->d_bw_guide, t->f_qs_guide,
                                                              t->f_bw_guide);
    QED_LAUNCH_CHECK();
    QED_CUDA_TRY(cudaStreamSynchronize(st));
    return QED_OK;
}

template <typename T>
static Table1D<T> view1(const T *f, const qed_table_axis &a, const FixAxis &fix)
{
    Table1D<T> v;
    v.ln_f = f;
    const double l0 = std::log(a.chi_min), l1 = std::log(a.chi_max);
    v.ln_min = (T)l0;
    v.inv_d = (T)((a.n_chi - 1) / (l1 - l0));
    v.chi_min = (T)a.chi_min;
    v.chi_max = (T)a.chi_max;
    v.n = a.n_chi;
    v.fix = fix;
    return v;
}

template <typename T>
static Table2D<T> view2(const T *f, const T *df, const int32_t *guide, const qed_table_axis &a, const FixAxis &fix,
                        bool qs)
{
    Table2D<T> v;
    v.fix = fix;
    v.dx_fix = Fix{0, 0};
    v.dx_shift = 0;
    v.v = f;
    v.dv = df;
    v.guide = guide;
    const double l0 = std::log(a.chi_min), l1 = std::log(a.chi_max);
    v.ln_min = (T)l0;
    v.inv_d = (T)((a.n_chi - 1) / (l1 - l0));
    v.chi_min = (T)a.chi_min;
    v.chi_max = (T)a.chi_max;
    v.n_chi = a.n_chi;
    v.n_xi = a.n_xi;
    v.pitch = sizeof(T) == 4 ? pitch32(a.n_xi) : a.n_xi;
    const double dx = qs ? -std::log(a.xi_min) / (a.n_xi - 1) : 0.5 / (a.n_xi - 1);
    v.x0 = qs ? (T)std::log(a.xi_min) : (T)0;
    v.dx = (T)dx;
    const int s = 61 - std::ilogb(dx);
    if (s <= 100 && (s >= 63 || !qs)) v.dx_shift = s, v.dx_fix = fix_limbs((int64_t)std::ldexp(dx, s));
    return v;
}

template <>
TablesView<double> make_view<double>(const qed_tables *t)
{
    TablesView<double> v;
    v.qs_G = view1<double>(t->d_qs_lnG, t->params.qs, t->qs_fix);
    v.bw_T = view1<double>(t->d_bw_lnT, t->params.bw, t->bw_fix);
    v.qs_P = view2<double>(t->d_qs_lnP, t->d_qs_dlnP, t->d_qs_guide, t->params.qs, t->qs_fix,
                           true);
    v.bw_P = view2<double>(t->d_bw_P, t->d_bw_dP, t->d_bw_guide, t->params.bw, t->bw_fix, false);
    return v;
}

template <>
TablesView<float> make_view<float>(const qed_tables *t)
{
    TablesView<float> v;
    v.qs_G = view1<float>(t->f_qs_lnG, t->params.qs, t->qs_fix);
    v.bw_T = view1<float>(t->f_bw_lnT, t->params.bw, t->bw_fix);
    v.qs_P = view2<float>(t->f_qs_lnP, t->f_qs_dlnP, t->f_qs_guide, t->params.qs, t->qs_fix,
                           true);
    v.bw_P = view2<float>(t->f_bw_P, t->f_bw_dP, t->f_bw_guide, t->params.bw, t->bw_fix, false);
    return v;
}

}  // namespace qed

using namespace qed;

extern "C" qed_status qed_tables_create(const qed_table_params *params, const double *qs_lnG,
                                        const double *qs_lnP, const double *bw_lnT,
                                        const double *bw_P, qed_tables **out, void *stream)
{
    clear_error();
    if (out == nullptr) QED_FAIL(QED_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    qed_status s = check_params(params);
    if (s) return s;
    if (!qs_lnG || !qs_lnP || !bw_lnT || !bw_P) QED_FAIL(QED_ERR_INVALID_ARG, "a table array is NULL");
    qed_tables *t = nullptr;
    if ((s = alloc_tables(params, &t))) return s;
    cudaStream_t st = as_stream(stream);
    const qed_table_params &p = *params;
    const size_t sz[4] = {(size_t)p.qs.n_chi, n_qs2(p), (size_t)p.bw.n_chi, n_bw2(p)};
    const double *src[4] = {qs_lnG, qs_lnP, bw_lnT, bw_P};
    double *dst[4] = {t->d_qs_lnG, t->d_qs_lnP, t->d_bw_lnT, t->d_bw_P};
    for (int k = 0; k < 4; ++k) {
        cudaError_t e = cudaMemcpyAsync(dst[k], src[k], sz[k] * sizeof(double), cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) {
            free_tables(t);
            QED_FAIL(QED_ERR_CUDA, "table upload failed: %s", cudaGetErrorString(e));
        }
    }
    if ((s = finish_tables(t, st))) {
        free_tables(t);
        return s;
    }
    *out = t;
    return QED_OK;
}

extern "C" qed_status qed_tables_copy_to_host(const qed_tables *t, double *qs_lnG, double *qs_lnP,
                                              double *bw_lnT, double *bw_P)
{
    clear_error();
    qed_status s = check_tables(t);
    if (s) return s;
    const qed_table_params &p = t->params;
    const size_t sz[4] = {(size_t)p.qs.n_chi, n_qs2(p), (size_t)p.bw.n_chi, n_bw2(p)};
    const double *src[4] = {t->d_qs_lnG, t->d_qs_lnP, t->d_bw_lnT, t->d_bw_P};
    double *dst[4] = {qs_lnG, qs_lnP, bw_lnT, bw_P};
    for (int k = 0; k < 4; ++k)
        if (dst[k]) QED_CUDA_TRY(cudaMemcpy(dst[k], src[k], sz[k] * sizeof(double), cudaMemcpyDeviceToHost));
    return QED_OK;
}

extern "C" qed_status qed_tables_get_params(const qed_tables *t, qed_table_params *out)
{
    clear_error();
    qed_status s = check_tables(t);
    if (s) return s;
    if (!out) QED_FAIL(QED_ERR_INVALID_ARG, "out is NULL");
    *out = t->params;
    return QED_OK;
}

extern "C" qed_status qed_tables_destroy(qed_tables *t)
{
    clear_error();
    free_tables(t);
    return QED_OK;
}

// ---------------------------------------------------------------------------
// file format: "QEDTAB\0\1" | u32 version | params (5 doubles/ints per axis) |
// qs_lnG | qs_lnP | bw_lnT | bw_P (FP64, little-endian host order) | u64 FNV-1a
// ---------------------------------------------------------------------------
static const char kMagic[8] = {'Q', 'E', 'D', 'T', 'A', 'B', 0, 1};
static const uint32_t kFileVersion = 1;

static void put_axis(std::vector<unsigned char> &buf, const qed_table_axis &a)
{
    auto put = [&](const void *p, size_t n) { buf.insert(buf.end(), (const unsigned char *)p, (const unsigned char *)p + n); };
    put(&a.chi_min, 8);
    put(&a.chi_max, 8);
    put(&a.n_chi, 4);
    put(&a.n_xi, 4);
    put(&a.xi_min, 8);
}

extern "C" qed_status qed_tables_save(const qed_tables *t, const char *path)
{
    clear_error();
    qed_status s = check_tables(t);
    if (s) return s;
    if (!path) QED_FAIL(QED_ERR_INVALID_ARG, "path is NULL");
    const qed_table_params &p = t->params;
    std::vector<double> a(p.qs.n_chi), b(n_qs2(p)), c(p.bw.n_chi), d(n_bw2(p));
    if ((s = qed_tables_copy_to_host(t, a.data(), b.data(), c.data(), d.data()))) return s;
    std::vector<unsigned char> buf;
    buf.insert(buf.end(), kMagic, kMagic + 8);
    buf.insert(buf.end(), (const unsigned char *)&kFileVersion, (const unsigned char *)&kFileVersion + 4);
    put_axis(buf, p.qs);
    put_axis(buf, p.bw);
    for (auto *v : {&a, &b, &c, &d})
        buf.insert(buf.end(), (const unsigned char *)v->data(), (const unsigned char *)(v->data() + v->size()));
    const uint64_t h = fnv1a64(buf.data(), buf.size());
    FILE *f = fopen(path, "wb");
    if (!f) QED_FAIL(QED_ERR_IO, "cannot open %s for writing", path);
    bool ok = fwrite(buf.data(), 1, buf.size(), f) == buf.size() && fwrite(&h, 8, 1, f) == 1;
    ok = (fclose(f) == 0) && ok;
    if (!ok) QED_FAIL(QED_ERR_IO, "write to %s failed", path);
    return QED_OK;
}

extern "C" qed_status qed_tables_load(const char *path, qed_tables **out, void *stream)
{
    clear_error();
    if (!path || !out) QED_FAIL(QED_ERR_INVALID_ARG, "path/out is NULL");
    *out = nullptr;
    FILE *f = fopen(path, "rb");
    if (!f) QED_FAIL(QED_ERR_IO, "cannot open %s", path);
    std::vector<unsigned char> buf;
    unsigned char chunk[1 << 16];
    size_t n;
    while ((n = fread(chunk, 1, sizeof(chunk), f)) > 0) buf.insert(buf.end(), chunk, chunk + n);
    fclose(f);
    const size_t head = 8 + 4 + 2 * 32;
    if (buf.size() < head + 8) QED_FAIL(QED_ERR_IO, "%s: file too short", path);
    if (memcmp(buf.data(), kMagic, 8) != 0) QED_FAIL(QED_ERR_IO, "%s: bad magic", path);
    uint32_t ver;
    memcpy(&ver, buf.data() + 8, 4);
    if (ver != kFileVersion) QED_FAIL(QED_ERR_IO, "%s: unsupported version %u", path, ver);
    qed_table_params p;
    const unsigned char *q = buf.data() + 12;
    for (qed_table_axis *a : {&p.qs, &p.bw}) {
        memcpy(&a->chi_min, q, 8);
        memcpy(&a->chi_max, q + 8, 8);
        memcpy(&a->n_chi, q + 16, 4);
        memcpy(&a->n_xi, q + 20, 4);
        memcpy(&a->xi_min, q + 24, 8);
        q += 32;
    }
    qed_status s = check_params(&p);
    if (s) QED_FAIL(QED_ERR_IO, "%s: bad table parameters", path);
    const size_t body = 8 * ((size_t)p.qs.n_chi + n_qs2(p) + (size_t)p.bw.n_chi + n_bw2(p));
    if (buf.size() != head + body + 8) QED_FAIL(QED_ERR_IO, "%s: size mismatch", path);
    uint64_t h;
    memcpy(&h, buf.data() + head + body, 8);
    if (h != fnv1a64(buf.data(), head + body)) QED_FAIL(QED_ERR_IO, "%s: checksum mismatch", path);
    const double *d = (const double *)(buf.data() + head);
    std::vector<double> arr(body / 8);
    memcpy(arr.data(), d, body);
    const double *a0 = arr.data();
    const double *a1 = a0 + p.qs.n_chi;
    const double *a2 = a1 + n_qs2(p);
    const double *a3 = a2 + p.bw.n_chi;
    return qed_tables_create(&p, a0, a1, a2, a3, out, stream);
}
