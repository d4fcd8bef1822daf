"""The FP64 evolution's integer arithmetic (csrc/fixed64.cuh), compiled for the
host, against extended precision: chi and the rate of random and special
particles, beside the same formulas in FP64, and the particles that it must leave
to the FP64 path."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2110_00256_gb300", "csrc")
GEV = 1956.95
LD = np.longdouble


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fixed") / "fixed.so")
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-shared", "-fPIC", "-I", CSRC, os.path.join(HERE, "fixed_shim.cpp"),
                    "-o", so], check=True)
    return ctypes.CDLL(so)


def ln_table(qs, n, lo, hi):
    """A table with the size and slopes of the real ones (their exact values do not matter here)."""
    x = np.linspace(np.log(lo), np.log(hi), n)
    y = np.where(x < 0, 0.9 + x, 0.9 + 0.667 * x) if qs else -1.47 - 2.667 * np.exp(-x) + 0.3 * x
    fixed = np.array([int(round(LD(v) * LD(2) ** 53)) for v in y], dtype=np.int64)
    return y, fixed


def run(lib, qs, p, n_tab=256, lo=None, hi=1e3):
    lo = lo or (1e-3 if qs else 2e-2)
    y, fixed = ln_table(qs, n_tab, lo, hi)
    p = np.ascontiguousarray(p, dtype=np.float64)
    n = p.shape[1]
    rate, lc, chi, ok = np.zeros(n), np.zeros(n), np.zeros(n), np.zeros(n, dtype=np.int32)
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    lib.fixed_rates(int(qs), ctypes.c_int64(n), ptr(p), ctypes.c_double(lo), ctypes.c_double(hi), n_tab, ptr(fixed),
                    ptr(rate), ptr(lc), ptr(chi), ptr(ok))
    return rate, lc, chi, ok.astype(bool), reference(qs, p, y, lo, hi, LD), reference(qs, p, y, lo, hi, np.float64)


def reference(qs, p, y, lo, hi, t):
    """rate / coef, chi and |f| |p| |F| in the type t, the formulas of the FP64 path; f is the force, |p| and |F| the
    largest components (a lepton's |p| at least 1)."""
    p, y = p.astype(t), y.astype(t)
    px, py, pz, ex, ey, ez, bx, by, bz = p
    p2 = px * px + py * py + pz * pz
    g = np.sqrt(p2 + (1 if qs else 0))
    fx, fy, fz = g * ex + (py * bz - pz * by), g * ey + (pz * bx - px * bz), g * ez + (px * by - py * bx)
    pe = px * ex + py * ey + pz * ez
    f2 = fx * fx + fy * fy + fz * fz
    scale = np.sqrt(f2) * np.maximum(np.abs(p[:3]).max(0), 1 if qs else 0) * np.abs(p[3:]).max(0)
    chi = np.sqrt(np.maximum(f2 - pe * pe, 0))
    lc = np.log(chi)
    n = len(y)
    c = np.clip((lc - np.log(t(lo))) * ((n - 1) / (np.log(t(hi)) - np.log(t(lo)))), 0, n - 1)
    i = np.minimum(np.where(np.isfinite(c), c, 0).astype(np.int64), n - 2)
    ln = y[i] + (c - i) * (y[i + 1] - y[i])
    if qs:
        return np.exp(ln) / g, chi, scale
    ln = np.where(chi < lo, t(-1.4712438795175893) - t(8) / 3 / chi, ln)
    ln = np.where(chi > hi, t(-0.9686047877362934) - lc / 3, ln)
    return chi * np.exp(ln) / g, chi, scale


def particles(kind, n, seed):
    r = np.random.default_rng(seed)
    p = np.concatenate([r.uniform(-GEV, GEV, (3, n)), r.uniform(-0.01, 0.01, (6, n))])
    if kind == "gauss":
        p[3:] = r.normal(size=(6, n)) * 10.0 ** r.uniform(-8, -3, n)
    elif kind == "beam":
        p[3:8] = 0.0
        p[8] = 0.01
    elif kind == "slow":
        p[:3] *= 10.0 ** r.uniform(-9, -3, n)
        p[:3, ::10] = 0.0
        p[3:] *= 100.0
    elif kind == "scales":
        p[:3] *= 10.0 ** r.uniform(-8, 0, (3, n))
        p[3:] *= 10.0 ** r.uniform(-2, 6, (6, n))
    elif kind == "wave":  # head-on against a plane wave along -x
        p[0] = 10.0 ** r.uniform(0, 3.3, n)
        p[1], p[2] = p[0] * 0.03 * r.normal(size=n), 0.0
        p[3:] = 0.0
        p[4] = 3e-4 * r.normal(size=n)
        p[8] = -p[4]
    return p


@pytest.mark.parametrize("qs", [True, False])
@pytest.mark.parametrize("kind", ["bench", "gauss", "beam", "slow", "scales", "wave"])
@pytest.mark.parametrize("n_tab", [2, 64, 256, 1024])
@np.errstate(divide="ignore", invalid="ignore")  # (particles at rest in the references)
def test_rate_and_chi_against_extended_precision(lib, qs, kind, n_tab):
    p = particles(kind, 20000, 5)
    rate, lc, chi, ok, (r_ref, c_ref, scale), (r_64, c_64, _) = run(lib, qs, p, n_tab)
    assert ok.mean() > 0.85  # (at rest against strong fields and the widest scales some are left to FP64)
    sel = ok & (r_ref > 1e-280)
    # chi: each component of the force is off by at most 10 units of 2^-60 of the blocks' scale (at
    # most 4 |p| |F|), so chi by sqrt(3) 2^-54.7 |f| |p| |F| / chi^2, the squares by less, and the
    # conversion to FP64 by 2^-52; the rate: those times its slope in ln chi (at most 1 + 8/(3 chi) for pairs below the table), the 2^-53 units of ln chi and of the
    # table values with their interpolation, and one rounding of the result
    slope = 1.0 + np.abs(np.gradient(ln_table(qs, n_tab, 1e-3 if qs else 2e-2, 1e3)[0])).max() * (n_tab - 1) / 10.0
    slope = np.maximum(slope, 1.0 if qs else (1.0 + 8.0 / 3.0 / c_ref).astype(np.float64))
    e_chi = np.abs(chi[sel] / c_ref[sel] - 1).astype(np.float64)
    tol = (2.0 ** -53 * (scale[sel] / c_ref[sel] ** 2) + 2.0 ** -51).astype(np.float64)
    assert np.all(e_chi <= tol)
    assert np.all(np.abs(lc[sel] - np.log(c_ref[sel])) <= tol + 2.0 ** -50 + 2.0 ** -52 * np.abs(lc[sel]))
    e_rate = np.abs(rate[sel] / r_ref[sel] - 1).astype(np.float64)
    assert np.all(e_rate <= tol * slope[sel] if np.ndim(slope) else tol * slope)
    # no less exact than the FP64 path, in the mean and at the worst particle
    e_64 = np.abs(r_64[sel] / r_ref[sel] - 1).astype(np.float64)
    assert np.sqrt(np.mean(e_rate ** 2)) <= np.sqrt(np.mean(e_64 ** 2))
    assert e_rate.max() <= e_64.max()


@pytest.mark.parametrize("qs", [True, False])
def test_what_is_left_to_the_fp64_path(lib, qs):
    n = 64
    p = particles("bench", n, 9)
    for k, v in enumerate((np.nan, np.inf, -np.inf, 1e200, 1e-310)):
        p[k % 3, k] = v if v != 1e-310 else p[k % 3, k]
        p[3 + k, 8 + k] = v if v != 1e-310 else p[3 + k, 8 + k]
    p[:3, 16] = 1e-200  # a block outside 2^+-400 (a lepton's is held at 1)
    p[3:, 17] = 0.0
    p[3:, 18] = 1e-310
    p[3:6, 19], p[6:, 19] = 0.0, p[:3, 19] * 1e-6  # B along p: no force
    p[3:, 20] = 1e160
    with np.errstate(all="ignore"):
        ok = run(lib, qs, p)[3]
    left = [0, 1, 2, 3, 8, 9, 10, 11, 17, 18, 19, 20] + ([] if qs else [16])
    assert not ok[left].any()
    rest = [i for i in range(n) if i not in left and i != 16]
    assert ok[rest].all()


def test_table_ends_of_the_pair_rate_are_left_to_fp64(lib):
    # a photon along x in a field across it: chi = |p| |E|; chi within rounding of the table's ends
    p = np.zeros((9, 4))
    p[0] = 1.0
    p[4] = [2e-2, 1e3, 2.1e-2, 1.9e-2]
    ok = run(lib, False, p)[3]
    assert list(ok) == [False, False, True, True]


def test_logarithm_against_extended_precision(lib):
    """The resets' and the sampling's logarithm: within 2^-57 absolute and one rounding (2^-53 and the integers' 2^-57) where
    the result is not small, over the significands next to every table edge, next to 1 and at random."""
    r = np.random.default_rng(2)
    m = r.integers(1 << 63, 1 << 64, 400_000, dtype=np.uint64)
    edge = (np.arange(256, dtype=np.uint64) << np.uint64(55)) + np.uint64(1 << 63)
    near = np.concatenate([edge, edge - np.uint64(1), edge + np.uint64(1 << 11)])
    near = near[near >= 1 << 63]
    m = np.concatenate([np.repeat(near, 8), (np.uint64(2 ** 64 - 1) - np.arange(1 << 12, dtype=np.uint64) * np.uint64(2048)), m])
    e = r.integers(-63 - 85, -63 + 85, m.size).astype(np.int32)
    e[::3] = -63
    e[1::3] = -64
    out = np.zeros(m.size)
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    lib.fixed_ln(ctypes.c_int64(m.size), ptr(m), ptr(e), ptr(out))
    k = e.astype(np.int64) + 64  # n 2^e = (n 2^-64) 2^k, n 2^-64 in [1/2, 1)
    x = m.astype(LD) / LD(2) ** 64
    # (ln x taken from 1 where k = 0, so that the reference keeps its digits there)
    ref = np.where(k == 0, np.log1p((m - np.uint64(2 ** 63)).astype(LD) / LD(2) ** 64 - LD(0.5)),
                   np.log(x) + k * np.log(LD(2)))
    err = np.abs(out - ref).astype(np.float64)
    assert np.all(err <= 2.0 ** -57 + 2.0 ** -53 * np.abs(ref).astype(np.float64))


def test_roots_and_quotients_against_extended_precision(lib):
    """sqrt, 1/sqrt and a/b: one rounding (2^-53) and the integers' 2^-58; exact squares and powers of two; what is not
    ordinary is refused."""
    r = np.random.default_rng(4)
    n = 300_000
    b = r.uniform(1, 2, n) * 2.0 ** r.integers(-499, 499, n)
    b[:1000] = np.arange(1, 1001, dtype=np.float64) ** 2
    b[1000:1900] = 2.0 ** np.arange(-450, 450)
    b[1900:2900] = 4.0 + np.arange(-500, 500) * 2.0 ** -50
    b[2900:3900] = np.nextafter(1.0, 0.0) - np.arange(1000) * 2.0 ** -53
    a = r.uniform(-2, 2, n) * 2.0 ** r.integers(-400, 400, n)
    a[:1900] = b[:1900] * r.integers(1, 100, 1900)  # exact products
    a[2900:3900] = 1.0
    a = np.where(a == 0, 1.0, a)
    bad = [0.0, -1.0, np.nan, np.inf, 1e-310, 1e200, 1e-200]
    b[-len(bad):] = bad
    root, inv, quot, ok = np.zeros(n), np.zeros(n), np.zeros(n), np.zeros(n, dtype=np.int32)
    ptr = lambda v: v.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    lib.fixed_roots(ctypes.c_int64(n), ptr(a), ptr(b), ptr(root), ptr(inv), ptr(quot), ptr(ok))
    assert not ok[-len(bad):].any() and ok[:-len(bad)].all()
    a, b, root, inv, quot = (v[:-len(bad)] for v in (a, b, root, inv, quot))
    tol = 2.0 ** -53 + 2.0 ** -58
    s = np.sqrt(b.astype(LD))
    assert np.all(np.abs(root / s - 1) <= tol) and np.all(np.abs(inv * s - 1) <= tol)
    assert np.all(np.abs(quot / (a.astype(LD) / b.astype(LD)) - 1) <= tol)
    assert np.array_equal(root[:1000], np.arange(1, 1001)) and np.array_equal(quot[:1900], a[:1900] / b[:1900])
