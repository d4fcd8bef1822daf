"""The FP64 inverse CDF of photon emission (csrc/physics.cuh), compiled for the host,
against the same interpolation in extended precision."""
import ctypes

import numpy as np
import pytest

import oracle
from host_build import compile_shim, ptr

LD = np.longdouble
EPS = LD(2) ** -53
N_CHI, N_XI, LO, HI, XI_MIN = 48, 80, 1e-3, 1e3, 1e-12


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return compile_shim("sampling_shim.cpp", tmp_path_factory.mktemp("sampling"))


@pytest.fixture(scope="module")
def rows():
    t = oracle.tables(qs_chi_min=LO, qs_chi_max=HI, qs_n_chi=N_CHI, qs_n_xi=N_XI, qs_xi_min=XI_MIN, bw_n_chi=8, bw_n_xi=8)
    return np.ascontiguousarray(t.qs_lnP, dtype=np.float64).reshape(N_CHI, N_XI)


def draws(lib, rows, chi, r):
    """xi by the integers, which draws they took, by the general form and with FP64 logarithms throughout."""
    n = r.size
    out, ok = [np.zeros(n) for _ in range(3)], np.zeros(n, dtype=np.int32)
    lib.host_qs(N_CHI, N_XI, ctypes.c_double(LO), ctypes.c_double(HI), ctypes.c_double(XI_MIN), ptr(rows),
                ctypes.c_int64(n), ptr(chi), ptr(r), ptr(out[0]), ptr(ok), ptr(out[1]), ptr(out[2]))
    return out[0], ok.astype(bool), out[1], out[2]


def reference(rows, chi, r):
    """xi in extended precision, and a bound of its relative error by roundings of the rows, of ln r and of the weight
    between the rows (2^-53 of their magnitudes, the weight's by the logarithms in it), and of ln xi."""
    lr = np.where(r > 0.5, np.log1p((r - 1.0).astype(LD)), np.log(r.astype(LD)))
    l0, l1, lc = np.log(LD(LO)), np.log(LD(HI)), np.log(chi.astype(LD))
    pos = np.clip((lc - l0) * (N_CHI - 1) / (l1 - l0), 0, N_CHI - 1)
    k = np.minimum(pos.astype(int), N_CHI - 2)
    a, b = rows[k].astype(LD), rows[k + 1].astype(LD)
    row = a + (pos - k)[:, None] * (b - a)
    m, i = np.clip((row <= lr[:, None]).sum(axis=1) - 1, 0, N_XI - 2), np.arange(r.size)
    dp = row[i, m + 1] - row[i, m]
    f = (lr - row[i, m]) / dp
    dx = LD(-np.log(XI_MIN) / (N_XI - 1))
    y = np.minimum((m + f - (N_XI - 1)) * dx, 0)
    err_w = 4 * EPS * (np.abs(lc) + abs(l0)) * (N_CHI - 1) / (l1 - l0)
    err_p = 3 * EPS * np.abs(row[i, m]) + err_w * np.maximum(np.abs(b - a)[i, m], np.abs(b - a)[i, m + 1]) + EPS * np.abs(lr)
    return np.exp(y), err_p * (1 + np.abs(f)) / dp * dx + 4 * EPS * (1 + np.abs(y) + abs(np.log(LD(XI_MIN))))


def test_photon_sampling_on_integers(lib, rows):
    """A draw's xi on the integers is the interpolation's, whatever order a compiler evaluates arguments in."""
    rng = np.random.default_rng(3)
    n = 40_000
    chi = np.exp(rng.uniform(np.log(LO), np.log(HI), n))
    r = np.exp(rng.uniform(np.log(2.0 ** -20), 0.0, n))
    r[::2] = rng.uniform(0.0, 0.95, r[::2].size)
    xi, ok, general, _ = draws(lib, rows, chi, r)
    assert ok.mean() > 0.8
    ref, tol = reference(rows, chi, r)
    assert np.all(np.abs(xi[ok] / ref[ok] - 1) <= tol[ok])
    assert np.all(np.abs(general / ref - 1) <= tol)


def rms(x):
    return float(np.sqrt(np.mean(np.asarray(x, dtype=np.float64) ** 2)))


@pytest.mark.parametrize("e", [*range(1, 20), 23, 27, 31, 35, 39, 43])
def test_hard_photons_are_no_further_off_than_in_fp64(lib, rows, e):
    """1 - r in [2^-(e+1), 2^-e]: the draw as the library makes it (integers, else the general form) has an rms error no
    larger than the general form with FP64 logarithms; 2 % for what the two share, the table's arithmetic in FP64."""
    rng = np.random.default_rng(100 + e)
    n = 20_000
    chi = np.exp(rng.uniform(np.log(LO), np.log(HI), n))
    r = 1.0 - 2.0 ** -e * rng.uniform(0.5, 1.0, n)
    xi, ok, general, tang = draws(lib, rows, chi, r)
    ref, _ = reference(rows, chi, r)
    now = np.where(ok, xi, general)
    assert rms(now / ref - 1) <= 1.02 * rms(tang / ref - 1)


@pytest.mark.parametrize("lo,hi", [(2.0 ** -(k + 1), 2.0 ** -k) for k in range(16)] + [(1, 2), (2, 4), (4, 8), (8, 16), (16, 36)])
def test_optical_depth_draws_are_no_further_off_than_in_fp64(lib, lo, hi):
    """-ln U over its octaves, U with 53 random bits: rms and largest error no larger than with the table-driven FP64
    logarithm (the series above U = 1 - 2^-8 is the same in both), and the largest at most 1.5 roundings (2^-53)."""
    rng = np.random.default_rng(7)
    n = 200_000
    v = np.exp(-rng.uniform(lo, hi, n))
    bits = (np.minimum((v * 2.0 ** 53).astype(np.uint64), np.uint64(2 ** 53 - 1)) << np.uint64(11)) | rng.integers(
        0, 2048, n, dtype=np.uint64)
    w0, w1 = (bits & np.uint64(0xffffffff)).astype(np.uint32), (bits >> np.uint64(32)).astype(np.uint32)
    u, tau, tang = np.zeros(n), np.zeros(n), np.zeros(n)
    lib.host_draw(ctypes.c_int64(n), ptr(w0), ptr(w1), ptr(u), ptr(tau), ptr(tang))
    ref = np.where(u > 0.5, -np.log1p((u - 1.0).astype(LD)), -np.log(u.astype(LD)))
    err, err64 = (np.abs(x / ref - 1).astype(np.float64) for x in (tau, tang))
    assert rms(err) <= rms(err64) and err.max() <= err64.max() and err.max() <= 1.5 * 2.0 ** -53


@np.errstate(all="ignore")
def test_logarithm_and_exponential_of_the_rates_fp64_form(lib):
    """On the integers within their range (e^x: x rounded to 2^-53 where that is coarser, the integers' 2^-58, one rounding;
    ln x: 2^-57 and one rounding), the table-driven forms' values beyond it and for IEEE's special values."""
    rng = np.random.default_rng(11)
    x = np.concatenate([rng.uniform(-690, 690, 200_000), rng.uniform(-1, 1, 100_000), 10.0 ** rng.uniform(-25, 0, 50_000),
                        2.0 ** rng.uniform(-1074, 1023, 50_000), -2.0 ** rng.uniform(-1074, 10, 50_000),
                        [0.0, -0.0, np.inf, -np.inf, np.nan, 690.0, -690.0, np.nextafter(690, 0), -np.nextafter(690, 0), 5e-324, -1.0]])
    e, e64, ln, l64 = (np.zeros(x.size) for _ in range(4))
    lib.host_logexp(ctypes.c_int64(x.size), ptr(x), ptr(e), ptr(e64), ptr(ln), ptr(l64))
    ins = np.abs(x) < 690
    assert np.all(np.abs(e[ins] / np.exp(x[ins].astype(LD)) - 1) <= 2.0 ** -53 + 2.0 ** -54 + 2.0 ** -58)
    assert np.array_equal(e[~ins], e64[~ins], equal_nan=True)
    pos = (x >= 2.0 ** -86) & (x < 2.0 ** 86)
    ref = np.log(x[pos].astype(LD))
    assert np.all(np.abs(ln[pos] - ref) <= 2.0 ** -57 + 2.0 ** -53 * np.abs(ref))
    assert np.array_equal(ln[~pos], l64[~pos], equal_nan=True)
