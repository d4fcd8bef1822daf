"""Particles whose force nearly cancels (along a wave, crossed fields, E along p) on the integers of csrc/fixed64.cuh: taken
there, and chi and the rate no further from extended precision than the FP64 path's."""
import numpy as np
import pytest

from host_build import compile_shim
from test_fixed_host import particles, run

N = 20_000


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return compile_shim("fixed_shim.cpp", tmp_path_factory.mktemp("guard"))


def along(angle, seed=3):
    """Within `angle` of a linearly polarised wave's direction, gamma up to 4000."""
    r = np.random.default_rng(seed)
    g, a, b = np.exp(r.uniform(np.log(2.0), np.log(4000.0), N)), r.normal(size=N) * angle, r.normal(size=N) * angle
    p = np.zeros((9, N))
    p[0], p[1], p[2] = g * np.cos(a) * np.cos(b), g * np.sin(a), g * np.sin(b) * np.cos(a)
    p[4] = p[8] = 0.01 * np.cos(r.uniform(0, 6.283, N))
    return p


def crossed(spread):
    """E across p and B = n x E within `spread`, in every direction."""
    p = particles("gauss", N, 8)
    n = p[:3] / np.sqrt((p[:3] ** 2).sum(0))
    p[3:6] -= n * (n * p[3:6]).sum(0)
    p[6:] = np.cross(n.T, p[3:6].T).T * (1 + spread * np.random.default_rng(2).normal(size=(3, N)))
    return p


def e_along_p():
    p = particles("gauss", N, 8)
    p[6:] = 0.0
    p[3:6] = p[:3] * 1e-6 * (1 + 0.01 * np.random.default_rng(1).normal(size=(3, N)))
    return p


KINDS = {f"along {a}": (lambda a=a: along(a)) for a in (1.0, 0.3, 0.1, 0.03, 0.01, 0.003, 0.001)}
KINDS |= {"crossed": lambda: crossed(0.003), "E along p": e_along_p}


@pytest.mark.parametrize("qs", [True, False])
@pytest.mark.parametrize("kind", KINDS)
@np.errstate(divide="ignore", invalid="ignore")
def test_cancelling_forces(lib, qs, kind):
    rate, _, chi, ok, (r_ref, c_ref, _), (r_64, c_64, _) = run(lib, qs, KINDS[kind]())
    assert ok.mean() > 0.999
    sel = ok & (r_ref > 1e-280)
    if not sel.any():
        return  # (photons whose rate is zero)
    for got, f64, ref in ((chi, c_64, c_ref), (rate, r_64, r_ref)):
        e, e64 = (np.abs(x[sel] / ref[sel] - 1).astype(np.float64) for x in (got, f64))
        assert np.sqrt(np.mean(e ** 2)) <= np.sqrt(np.mean(e64 ** 2)) and e.max() <= e64.max()


def test_a_force_that_fp64_holds_is_left_to_it(lib):
    """No E, and p and B along one axis but for small components: each product of FP64 is small, and its rounding too."""
    r = np.random.default_rng(4)
    p = np.zeros((9, N))
    p[0], p[6] = 1000.0, 0.01
    p[1:3] = r.normal(size=(2, N))
    p[7:] = 1e-6 * r.normal(size=(2, N))
    assert not run(lib, True, p)[3].any()


@np.errstate(divide="ignore", invalid="ignore")
def test_leptons_at_rest(lib):
    """No momentum, or one far below 1 (subnormal too): chi = |E| and the rate as exact as the FP64 path's; taken where E is
    of the fields' size (elsewhere FP64 holds gamma E better than a block scaled by B)."""
    p = particles("gauss", N, 6)
    p[:3] = 0.0
    p[0, ::4] = 1e-310
    p[1, 1::4] = -1e-200
    p[:3, 2::4] = 1e-30
    rate, _, chi, ok, (r_ref, c_ref, _), (r_64, c_64, _) = run(lib, True, p)
    assert ok[np.abs(p[3:6]).max(0) >= np.abs(p[6:]).max(0) / 4].all() and ok.mean() > 0.9
    assert np.all(np.abs(chi[ok] / c_ref[ok] - 1) <= 2.0 ** -51)
    e, e64 = (np.abs(x[ok] / r_ref[ok] - 1).astype(np.float64) for x in (rate, r_64))
    assert np.sqrt(np.mean(e ** 2)) <= np.sqrt(np.mean(e64 ** 2)) and e.max() <= e64.max()
