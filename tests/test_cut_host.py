"""The FP64 evolution's chi cut-offs on 64-bit integers (csrc/fixed64.cuh), compiled for the host: which
side of a cut-off a particle is on, and which particles are left to the FP64 form."""
import ctypes

import numpy as np
import pytest

from host_build import compile_shim, ptr

LD = np.longdouble


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return compile_shim("sampling_shim.cpp", tmp_path_factory.mktemp("cut"))


def sides(lib, cut, ln_chi):
    ln_chi = np.ascontiguousarray(ln_chi, dtype=np.int64)
    out, lc = np.zeros(ln_chi.size, dtype=np.int32), np.zeros(1, dtype=np.int64)
    lib.host_cut(ctypes.c_double(cut), ctypes.c_int64(ln_chi.size), ptr(ln_chi), ptr(lc), ptr(out))
    return int(lc[0]), out


@pytest.mark.parametrize("cut", [1e-3, 0.02, np.nextafter(1.0, 0.0), 1.0, np.nextafter(1.0, 2.0), 15.0, 1e3, 1e-140, 1e140,
                                 3e-216, 3e216])
def test_side_of_a_cut(lib, cut):
    """ln cut to 8 units of 2^-53 (of which it has |ln cut| 2^-10 at most by the width of ln 2's integer); a particle within
    1024 units is near, another one on the side that the extended-precision logarithm gives."""
    exact = int(np.rint(np.log(LD(cut)) * LD(2) ** 53))
    step = np.array([-(1 << 58), -(1 << 40), -2048, -1040, -1000, -9, 9, 1000, 1040, 2048, 1 << 40, 1 << 58])
    ln_cut, side = sides(lib, cut, exact + step)
    assert abs(ln_cut - exact) <= 8
    assert np.array_equal((side & 1) != 0, step < 0)
    assert np.array_equal((side & 2) != 0, np.abs(step) <= 1000)


def test_cuts_that_decide_without_chi(lib):
    """No cut-off (zero, negative) or one far below or above every particle on the integers."""
    far = np.array([-333, -300, 0, 300, 333]) * (1 << 53)
    for cut in (0.0, -0.0, -1.0, -np.inf, 5e-324, 1e-310, 1e-300):
        assert not sides(lib, cut, far)[1].any(), cut
    for cut in (np.inf, 1e300):
        assert np.all(sides(lib, cut, far)[1] == 1), cut
