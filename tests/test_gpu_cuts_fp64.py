"""FP64 chi cut-offs through the evolution's forms: a particle above the cut-off ends with the bits that it has
without one, a particle below keeps its optical depth."""
import numpy as np
import pytest

import oracle
from helpers import as_f64, gpu_tables

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
NAMES = ("electrons", "positrons", "photons")
MOVED = ("px", "py", "pz", "ex", "ey", "ez", "bx", "by", "bz")


@pytest.fixture(scope="module")
def api():
    from paper_2110_00256_gb300 import api as a
    return a


def _optical_depths(api, t, host, form, cuts, caps):
    sp = {k: api.SpeciesBuffers(caps, api.QED_F64, positions=True) for k in NAMES}
    for k in NAMES:
        sp[k].set(host[k])
    fire = [api.FireBuffers(64) for _ in NAMES]
    if form == "substep":
        api.SubstepCall(t, *[sp[k] for k in NAMES], fire, 10.0, 3, qs_chi_cut=cuts[0], bw_chi_cut=cuts[1])(0)
    else:
        b = api.Batch([dict(sp, fire=fire)], api.QED_F64)
        o = api.make_opts(qs_chi_cut=cuts[0], bw_chi_cut=cuts[1])
        if form == "batched":
            api.qed_substep_batched(t, b, 10.0, 3, 0, o)
        else:
            api.qed_push_substep_batched(t, b, api.plane_wave(0.01, 1e-3), 0.0, 10.0, 3, 0, o, store_fields=True)
    torch.cuda.synchronize()
    return {k: sp[k].to_host() for k in NAMES}


@pytest.mark.parametrize("cuts", [(5.0, 8.0), (1e-4, 0.0), (0.0, 20.0), (np.inf, 1e300), (1e-310, 1e-300)])
@pytest.mark.parametrize("form,caps", [("substep", 3001), ("substep", 200_001), ("batched", 3001), ("batched", 200_001),
                                       ("fused", 3001)])
def test_particles_above_a_cut_keep_their_bits(api, oracle_tables_256, form, caps, cuts):
    from paper_2110_00256_gb300 import workloads
    t = gpu_tables(api, oracle_tables_256)
    n = 3000
    host = {k: workloads.paper_benchmark(n, 40 + i, i * 10 ** 9) for i, k in enumerate(NAMES)}
    for k in NAMES:
        host[k]["tau"] = host[k]["tau"] + 1e3  # no events
        host[k] |= {c: np.linspace(0.0, 100.0, n) for c in "xyz"}
    first, chi = _optical_depths(api, t, host, form, (0.0, 0.0), caps), {}
    for k in NAMES:  # an optical depth near its decrement, so that the decrement's last bit counts
        state = as_f64(dict(host[k], **{c: first[k][c] for c in MOVED}), np.float64)
        _, chi[k], rate, _ = oracle.evolve(1 if k == "photons" else 0, oracle_tables_256, state, 10.0)
        host[k]["tau"] = np.where(rate > 1e-200, 1.25 * 10.0 * rate, 1.0)
    without, with_ = (_optical_depths(api, t, host, form, c, caps) for c in ((0.0, 0.0), cuts))
    for k in NAMES:
        cut = cuts[1] if k == "photons" else cuts[0]
        below, above = chi[k] < cut * (1 - 1e-6), chi[k] > cut * (1 + 1e-6)
        assert np.all(below | above | (cut == 0.0))
        assert np.array_equal(with_[k]["tau"][below], host[k]["tau"][below]), k
        assert np.array_equal(with_[k]["tau"][~below], without[k]["tau"][~below]), k
        assert (without[k]["tau"] < host[k]["tau"]).mean() > 0.5
