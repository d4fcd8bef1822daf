"""A batched step that fails after its evolution (an event of another context, which the runtime refuses to
record on the stream) leaves nothing behind for the next one."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def foreign_event():
    """A CUDA event of a second context on the same GPU."""
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    ctx, event, popped, dev = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_int()
    assert cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
    assert cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, dev) == 0  # (becomes the current one)
    try:
        made = cu.cuEventCreate(ctypes.byref(event), 0)
    finally:
        assert cu.cuCtxPopCurrent_v2(ctypes.byref(popped)) == 0
    assert made == 0
    yield event.value
    assert cu.cuCtxDestroy_v2(ctx) == 0


@pytest.mark.parametrize("sampler", ["table", "learned"])
@pytest.mark.parametrize("prec_name", ["f32", "f64"])
def test_step_after_a_failed_one(foreign_event, prec_name, sampler):
    from paper_2110_00256_gb300 import api, workloads
    prec = api.QED_F64 if prec_name == "f64" else api.QED_F32
    t = api.qed_tables_generate(api.table_params(qs_n_chi=32, qs_n_xi=64, bw_n_chi=32, bw_n_xi=64))
    mlp = api.Mlp(t, 0) if sampler == "learned" else None
    n = 2000
    patch = {}
    for i, k in enumerate(("electrons", "positrons", "photons")):
        host = workloads.paper_benchmark(n, 60 + i, i * 10 ** 9)
        host["tau"] = np.where(np.arange(n) % 10 == 0, -1.0, 1e3)
        patch[k] = api.SpeciesBuffers(4 * n, prec).set(host)
    patch["fire"] = [api.FireBuffers(4 * n) for _ in range(3)]
    b = api.Batch([patch], prec)
    stats = api.Stats()
    bad = api.make_opts(mlp=mlp)
    bad.evolve_end = foreign_event
    with pytest.raises(api.QedError, match="cudaEventRecord"):
        api.qed_substep_batched(t, b, 10.0, 1, 0, bad)
    api.qed_substep_batched(t, b, 10.0, 1, 1, api.make_opts(stats=stats, mlp=mlp))
    torch.cuda.synchronize()
    for f in patch["fire"]:
        assert f.n() == n // 10
        assert np.array_equal(np.sort(f.idx[:f.n()].cpu().numpy()), np.arange(0, n, 10))
    assert stats.as_dict()["qs_events"] == 2 * (n // 10) and stats.as_dict()["bw_events"] == n // 10
