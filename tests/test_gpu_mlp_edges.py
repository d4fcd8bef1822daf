"""The training kernel at the edges of its tiles (32 samples per tile, tiles dealt
to as many CTAs as there are SMs): the gradient and the loss of a batch are the
means over its samples, so that a batch equals the weighted sum of its parts
whatever their sizes.  Tolerance: the parts' sums are FP32 sums of n products in
another order, at most n 2^-24 and typically sqrt(n) 2^-24 of the terms' magnitudes,
which exceed the sum's norm at most tenfold here: 1e-4 of the norm covers n = 1e4."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 31, 32, 33, 152 * 32 - 1, 152 * 32, 152 * 32 + 1, 10_007])
@pytest.mark.parametrize("proc", [0, 1])
def test_batch_gradient_is_the_sum_of_its_parts(proc, n):
    from paper_2110_00256_gb300 import api
    t = api.qed_tables_generate(api.table_params(qs_n_chi=32, qs_n_xi=64, bw_n_chi=32, bw_n_xi=64))
    m = api.Mlp(t, seed=3 + proc)
    ax = t.params.bw if proc else t.params.qs
    r = np.random.default_rng(n)
    chi = torch.tensor(np.exp(r.uniform(np.log(ax.chi_min), np.log(ax.chi_max), n)), device="cuda")
    u = torch.tensor(r.uniform(1e-6, 1 - 1e-6, n), device="cuda")
    xi = api.qed_table_sample(t, proc, api.QED_F64, chi, u)

    def grad(a, b):
        g, loss = m.gradients(proc, chi[a:b].clone(), u[a:b].clone(), xi[a:b].clone())
        return g.double().cpu().numpy(), float(loss.item())

    whole, loss = grad(0, n)
    cuts = sorted({0, n, *(c for c in (1, 32, 63, 64, 1100, 1101) if c < n)})
    parts = [((b - a) / n, *grad(a, b)) for a, b in zip(cuts, cuts[1:])]
    want = sum(f * g for f, g, _ in parts)
    assert np.linalg.norm(whole - want) <= 1e-4 * np.linalg.norm(want)
    assert loss == pytest.approx(sum(f * v for f, _, v in parts), rel=1e-4)
