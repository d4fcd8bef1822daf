"""The FP64 inverse CDFs on integers and their general forms (qed_table_sample)
against the same interpolation in extended precision on the host, over what
decides between the two: the smallest and odd table sizes, flat stretches, rows
that do not start at 0 or that leave the integers' range, chi outside the table
and outside the range of the integer logarithm, and draws around 2^-20, 2^-9, 1/2
and both ends.

Tolerance: a row value may be off by three roundings (2^-53 of the largest magnitude
in use) and by the error of the interpolation weight (the logarithm's and the
coordinate's roundings, 4 2^-53 (|ln chi| + |ln chi_min|) per interval) times the
rows' difference; that over the column difference is the error in columns, as is
the quotient's share of the column difference's own error.  The result itself: four
roundings (photon emission: of ln xi, then relative to xi)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
L = np.longdouble
EPS = L(2) ** -53
XI_MIN = 1e-8


def _rows(rng, n_chi, n_xi, form):
    """non-decreasing rows from 0 to 1"""
    steps = rng.uniform(0.2, 1.0, (n_chi, n_xi - 1))
    if form == "flat":
        steps[rng.uniform(size=steps.shape) < 0.3] = 0.0
        steps[:, 0] += 0.1
    p = np.concatenate([np.zeros((n_chi, 1)), np.cumsum(steps, axis=1)], axis=1)
    return np.minimum(p / p[:, -1:], 1.0)


@pytest.mark.parametrize("form", ["plain", "flat", "offset", "outside"])
@pytest.mark.parametrize("n_chi,n_xi", [(2, 2), (3, 17), (33, 257), (1024, 61)])
@pytest.mark.parametrize("proc", [0, 1])
def test_fp64_sampling_over_its_forms(proc, n_chi, n_xi, form):
    from paper_2110_00256_gb300 import api
    rng = np.random.default_rng(n_chi * 1000 + n_xi + proc)
    lo, hi = 0.02, 700.0
    par = api.table_params(qs_n_chi=n_chi, qs_n_xi=n_xi, qs_chi_min=lo, qs_chi_max=hi, qs_xi_min=XI_MIN,
                           bw_n_chi=n_chi, bw_n_xi=n_xi, bw_chi_min=lo, bw_chi_max=hi)
    rows = _rows(rng, n_chi, n_xi, form)
    first = {"offset": (-2.0, 0.01), "outside": (-40.0, -0.01)}.get(form, (-9.0, 0.0))
    qs = first[0] * (1.0 - rows)
    bw = np.minimum(first[1] + (0.5 - first[1]) * rows, 0.5)
    one = np.linspace(-9, -1, n_chi)
    t = api.qed_tables_create(par, one, qs, one, bw)
    tab = bw if proc else qs
    near = 1 + np.array([-1e-3, -1e-15, 1e-15, 1e-3])
    edge = np.concatenate([2.0 ** -np.arange(1, 54), 2.0 ** -9 * near, 2.0 ** -20 * near])
    u = np.concatenate([rng.uniform(0, 1, 4000), rng.uniform(0, 2.0 ** -8, 1000), edge, 1 - edge, [1.0]])
    u = np.minimum(np.floor(u * 2.0 ** 54 + 1) * 2.0 ** -54, 1.0)
    chi = np.exp(rng.uniform(np.log(lo), np.log(hi), u.size))
    chi[::13] = rng.choice([lo, hi, lo / 2, 2 * hi, 1e-30, 1e30, 1.0], chi[::13].size)
    got = api.qed_table_sample(t, proc, api.QED_F64, torch.tensor(chi, device="cuda"),
                               torch.tensor(u, device="cuda")).cpu().numpy()

    if proc:
        x, dx = np.where(u <= 0.5, u, 1.0 - u).astype(L), L(0.5) / (n_xi - 1)
    else:
        x, dx = np.log(u.astype(L)), -np.log(L(XI_MIN)) / (n_xi - 1)
    l0, l1 = np.log(L(lo)), np.log(L(hi))
    lc = np.log(chi.astype(L))
    pos = np.clip((lc - l0) * (n_chi - 1) / (l1 - l0), 0, n_chi - 1)
    k = np.minimum(pos.astype(int), n_chi - 2)
    a, b = tab[k].astype(L), tab[k + 1].astype(L)
    row = a + (pos - k)[:, None] * (b - a)
    m = np.clip((row <= x[:, None]).sum(axis=1) - 1, 0, n_xi - 2)
    i = np.arange(u.size)
    dp = row[i, m + 1] - row[i, m]
    f = np.where(dp > 0, (x - row[i, m]) / np.where(dp > 0, dp, 1), 0)
    v = (m + f) * dx
    err_w = 4 * EPS * (np.abs(lc) + abs(l0)) * (n_chi - 1) / (l1 - l0)
    err_p = 3 * EPS * max(1, abs(first[0])) + err_w * np.maximum(np.abs(b - a)[i, m], np.abs(b - a)[i, m + 1])
    if proc == 0:
        err_p = err_p + EPS * np.abs(x)
    tol = err_p * (1 + np.abs(f)) / np.maximum(dp, L(1e-300)) * dx
    if proc:
        v = np.clip(v, 0, 0.5)
        ref, tol = np.where(u <= 0.5, v, 1 - v), tol + 4 * EPS
    else:
        v = np.minimum(np.log(L(XI_MIN)) + v, 0)
        ref, tol = np.exp(v), np.exp(v) * (tol + 4 * EPS * (1 + np.abs(v) + abs(np.log(L(XI_MIN))))) + L(1e-300)
    # (a draw within rounding of a node next to a flat stretch may take either side of the jump)
    clear = np.abs(row - x[:, None]).min(axis=1) > EPS * max(4, abs(first[0])) + err_w * np.abs(b - a).max(axis=1)
    if form == "plain":
        clear[:] = True
    assert clear.mean() > 0.9
    bad = clear & ~(np.abs(got - ref) <= tol)
    assert not bad.any(), (chi[bad][:3], u[bad][:3], got[bad][:3], ref[bad][:3].astype(float))
