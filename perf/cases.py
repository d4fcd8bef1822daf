"""The library's work in a user's program, as cases that can be timed and compared.

A case is a dict of plain values; `kind` says which part of the library it runs:

* step      -- qed_substep on one electron, one positron and one photon species with the benchmark distribution
               (uniform momenta and fields), the call a particle-in-cell code makes for one region every timestep;
               `steps` calls in a row.
* beam      -- one qed_substep on a small electron beam in a static field (64-point tables, a short time step):
               the smallest call, where launches and latency count.
* block     -- a CUDA graph of qed_substep_batched steps on one patch whose chi spreads over five decades (Gaussian
               fields): how a program runs many steps of a mid-sized region.
* patches   -- a CUDA graph of qed_substep_batched steps over 64 patches of very uneven size.
* cascade   -- a CUDA graph of qed_push_substep_batched steps: an electron beam meets a strong plane wave, with the
               photons that it has already emitted.
* emission  -- qed_generate_photons with every lepton firing (a burst in a strong field; the paper times this call).
* pairs     -- qed_generate_pairs with every photon firing.
* sampler   -- inference of the learned sampler on a batch of (chi, U).
* gradients -- loss and gradients of the learned sampler on one minibatch: forward and backward.
* tables    -- generation of the four lookup tables and their copy to the host (once per program and table size).

Every step case ends with the appended products in the order of their ids, since the order in which the kernels append
them is not fixed; the outputs are then the particle arrays themselves.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2110_00256_gb300 import api

ALPHA = 7.2973525693e-3
GEV = 1.0e3 / 0.51099895000  # 1 GeV/c in m_e c
OMEGA = 3.0328877982211224e-6  # 0.8 um
M32 = 0xFFFFFFFF
MAX64 = 2 ** 63 - 1
SEED = 20211001  # of the library's own random numbers

# rows of a species' data: what a step changes first (positions where they are tracked), then the fields
FIELDS = ("ex", "ey", "ez", "bx", "by", "bz")
ROWS = ("px", "py", "pz", "tau", "tau_c", "weight", "x", "y", "z") + FIELDS


def listed():
    return [
        # the headline: 1e8 particles of one region in FP32, and the FP64 path at an ordinary size
        {"name": "step f32 1e8", "kind": "step", "prec": "f32", "n": 50_000_000, "steps": 8},
        {"name": "step f64 1e7", "kind": "step", "prec": "f64", "n": 5_000_011, "steps": 4},
        # the smallest call: 10^4 electrons, photon emission only
        {"name": "beam f64 1e4", "kind": "beam", "prec": "f64", "n": 10_000},
        # a mid-sized region over many steps, both precisions
        {"name": "block f32 2e6", "kind": "block", "prec": "f32", "n": 1_000_000, "steps": 50},
        {"name": "block f64 2e6", "kind": "block", "prec": "f64", "n": 1_000_003, "steps": 12},
        # a domain of 64 patches, 10^3 to 10^7 particles each
        {"name": "patches f32 6e7", "kind": "patches", "prec": "f32", "scale": 1.0, "steps": 8},
        # the cascade in a plane wave, photons in the majority
        {"name": "cascade f32 2e7", "kind": "cascade", "prec": "f32", "scale": 0.03, "photons": 10, "steps": 20},
        # bursts: every particle fires
        {"name": "emission f32 4e6", "kind": "emission", "prec": "f32", "n": 3_999_971},
        {"name": "pairs f64 2e6", "kind": "pairs", "prec": "f64", "n": 1_999_993},
        # the learned sampler: inference on a large batch, one training minibatch
        {"name": "sampler 1e7", "kind": "sampler", "proc": 0, "n": 10_000_000},
        {"name": "gradients 4096", "kind": "gradients", "proc": 1, "n": 4096},
        # the paper's table size
        {"name": "tables 256", "kind": "tables", "n_chi": 256, "n_xi": 256},
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "beam", "block", "patches", "cascade", "emission", "pairs", "sampler", "gradients",
                       "tables"])
    prec = rng.choice(["f32", "f64"])
    if kind == "step":
        return {"kind": kind, "prec": prec, "n": spread(3e4, 2e7 if prec == "f32" else 4e6), "steps": rng.randint(2, 6)}
    if kind == "beam":
        return {"kind": kind, "prec": prec, "n": spread(1e3, 2e5)}
    if kind == "block":
        return {"kind": kind, "prec": prec, "n": spread(3e4, 1e6), "steps": rng.randint(5, 12)}
    if kind == "patches":
        return {"kind": kind, "prec": "f32", "scale": math.exp(rng.uniform(math.log(0.01), 0.0)),
                "steps": rng.randint(2, 8)}
    if kind == "cascade":
        return {"kind": kind, "prec": prec, "scale": math.exp(rng.uniform(math.log(0.001), math.log(0.01))),
                "photons": rng.randint(0, 12), "steps": rng.randint(5, 12)}
    if kind in ("emission", "pairs"):
        return {"kind": kind, "prec": prec, "n": spread(1e3, 2e6)}
    if kind == "sampler":
        return {"kind": kind, "proc": rng.randint(0, 1), "n": spread(1e3, 1e7)}
    if kind == "gradients":
        return {"kind": kind, "proc": rng.randint(0, 1), "n": spread(100, 4e4)}
    return {"kind": kind, "n_chi": rng.randint(32, 200), "n_xi": rng.randint(32, 200)}


def work(case):
    k = case["kind"]
    f32 = case.get("prec") == "f32"
    n, steps = case.get("n", 0), case.get("steps", 1)
    if k in ("step", "block", "beam", "patches"):
        # p, E, B and the optical depth (FP32: a pair of floats) read, the optical depth written
        if k == "patches":
            n = int(patch_sizes(case["scale"]).sum()) * 0.5
        parts = steps * n * (1 if k == "beam" else 2)
        return {"bytes": parts * (52 if f32 else 88), "flops": parts * 90}
    if k == "cascade":
        # position, momentum and optical depth read and written (a photon's momentum is not written)
        n = int(patch_sizes(case["scale"]).sum())
        word = 4 if f32 else 8
        rows = (16 + 13 * case["photons"]) if f32 else (14 + 11 * case["photons"])
        return {"bytes": steps * n * rows * word, "flops": steps * n * (1 + case["photons"]) * 120}
    if k == "emission":
        return {"bytes": n * (164 if f32 else 296), "flops": n * 120}
    if k == "pairs":
        return {"bytes": n * (224 if f32 else 384), "flops": n * 160}
    if k == "sampler":
        return {"bytes": n * 24, "flops": n * 2 * (2 * 64 + 64 * 64 + 64)}
    if k == "gradients":
        return {"bytes": n * 24 + 2 * 4 * api.Mlp.NPARAM, "flops": n * 6 * (2 * 64 + 64 * 64 + 64)}
    entries = case["n_chi"] * case["n_xi"] * 2
    return {"bytes": entries * 8, "flops": entries * 8 * 30 * 8}


# ------------------------------------------------------------------------------------------------------------------
# tables (what a program loads or is given): quadrature of the spectra in 64 bits
# ------------------------------------------------------------------------------------------------------------------
def bessel_scaled(x, nu_a, nu_b):
    """e^x int_x^inf K_a and e^x K_b by the trapezoid rule in K_nu(x) = int_0^inf exp(-x cosh t) cosh(nu t) dt."""
    h = torch.clamp(0.6 / torch.sqrt(x), max=0.25)
    sa, sb = torch.full_like(x, 0.5), torch.full_like(x, 0.5)
    for k in range(1, 800):
        t = k * h
        arg = 2.0 * x * torch.sinh(0.5 * t) ** 2
        if k % 32 == 0 and bool(((arg - max(nu_a, nu_b) * t > 45.0) & (arg > 45.0)).all()):
            break
        sa += torch.exp(nu_a * t - arg) * (1.0 + torch.exp(-2.0 * nu_a * t)) / (torch.exp(t) * (1.0 + torch.exp(-2.0 * t)))
        sb += torch.exp(nu_b * t - arg) * 0.5 * (1.0 + torch.exp(-2.0 * nu_b * t))
    return h * sa, h * sb


def qs_number(chi, xi, om):
    """S(chi, xi) of the photon spectrum (number density in ln xi), om = 1 - xi."""
    y = (2.0 / 3.0) * xi / (chi * om)
    ia, kb = bessel_scaled(torch.clamp(y, max=745.0), 5.0 / 3.0, 2.0 / 3.0)
    s = math.sqrt(3.0) / (2.0 * math.pi) * xi * torch.exp(-y) * (ia + xi * xi / om * kb)
    return torch.where(y > 745.0, torch.zeros_like(s), s)


def bw_bracket(chi, xi):
    """The pair spectrum's bracket in xi = chi_- / chi_gamma."""
    om = 1.0 - xi
    z = 2.0 / (3.0 * chi * xi * om)
    ia, kb = bessel_scaled(torch.clamp(z, max=745.0), 1.0 / 3.0, 2.0 / 3.0)
    s = torch.exp(-z) * (ia + (xi / om + om / xi) * kb)
    return torch.where(z > 745.0, torch.zeros_like(s), s)


def panels(lo, hi, count):
    """Nodes and weights of Gauss-Legendre (14 points) on `count` equal panels of [lo, hi] (tensors): (..., count*14)."""
    gx, gw = (torch.tensor(v, dtype=torch.float64, device=lo.device) for v in np.polynomial.legendre.leggauss(14))
    half = ((hi - lo) / (2 * count))[..., None, None]
    mid = lo[..., None, None] + half * (2 * torch.arange(count, device=lo.device, dtype=torch.float64)[:, None] + 1)
    return (mid + half * gx).flatten(-2), (half * gw).expand(mid.shape[:-1] + (14,)).flatten(-2)


@functools.lru_cache(maxsize=4)
def table_arrays(n_chi, n_xi, chi_qs=(1e-3, 1e3), chi_bw=(2e-2, 1e3), xi_min=1e-12):
    """ln G, ln P (photon emission), ln T, P (pair production) as numpy arrays in the layout of qed_tables_create."""
    dev = "cuda"
    grid = lambda a, b, n: torch.linspace(math.log(a), math.log(b), n, dtype=torch.float64, device=dev).exp()  # noqa: E731
    # photon emission: intervals of ln xi; below xi_min in w = xi^(1/3), the last one in v = ln(xi / (1 - xi))
    chi = grid(*chi_qs, n_chi)[:, None, None]
    u = torch.linspace(math.log(xi_min), 0.0, n_xi, dtype=torch.float64, device=dev)
    x, w = panels(u[:-2], u[1:-1], 1)
    mid = (qs_number(chi, x.exp()[None], -torch.expm1(x)[None]) * w).sum(-1)
    one = torch.ones(1, dtype=torch.float64, device=dev)
    x, w = panels(0 * one, one * xi_min ** (1 / 3), 2)
    low = (3.0 * qs_number(chi, (x ** 3)[None], 1.0 - (x ** 3)[None]) / x * w).sum(-1)
    v0 = u[-2] - torch.log(-torch.expm1(u[-2]))
    x, w = panels(v0 * one, math.log(1200.0 * chi_qs[1]) * one, 64)
    top = (qs_number(chi, torch.sigmoid(x)[None], torch.sigmoid(-x)[None]) * torch.sigmoid(-x) * w).sum(-1)
    part = torch.cat([low, mid, top], 1)
    total = part.sum(1, keepdim=True)
    tail = (part.flip(1).cumsum(1).flip(1) - part) / total
    ln_p = torch.where(tail < 0.5, torch.log1p(-tail), torch.log(part.cumsum(1) / total))
    ln_p[:, -1] = 0.0
    ln_g = total[:, 0].log()
    # pair production: intervals of xi on [0, 1/2], the first one in ln xi
    chi = grid(*chi_bw, n_chi)[:, None, None]
    xi = torch.linspace(0.0, 0.5, n_xi, dtype=torch.float64, device=dev)
    x, w = panels(xi[1:-1], xi[2:], 2)
    mid = (bw_bracket(chi, x[None]) * w).sum(-1)
    lo = torch.log(2.0 / (3.0 * 746.0 * chi[:, 0]))
    x, w = panels(torch.minimum(lo, xi[1].log() - 1e-3), xi[1].log().expand_as(lo), 32)
    first = (bw_bracket(chi, x.exp()) * x.exp() * w).sum(-1)
    part = torch.cat([torch.zeros_like(first), first, mid], 1)
    half = part.sum(1, keepdim=True)
    ln_t = torch.log(2.0 * half[:, 0] / (math.pi * math.sqrt(3.0) * chi[:, 0, 0]))
    p = part.cumsum(1) / (2.0 * half)
    p[:, -1] = 0.5
    return tuple(a.cpu().numpy() for a in (ln_g, ln_p, ln_t, p))


def make_tables(n=256):
    return api.qed_tables_create(api.table_params(qs_n_chi=n, qs_n_xi=n, bw_n_chi=n, bw_n_xi=n), *table_arrays(n, n))


# ------------------------------------------------------------------------------------------------------------------
# particles: one species of every patch in one (rows, particles) array
# ------------------------------------------------------------------------------------------------------------------
class Pool:
    def __init__(self, sizes, room, prec, positions=False):
        self.prec = api.QED_F32 if prec == "f32" else api.QED_F64
        self.sizes = np.asarray(sizes, dtype=np.int64)
        caps = self.sizes + np.asarray(room, dtype=np.int64)
        off = np.concatenate([[0], np.cumsum((caps + 63) // 64 * 64)])
        self.moving = 9 if positions else 6
        self.names = ROWS[:self.moving] + FIELDS
        dt = torch.float32 if prec == "f32" else torch.float64
        self.data = torch.zeros(len(self.names), int(off[-1]), dtype=dt, device="cuda")
        self.ids = torch.zeros(int(off[-1]), dtype=torch.int64, device="cuda")
        self.start = torch.tensor(self.sizes, device="cuda")
        self.counts = self.start.clone()
        self.first = None
        self.species = []
        for i, cap in enumerate(caps):
            s = api.SpeciesBuffers(1, self.prec, positions=positions)
            s.capacity = int(cap)
            a, b = int(off[i]), int(off[i] + cap)
            s.arrays = {k: self.data[r, a:b] for r, k in enumerate(self.names)}
            s.arrays["id"] = self.ids[a:b]
            s.count = self.counts[i:i + 1]
            self.species.append(s)
        # where the particles at the start are, and the slots of the products
        spans = lambda lo, hi: torch.from_numpy(np.concatenate([np.arange(a, b) for a, b in zip(lo, hi)] or [[]])  # noqa: E731
                                                .astype(np.int64)).cuda()
        self.primary = slice(0, int(self.sizes[0])) if len(caps) == 1 else spans(off[:-1], off[:-1] + self.sizes)
        self.slots = spans(off[:-1] + self.sizes, off[:-1] + caps)
        self.patch = torch.repeat_interleave(torch.arange(len(caps), device="cuda"),
                                             torch.tensor(caps - self.sizes, device="cuda"))
        self.local = self.slots - torch.tensor(off[:-1], device="cuda")[self.patch]

    def put(self, rows):
        """Values of the particles at the start, a dict of tensors by row name (and "id")."""
        for k, v in rows.items():
            if k == "id":
                self.ids[self.primary] = v
            else:
                self.data[self.names.index(k), self.primary] = v.to(self.data.dtype)

    def keep(self):
        """Remember the start, for reset()."""
        self.first = self.data[:self.moving].clone()

    def reset(self):
        """The products have left the region; the others are back at the start if it was kept."""
        if self.first is not None:
            self.data[:self.moving].copy_(self.first)
        self.counts.copy_(self.start)

    def settle(self):
        """The products in the order of their ids, patch by patch; free slots zero."""
        if not self.slots.numel():
            return
        live = self.local < self.counts[self.patch]
        order = torch.argsort(torch.where(live, self.ids[self.slots], MAX64))
        if len(self.species) > 1:
            order = order[torch.argsort(self.patch[order], stable=True)]
        src = self.slots[order]
        self.data.index_copy_(1, self.slots, torch.where(live, self.data.index_select(1, src), 0))
        self.ids[self.slots] = torch.where(live, self.ids[src], 0)

    def out(self):
        d = {"p": self.data[:3], "tau": self.data[3], "w": self.data[5], "x": self.data[6:self.moving],
             "fields": self.data[self.moving:], "id": self.ids, "count": self.counts}
        if self.prec == api.QED_F32:
            d["tau_c"] = self.data[4]
        return d


def generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def uniform(g, n, lo=0.0, hi=1.0):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64).mul_(hi - lo).add_(lo)


def exponential(g, n):
    return torch.empty(n, device="cuda", dtype=torch.float64).exponential_(1.0, generator=g)


def benchmark_rows(g, n, first_id, fields=0.01):
    """Momenta uniform in +-1 GeV/c, fields uniform in +-`fields` of the critical field."""
    d = {k: uniform(g, n, -GEV, GEV) for k in ("px", "py", "pz")}
    d |= {k: uniform(g, n, -fields, fields) for k in ("ex", "ey", "ez", "bx", "by", "bz")}
    d |= {"tau": exponential(g, n), "weight": torch.ones(n, device="cuda"),
          "id": torch.arange(first_id, first_id + n, device="cuda")}
    return d


def patch_sizes(scale):
    r = np.random.Generator(np.random.PCG64(7))
    n = np.round(10.0 ** (3.0 + 4.0 * r.uniform(0.0, 1.0, 64)))
    return np.maximum((n * scale).astype(np.int64), 2)


def pools(case, seed):
    """The electrons, positrons and photons of a case, in its precision."""
    g, k, prec = generator(seed), case["kind"], case["prec"]
    n, steps = case.get("n", 0), case.get("steps", 1)
    if k == "beam":
        e, p, ph = Pool([n], [256], prec), Pool([0], [256], prec), Pool([0], [4096], prec)
        gam = 10.0 ** uniform(g, n, 2.0, 4.0)
        cth, phi, pm = uniform(g, n, -1.0, 1.0), uniform(g, n, 0.0, 2.0 * math.pi), torch.sqrt(gam * gam - 1.0)
        sth = torch.sqrt(1.0 - cth * cth)
        e.put({"px": pm * sth * torch.cos(phi), "py": pm * sth * torch.sin(phi), "pz": pm * cth,
               "bz": torch.full_like(gam, 0.01), "tau": exponential(g, n), "weight": torch.ones_like(gam),
               "id": torch.arange(n, device="cuda")})
        return e, p, ph
    if k == "step":
        room = lambda rate: [256 + int(n * steps * rate)]  # noqa: E731
        e, p, ph = Pool([n], room(1.2e-4), prec), Pool([0], room(1.2e-4), prec), Pool([n], room(5e-4), prec)
        e.put(benchmark_rows(g, n, 0))
        ph.put(benchmark_rows(g, n, 10 ** 12))
        return e, p, ph
    if k == "block":
        room = lambda rate: [256 + int(n * steps * rate)]  # noqa: E731
        e, p, ph = Pool([n], room(5e-5), prec), Pool([0], room(5e-5), prec), Pool([n], room(2.5e-4), prec)
        for pool, offset, lepton in ((e, 0, True), (ph, 10 ** 12, False)):
            d = benchmark_rows(g, n, offset)
            d |= {c: torch.randn(n, generator=g, device="cuda", dtype=torch.float64) for c in FIELDS}
            scale = 10.0 ** uniform(g, n, -3.0, 2.0) / chi_of(d, lepton)[0]
            pool.put(d | {c: d[c] * scale for c in FIELDS})
        return e, p, ph
    sizes = patch_sizes(case["scale"])
    if k == "patches":
        ne = sizes // 2
        room = lambda m, rate: 64 + (m * steps * rate).astype(np.int64)  # noqa: E731
        e, ph = Pool(ne, room(ne, 1.2e-4), prec), Pool(sizes - ne, room(ne, 5e-4), prec)
        p = Pool(0 * ne, room(ne, 1.2e-4), prec)
        e.put(benchmark_rows(g, int(ne.sum()), 0))
        ph.put(benchmark_rows(g, int((sizes - ne).sum()), 10 ** 12))
        return e, p, ph
    # cascade: electrons against the wave, the photons that they emitted ahead of them
    few, m = 64 + sizes // 500, case["photons"] * sizes
    e, p = Pool(sizes, few, prec, True), Pool(0 * sizes, few, prec, True)
    ph = Pool(m, 64 + (sizes * steps * 0.035).astype(np.int64), prec, True)
    for pool, count, offset in ((e, int(sizes.sum()), 0), (ph, int(m.sum()), 10 ** 12)):
        if pool is e:
            gam = 2000.0 * uniform(g, count, 0.95, 1.05)
            d = {"px": torch.sqrt(gam * gam - 1.0)}
        else:
            gam = torch.exp(uniform(g, count, math.log(2.0), math.log(1500.0)))
            angle = torch.randn(count, generator=g, device="cuda", dtype=torch.float64) * 0.03
            d = {"px": gam * torch.cos(angle), "py": gam * torch.sin(angle)}
        wave = 2.0 * math.pi / OMEGA
        d |= {c: uniform(g, count, 0.0, wave) for c in ("x", "y", "z")}
        d |= {"tau": exponential(g, count), "weight": torch.ones_like(gam),
              "id": torch.arange(offset, offset + count, device="cuda")}
        pool.put(d)
    return e, p, ph


DT_CASCADE = 2.0 * math.pi / OMEGA / 200


def step_of(case):
    """Time step and photon threshold."""
    if case["kind"] == "beam":
        return 1e-3, 0.0
    return (DT_CASCADE, 2.0) if case["kind"] == "cascade" else (10.0, 0.0)


def prepare(case, seed):
    k = case["kind"]
    if k == "tables":
        # a program asks for its own range of chi
        top = 1e3 * (1.0 + (seed % 1000) / 2000.0)
        return {"params": api.table_params(qs_chi_max=top, qs_n_chi=case["n_chi"], qs_n_xi=case["n_xi"],
                                           bw_chi_max=top, bw_n_chi=case["n_chi"], bw_n_xi=case["n_xi"])}
    s = {"case": case, "tables": make_tables(64 if k == "beam" else 256)}
    if k in ("sampler", "gradients"):
        d = network_inputs(case, seed)
        s["mlp"] = api.Mlp(s["tables"], 0)
        s["mlp"].set_params(case["proc"], d["theta"])
        s |= {c: d[c] for c in ("chi", "u", "xi")}
        return s
    if k in ("emission", "pairs"):
        s |= burst(case, seed)
        return s
    e, p, ph = s["pools"] = pools(case, seed)
    dt, threshold = step_of(case)
    s["stats"] = api.Stats()
    s["out"] = {"e": e.out(), "p": p.out(), "ph": ph.out(), "stats": s["stats"].t}
    fire = lambda a, i: api.FireBuffers(a.species[i].capacity)  # noqa: E731
    if k in ("step", "beam"):
        s["call"] = api.SubstepCall(s["tables"], e.species[0], p.species[0], ph.species[0],
                                    [fire(a, 0) for a in (e, p, ph)], dt, SEED, threshold, s["stats"])
        s["step"] = 0
        return s
    # the steps of a pass in one CUDA graph, from the start's particles
    s["batch"] = api.Batch([{"electrons": e.species[i], "positrons": p.species[i], "photons": ph.species[i],
                             "fire": [fire(e, i), fire(p, i), fire(ph, i)]} for i in range(len(e.species))], e.prec)
    s["d_step"] = torch.zeros(1, dtype=torch.int64, device="cuda")
    opts = api.make_opts(photon_threshold=threshold, stats=s["stats"], d_step=s["d_step"])
    if k == "cascade":
        wave = api.plane_wave(100.0 * OMEGA, OMEGA)
        one = lambda dt, o, st: api.qed_push_substep_batched(s["tables"], s["batch"], wave, 0.0, dt, SEED, 0, o,  # noqa: E731
                                                             stream=st)
    else:
        one = lambda dt, o, st: api.qed_substep_batched(s["tables"], s["batch"], dt, SEED, 0, o, stream=st)  # noqa: E731
    if k != "patches":
        for a in (e, p, ph):
            a.keep()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    s["graph"] = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        one(0.0, api.make_opts(), stream)  # first calls outside the capture
        with torch.cuda.graph(s["graph"], stream=stream):
            for a in (e, p, ph):
                a.reset()
            if e.first is not None:
                s["d_step"].zero_()
            for _ in range(case["steps"]):
                one(dt, opts, stream)
            for a in (e, p, ph):
                a.settle()
    torch.cuda.current_stream().wait_stream(stream)
    return s


def run(state):
    if "params" in state:
        return api.qed_tables_copy_to_host(api.qed_tables_generate(state["params"]))
    case, k = state["case"], state["case"]["kind"]
    if k == "sampler":
        return state["mlp"].sample(case["proc"], state["chi"], state["u"])
    if k == "gradients":
        return state["mlp"].gradients(case["proc"], state["chi"], state["u"], state["xi"])
    if k in ("emission", "pairs"):
        return run_burst(state)
    e, p, ph = state["pools"]
    if k == "beam":
        state["call"](state["step"])
        state["step"] += 1
    elif k == "step":
        for a in (e, p, ph):
            a.reset()
        for _ in range(case["steps"]):
            state["call"](state["step"])
            state["step"] += 1
        for a in (e, p, ph):
            a.settle()
    else:
        state["graph"].replay()
    return state["out"]


# ------------------------------------------------------------------------------------------------------------------
# bursts: every particle of a firing list
# ------------------------------------------------------------------------------------------------------------------
def burst(case, seed):
    n, prec, photons = case["n"], case["prec"], case["kind"] == "pairs"
    g = generator(seed)
    parent = Pool([n], [0], prec, True)
    out = [Pool([0], [n], prec, True) for _ in range(2 if photons else 1)]
    d = benchmark_rows(g, n, 0)
    number = torch.arange(n, device="cuda")
    d |= {"x": number, "y": uniform(g, n), "z": uniform(g, n)}  # x: the parent's number, which its products inherit
    parent.put(d | {"tau": -d["tau"]})
    fire = api.FireBuffers(n)
    # warps append their particles in the order in which they happen to come
    run64 = torch.argsort(torch.arange(-(-n // 64), device="cuda") + uniform(g, -(-n // 64), 0.0, 4096.0))
    index = (run64[:, None] * 64 + torch.arange(64, device="cuda")).flatten()
    fire.idx.copy_(index[index < n])
    exact = {c: parent.data[r].double() for r, c in enumerate(parent.names)}
    fire.chi.copy_(chi_of(exact, not photons)[0][fire.idx].to(parent.data.dtype))
    fire.count.fill_(n)
    parent.keep()
    # the products in the order of their parents (one place more for those that are not there)
    rows = [torch.zeros(len(o.names), n + 1, dtype=o.data.dtype, device="cuda") for o in out]
    return {"parent": parent, "out": out, "fire": fire, "rows": rows, "number": number}


def run_burst(state):
    parent, out, fire = state["parent"], state["out"], state["fire"]
    parent.data[:6].copy_(parent.first[:6])  # (the last pass's events have not happened)
    for o in out:
        o.counts.copy_(o.start)
    if len(out) == 1:
        api.qed_generate_photons(state["tables"], parent.species[0], out[0].species[0], fire, SEED, 3)
    else:
        api.qed_generate_pairs(state["tables"], parent.species[0], out[0].species[0], out[1].species[0], fire, SEED, 3)
    res = {"parent": parent.out()}
    n = int(parent.sizes[0])
    for i, (o, rows) in enumerate(zip(out, state["rows"])):
        # (a photon below the pair threshold makes no products)
        at = torch.where(state["number"] < o.counts, o.data[6, :n].long(), n)
        rows.index_copy_(1, at, o.data[:, :n])
        ids = torch.zeros(n + 1, dtype=torch.int64, device="cuda").index_copy_(0, at, o.ids[:n])
        res["out%d" % i] = {"p": rows[:3, :n], "tau": rows[3, :n], "tau_c": rows[4, :n], "rest": rows[5:, :n],
                            "id": ids[:n], "count": o.counts}
    return res


# ------------------------------------------------------------------------------------------------------------------
# the learned sampler
# ------------------------------------------------------------------------------------------------------------------
def network_inputs(case, seed):
    """(chi, U) over the tables' range, xi by the inverse CDF of the same tables, and a network's parameters."""
    n, proc = case["n"], case["proc"]
    g = generator(seed)
    lo, hi = ((1e-3, 1e3), (2e-2, 1e3))[proc]
    chi, u = torch.exp(uniform(g, n, math.log(lo), math.log(hi))), uniform(g, n, 1e-9, 1.0 - 1e-9)
    r = np.random.default_rng(seed)
    parts = [r.uniform(-1.0, 1.0, 128) * 0.3, r.uniform(-0.1, 0.1, 64), r.uniform(-1.0, 1.0, 4096) * 0.22,
             r.uniform(-0.1, 0.1, 64), r.uniform(-1.0, 1.0, 64) * 0.3, r.uniform(-0.1, 0.1, 1)]
    d = {"chi": chi, "u": u, "theta": np.concatenate(parts).astype(np.float32), "lo": lo, "hi": hi}
    d["xi"] = None
    if case["kind"] == "gradients":
        xi, electron = sample_xi(Lookup(256), proc == 0, chi, u)
        d["xi"] = torch.clamp(torch.where(electron, xi, 1.0 - xi), 1e-12, 1.0 - 1e-12)
    return d


def network(d, proc, theta):
    """y(chi, U) of the network in 64 bits, with its bf16 weights and activations."""
    c = torch.clamp(d["chi"], d["lo"], d["hi"])
    x1 = 2.0 * torch.log(c / d["lo"]) / math.log(d["hi"] / d["lo"]) - 1.0
    v = d["u"] if proc == 0 else 2.0 * torch.minimum(d["u"], 1.0 - d["u"])
    w1, b1, w2, b2, w3, b3 = torch.split(theta, [128, 64, 4096, 64, 64, 1])
    gelu = functools.partial(torch.nn.functional.gelu, approximate="tanh")
    h = gelu(torch.stack([x1, 2.0 * v - 1.0], 1) @ w1.view(64, 2).T + b1)
    h = h + (h.to(torch.bfloat16).double() - h).detach()
    return gelu(h @ w2.view(64, 64).T + b2) @ w3 + b3, c


def exact_network(case, seed):
    d, proc = network_inputs(case, seed), case["proc"]
    theta = torch.tensor(d["theta"], device="cuda").to(torch.bfloat16).double()
    if case["kind"] == "sampler":
        out = torch.empty_like(d["chi"])
        for a in range(0, case["n"], 1 << 20):
            e = {k: v[a:a + (1 << 20)] if k in ("chi", "u") else v for k, v in d.items()}
            y, c = network(e, proc, theta)
            if proc == 0:
                out[a:a + (1 << 20)] = torch.sigmoid(y + 3.0 * torch.log(e["u"]) + torch.log(c / (1.0 + c)))
            else:
                xs = torch.clamp(torch.sigmoid(-2.0 * torch.sqrt(c / (c + 16.0 / 3.0)) * y), max=0.5)
                out[a:a + (1 << 20)] = torch.where(e["u"] <= 0.5, xs, 1.0 - xs)
        return out
    theta.requires_grad_(True)
    y, c = network(d, proc, theta)
    if proc == 0:
        t = torch.log(d["xi"] / (1.0 - d["xi"])) - 3.0 * torch.log(d["u"]) - torch.log(c / (1.0 + c))
    else:
        xs = torch.clamp(torch.where(d["u"] <= 0.5, d["xi"], 1.0 - d["xi"]), max=0.5)
        t = torch.log((1.0 - xs) / xs) / (2.0 * torch.sqrt(c / (c + 16.0 / 3.0)))
    loss = ((y - t) ** 2).mean()
    loss.backward()
    return [theta.grad, loss.detach()[None]]


# ------------------------------------------------------------------------------------------------------------------
# the substep in 64 bits
# ------------------------------------------------------------------------------------------------------------------
def chi_of(d, lepton):
    """chi and the energy (gamma, or |p|): |E' + p x B|, E' = gamma E_perp, without the cancelling difference."""
    p, e, b = ([d[c] for c in names] for names in (("px", "py", "pz"), ("ex", "ey", "ez"), ("bx", "by", "bz")))
    p2 = p[0] * p[0] + p[1] * p[1] + p[2] * p[2]
    en = torch.sqrt(1.0 + p2) if lepton else torch.sqrt(p2)
    inv = torch.where(p2 > 0, 1.0 / torch.sqrt(p2), 0.0)
    ne = (p[0] * e[0] + p[1] * e[1] + p[2] * e[2]) * inv
    s = ne * ne if lepton else torch.zeros_like(ne)
    for i in range(3):
        j, k = (i + 1) % 3, (i + 2) % 3
        s = s + (en * (e[i] - ne * inv * p[i]) + (p[j] * b[k] - p[k] * b[j])) ** 2
    return torch.sqrt(s), en


class Lookup:
    def __init__(self, n):
        self.n = n
        self.a = [torch.from_numpy(v).cuda() for v in table_arrays(n, n)]
        self.lo = (math.log(1e-3), math.log(2e-2))
        self.hi = math.log(1e3)

    def place(self, proc, chi):
        t = (torch.log(chi) - self.lo[proc]) * ((self.n - 1) / (self.hi - self.lo[proc]))
        t = torch.clamp(t, 0.0, self.n - 1)
        i = torch.clamp(t.long(), max=self.n - 2)
        return i, t - i

    def rate(self, proc, chi, en):
        i, f = self.place(proc, chi)
        tab = self.a[2 * proc]
        ln = tab[i] + f * (tab[i + 1] - tab[i])
        if proc == 0:
            r = 2.0 / 3.0 * ALPHA * torch.exp(ln) / en
        else:
            ln = torch.where(chi < 2e-2, -1.4712438795175893 - (8.0 / 3.0) / chi, ln)
            ln = torch.where(chi > 1e3, -0.9686047877362934 - torch.log(chi) / 3.0, ln)
            r = ALPHA * chi * torch.exp(ln) / en
        return torch.where((chi > 0) & (en > 0), r, 0.0)


def sample_xi(tab, qs, chi, u):
    """Inverse CDF through the 2-D tables: xi and whether it is the electron's (photon emission: always)."""
    n, proc = tab.n, 0 if qs else 1
    i, w = tab.place(proc, chi)
    t = tab.a[2 * proc + 1]
    row = lambda m: t[i, m] + w * (t[i + 1, m] - t[i, m])  # noqa: E731
    dt = t[:, 1:] - t[:, :-1]
    electron = torch.ones_like(u, dtype=torch.bool) if qs else u <= 0.5
    r = torch.log(u) if qs else torch.where(electron, u, 1.0 - u)
    lo, hi = torch.zeros_like(i), torch.full_like(i, n)
    for _ in range(12):  # the last m with P_m <= r
        mid = (lo + hi) // 2
        up = (row(torch.clamp(mid, max=n - 1)) <= r) & (hi - lo > 1)
        lo, hi = torch.where(up, mid, lo), torch.where(up | (hi - lo <= 1), hi, mid)
    m = torch.clamp(lo, max=n - 2)
    p0, dp = row(m), dt[i, m] + w * (dt[i + 1, m] - dt[i, m])  # (differences first: neighbours are close)
    x0, dx = (math.log(1e-12), -math.log(1e-12) / (n - 1)) if qs else (0.0, 0.5 / (n - 1))
    x = x0 + dx * m.double() + torch.where(dp > 0, (r - p0) * dx / torch.where(dp > 0, dp, 1.0), 0.0)
    return (torch.exp(torch.clamp(x, max=0.0)) if qs else torch.clamp(x, 0.0, 0.5)), electron


def philox(ids, step, purpose):
    """Philox4x32-10 with the key SEED and the counter (id, step, purpose): four words."""
    c = [ids & M32, (ids >> 32) & M32, torch.full_like(ids, step), torch.full_like(ids, purpose)]
    k0, k1 = SEED & M32, SEED >> 32
    for _ in range(10):
        a, b = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [((b >> 32) & M32) ^ c[1] ^ k0, b & M32, ((a >> 32) & M32) ^ c[3] ^ k1, a & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def draw53(ids, step, purpose):
    w = philox(ids, step, purpose)
    return ((((w[1] << 32) | w[0]) >> 11) & (2 ** 53 - 1)).double().add_(0.5).mul_(2.0 ** -53)


def tau_draw(ids, step, purpose):
    return -torch.log(draw53(ids, step, purpose))


def child_ids(ids, step):
    w = philox(ids, step, 3)
    return (w[1] << 32) | w[0], (w[3] << 32) | w[2]


def emit(tab, d, i, chi, step, threshold):
    """Photon emission of the leptons `i` of `d`: the photons that are kept; the leptons recoil."""
    q = {k: v[i] for k, v in d.items()}
    xi, _ = sample_xi(tab, True, chi, draw53(q["id"], step, 0))
    p2 = q["px"] ** 2 + q["py"] ** 2 + q["pz"] ** 2
    gam, inv = torch.sqrt(1.0 + p2), 1.0 / torch.sqrt(p2)
    gg = p2 / (gam + 1.0) * xi  # (gamma - 1) xi
    left = p2 / (gam + 1.0) - gg
    pn = torch.sqrt(left * (left + 2.0))
    out = dict(q)
    out["id"] = child_ids(q["id"], step)[0]
    out["tau"] = tau_draw(out["id"], step, 2)
    for c in ("px", "py", "pz"):
        n = q[c] * inv
        out[c] = gg * n
        d[c][i] = pn * n
    d["tau"][i] = tau_draw(q["id"], step, 1)
    keep = gg >= threshold
    return {k: v[keep] for k, v in out.items()}


def decay(tab, d, i, chi, step):
    """Pair production of the photons `i` of `d`: the electrons and positrons; the photons are removed."""
    gg = torch.sqrt(d["px"][i] ** 2 + d["py"][i] ** 2 + d["pz"][i] ** 2)
    low = i[gg <= 2.0]
    d["tau"][low] = tau_draw(d["id"][low], step, 1)
    ok = gg > 2.0
    i, gg, chi = i[ok], gg[ok], chi[ok]
    q = {k: v[i] for k, v in d.items()}
    xs, electron = sample_xi(tab, False, chi, draw53(q["id"], step, 0))
    out = []
    for frac, ids in zip((torch.where(electron, xs, 1.0 - xs), torch.where(electron, 1.0 - xs, xs)),
                         child_ids(q["id"], step)):
        kin = (gg - 2.0) * frac
        pm = torch.sqrt(kin * (kin + 2.0))
        out.append(q | {c: pm / gg * q[c] for c in ("px", "py", "pz")} | {"id": ids, "tau": tau_draw(ids, step, 2)})
    d["tau"][i] = math.inf
    d["weight"][i] = 0.0
    return out


def exact_rows(pool):
    """The particles at the start in 64 bits, with the patch of each."""
    d = {k: pool.data[r, pool.primary].double() for r, k in enumerate(pool.names) if k != "tau_c"}
    d["id"] = pool.ids[pool.primary].clone()
    d["patch"] = torch.repeat_interleave(torch.arange(len(pool.sizes), device="cuda"), pool.start)
    return d


def exact_out(pool, d, n0):
    """The particles `d` (the first n0 from the start) laid out as the pool's outputs."""
    rows = torch.zeros(len(pool.names), pool.data.shape[1], dtype=torch.float64, device="cuda")
    order = torch.argsort(d["id"][n0:])
    order = order[torch.argsort(d["patch"][n0:][order], stable=True)]
    made = torch.bincount(d["patch"][n0:], minlength=len(pool.sizes))
    slots = pool.slots[(pool.local - pool.start[pool.patch]) < made[pool.patch]]
    for r, k in enumerate(pool.names):
        if k in d:
            rows[r, pool.primary] = d[k][:n0]
            rows[r, slots] = d[k][n0:][order][:slots.numel()]
    return {"p": rows[:3], "tau": rows[3], "w": rows[5], "x": rows[6:pool.moving], "fields": rows[pool.moving:]}


def push(q, d, t, dt):
    """The plane wave's fields at the particles, the Boris push (photons fly straight) and the move, in place."""
    wave = 100.0 * OMEGA * torch.cos(OMEGA * (t + d["x"]))
    for c in FIELDS:
        d[c].zero_()
    d["ey"].copy_(wave)
    d["bz"].copy_(-wave)
    p = [d[c] for c in ("px", "py", "pz")]
    norm = lambda v: v[0] * v[0] + v[1] * v[1] + v[2] * v[2]  # noqa: E731
    cross = lambda a, b: [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]  # noqa: E731
    h = 0.5 * q * dt
    if q:
        e, b = [d[c] for c in FIELDS[:3]], [d[c] for c in FIELDS[3:]]
        m = [a + h * f for a, f in zip(p, e)]
        g = torch.sqrt(1.0 + norm(m))
        t_ = [h * f / g for f in b]
        s_ = [2.0 * f / (1.0 + norm(t_)) for f in t_]
        w = [a + c for a, c in zip(m, cross(m, t_))]
        for i, c in enumerate(cross(w, s_)):
            p[i].copy_(m[i] + c + h * e[i])
    g = torch.sqrt(norm(p) + (1.0 if q else 0.0))
    for x, a in zip(("x", "y", "z"), p):
        d[x] += a / torch.where(g > 0, g, 1.0) * dt


def exact_steps(case, seed):
    ps = pools(case, seed)
    dt, threshold = step_of(case)
    tab = Lookup(64 if case["kind"] == "beam" else 256)
    species = [exact_rows(a) for a in ps]
    n0 = [d["px"].numel() for d in species]
    dt = float(np.float32(dt)) if case["prec"] == "f32" else dt
    for step in range(case.get("steps", 1)):
        fired = []
        for k, d in enumerate(species):
            hit, chis, n = [], [], d["px"].numel()
            for a in range(0, n, 1 << 24):
                part = {c: v[a:a + (1 << 24)] for c, v in d.items()}
                if case["kind"] == "cascade":
                    push((-1.0, 1.0, 0.0)[k], part, step * DT_CASCADE, dt)
                chi, en = chi_of(part, k < 2)
                part["tau"] -= tab.rate(k // 2, chi, en) * dt  # (views of d)
                f = torch.nonzero(part["tau"] < 0)[:, 0]
                hit.append(f + a)
                chis.append(chi[f])
            empty = torch.zeros(0, device="cuda", dtype=torch.float64)
            fired.append((torch.cat(hit) if hit else empty.long(), torch.cat(chis) if chis else empty))
        photons = [emit(tab, species[k], *fired[k], step, threshold) for k in (0, 1)]
        made = decay(tab, species[2], *fired[2], step)
        for k, more in ((0, made[:1]), (1, made[1:]), (2, photons)):
            species[k] = {c: torch.cat([v] + [m[c] for m in more]) for c, v in species[k].items()}
    out = dict(zip(("e", "p", "ph"), (exact_out(a, d, n) for a, d, n in zip(ps, species, n0))))
    if case["kind"] == "cascade":
        for o in out.values():
            o["fields"] = None  # (the fused push stores none)
        if case["prec"] == "f32":
            # of 10^6 emissions some come a step earlier or later than in 64 bits, and their products with them
            out["p"] = out["ph"] = None
    return out


def exact_burst(case, seed):
    s = burst(case, seed)
    parent, tab = s["parent"], Lookup(256)
    d = exact_rows(parent)
    n = case["n"]
    if case["kind"] == "emission":
        made = [emit(tab, d, s["fire"].idx, s["fire"].chi, 3, 0.0)]
    else:
        made = decay(tab, d, s["fire"].idx, s["fire"].chi, 3)
    res = {"parent": exact_out(parent, d, n)}
    for i, m in enumerate(made):
        rows = torch.zeros(len(ROWS), n, dtype=torch.float64, device="cuda")
        for r, c in enumerate(ROWS):
            if c in m:
                rows[r, m["x"].long()] = m[c]
        res["out%d" % i] = {"p": rows[:3], "tau": rows[3], "rest": rows[5:]}
    return res


def exact(case, seed):
    k = case["kind"]
    if k == "tables":
        top = prepare(case, seed)["params"].qs.chi_max
        arrays = table_arrays(case["n_chi"], case["n_xi"], (1e-3, top), (2e-2, top))
        return dict(zip(("qs_lnG", "qs_lnP", "bw_lnT", "bw_P"), arrays))
    if k in ("sampler", "gradients"):
        return exact_network(case, seed)
    if k in ("emission", "pairs"):
        return exact_burst(case, seed)
    return exact_steps(case, seed)
