"""What the estimator's speed is measured on: whole calls of the public entry points.

A case is a dict of plain values. ``call`` names the entry point:

* ``estimate``       one catalogue on the device, one ``Context.estimate``
* ``estimate_mu``    the same catalogue into (|k|, mu) bins, ``Context.estimate_mu``
* ``estimate_host``  a catalogue in pinned host memory, ``Context.estimate_host``
* ``batch``          many uneven catalogues, one ``BatchRunner`` pass

and ``source`` the particles: ``poisson`` (uniform), ``zeldovich`` (a displaced lattice,
n = n_side^3) or ``halos`` (an evolved snapshot: part of the particles in clumps of some
200 times the mean density, the rest uniform). One context serves a whole program, as it
does for a user: it keeps its cuFFT plans, tables and buffers from call to call.
"""
import math

import numpy as np
import torch

from paper_2005_06170_gb300 import catalogs, pkmom
from paper_2005_06170_gb300.batch import BatchRunner

THETA_SCALE = 0.02  # 1 / (H f) of the Zel'dovich velocities (f = 0.5, H = 100)


def _estimate(name, source, n, L, ng, nbins, **more):
    case = {"name": name, "call": "estimate", "source": source, "n": n, "L": L, "ng": ng, "nbins": nbins,
            "order": 4, "fp64": False, "mass": False, "bulk": True, "theta_sn": "tensor"}
    case.update(more)
    return case


def listed():
    return [
        # the smallest request of the serving loop: launches and latency count
        _estimate("request_100k_128", "poisson", 100_000, 300.0, 128, 64),
        # FP64, as used to validate: 32768 particles on 64^3 (the smallest benchmark workload)
        _estimate("fp64_32k_64", "poisson", 32_768, 256.0, 64, 32, fp64=True),
        # FP64 at a size that is used for reference spectra, weighted particles
        _estimate("fp64_1m_128", "poisson", 1_000_000, 400.0, 128, 64, fp64=True, mass=True),
        # one snapshot at one particle per cell: the medium and the default benchmark workload
        _estimate("zeldovich_256_256", "zeldovich", 256 ** 3, 1000.0, 256, 128),
        _estimate("zeldovich_512_512", "zeldovich", 512 ** 3, 1500.0, 512, 128),
        # the same snapshot on the finer grid of a resolution pair: the largest call
        _estimate("zeldovich_512_1024", "zeldovich", 512 ** 3, 1500.0, 1024, 128),
        # a sparse tracer sample on a fine grid (galaxies; 0.015 particle per cell), 3 * 2^7 grid
        _estimate("sparse_830k_384", "poisson", 830_584, 900.0, 384, 128),
        # an evolved, clustered snapshot with a mass per particle, particles in no order
        _estimate("halos_8m_256", "halos", 8_000_000, 500.0, 256, 128, mass=True),
        # TSC on a grid that is no multiple of 16, weighted, isotropic shot noise, no bulk rows
        _estimate("tsc_5m_200", "poisson", 5_000_000, 700.0, 200, 100, order=3, mass=True, bulk=False,
                  theta_sn="isotropic"),
        # direction-dependent spectra of a snapshot along a line of sight
        dict(_estimate("mu_256", "zeldovich", 256 ** 3, 1000.0, 256, 32), call="estimate_mu", nmu=8),
        # end to end from pinned host memory
        dict(_estimate("host_192", "zeldovich", 192 ** 3, 800.0, 192, 96), call="estimate_host"),
        # sixteen uneven catalogues in one pass, Poisson and Zel'dovich, grids 128, 256 and 384
        {"name": "batch_16", "call": "batch", "count": 16, "n_lo": 100_000, "n_hi": 4_000_000, "grids_seed": 1004,
         "nbins": 128},
    ]


def draw(rng):
    def log_uniform(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def grid(lo, hi):  # multiples of 8, the powers of two and their halves of three more often
        if rng.random() < 0.5:
            return rng.choice([g for g in (64, 96, 128, 192, 256, 384, 512) if lo <= g <= hi])
        return 8 * (log_uniform(lo, hi) // 8)

    kind = rng.choice(["estimate"] * 6 + ["fp64", "estimate_mu", "estimate_host", "batch"])
    if kind == "batch":
        return {"call": "batch", "count": rng.randint(2, 24), "n_lo": 100_000, "n_hi": log_uniform(200_000, 8_000_000),
                "grids_seed": rng.randrange(1 << 20), "nbins": rng.choice([32, 64, 128])}
    source = rng.choice(["poisson", "zeldovich", "halos"])
    if kind == "fp64":
        n, ng = log_uniform(30_000, 2_000_000), grid(48, 192)
    elif kind == "estimate_mu":
        n, ng = log_uniform(1_000_000, 20_000_000), grid(96, 256)
    elif kind == "estimate_host":
        n, ng = log_uniform(100_000, 8_000_000), grid(64, 256)
    else:
        n, ng = log_uniform(100_000, 40_000_000), grid(64, 512)
    if source == "zeldovich":
        n = (2 * max(8, round(0.5 * n ** (1.0 / 3.0)))) ** 3
    case = {"call": "estimate" if kind == "fp64" else kind, "source": source, "n": n,
            "L": round(rng.uniform(300.0, 1500.0), 1), "ng": ng, "nbins": rng.randint(12, ng // 2),
            "order": rng.choice([4, 4, 4, 4, 2, 3, 5]), "fp64": kind == "fp64", "mass": rng.random() < 0.4,
            "bulk": rng.random() < 0.8, "theta_sn": rng.choice(["tensor", "tensor", "isotropic"])}
    if kind == "estimate_mu":
        case.update(nbins=rng.randint(12, min(64, ng // 2)), nmu=rng.choice([2, 4, 5, 8, 10]), order=4)
    return case


# ---------------------------------------------------------------------------- inputs
def _halos(n, L, seed, dtype):
    """40 % of the particles in Gaussian clumps of 20 to 5000 particles (log-uniform sizes,
    about 200 times the mean density, a bulk velocity each and internal dispersion), the
    rest uniform, all in random order."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))

    def rand(*shape):
        return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)

    def randn(*shape):
        return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)

    want = (2 * n) // 5
    sizes = torch.exp(math.log(20.0) + math.log(250.0) * rand(want // 100 + 64)).long()
    halo = torch.repeat_interleave(torch.arange(sizes.numel(), device="cuda"), sizes)[:want]
    radius = (sizes.double() * (L ** 3 / n) / (200.0 * 4.0 / 3.0 * math.pi)) ** (1.0 / 3.0)
    centre, bulk = L * rand(sizes.numel(), 3), 300.0 * randn(sizes.numel(), 3)
    pos, vel = L * rand(n, 3), 300.0 * randn(n, 3)
    m = halo.numel()
    pos[:m] = centre[halo] + 0.5 * radius[halo, None] * randn(m, 3)
    vel[:m] = bulk[halo] + 200.0 * randn(m, 3)
    shuffle = torch.randperm(n, generator=g, device="cuda")
    pos = torch.remainder(pos[shuffle], L).to(dtype)
    pos[pos >= L] = 0
    return {"pos": pos.contiguous(), "vel": vel[shuffle].to(dtype).contiguous()}


def _particles(case, seed):
    """(pos, vel, mass or None) on the device."""
    dtype = torch.float64 if case["fp64"] else torch.float32
    if case["source"] == "zeldovich":
        side = round(case["n"] ** (1.0 / 3.0))
        cat = catalogs.zeldovich_torch(side, case["L"], seed=seed, dtype=dtype)
    elif case["source"] == "halos":
        cat = _halos(case["n"], case["L"], seed, dtype)
    else:
        cat = catalogs.poisson_torch(case["n"], case["L"], seed=seed, dtype=dtype)
    mass = None
    if case["mass"]:
        g = torch.Generator(device="cuda")
        g.manual_seed(int(seed) + 7)
        mass = 0.5 + torch.rand(case["n"], generator=g, device="cuda", dtype=dtype)
    return cat["pos"], cat["vel"], mass


def _params(case):
    return pkmom.params(case["L"], case["ng"], case["nbins"], order=case["order"],
                        precision=pkmom.F64 if case["fp64"] else pkmom.F32, theta_scale=THETA_SCALE,
                        bulk=case["bulk"], theta_sn=case["theta_sn"])


def _batch_shapes(case):
    """(n, ng, L, whether Zel'dovich) of each catalogue of a batch."""
    k = case["count"]
    counts = catalogs.log_uniform_counts(k, case["n_lo"], case["n_hi"], seed=case["grids_seed"])
    rng = np.random.Generator(np.random.PCG64(case["grids_seed"] + 1))
    lattice, grids, boxes = rng.random(k) < 0.5, rng.choice([128, 256, 384], size=k), rng.uniform(300.0, 1500.0, size=k)
    out = []
    for i in range(k):
        n = max(8, round(float(counts[i]) ** (1.0 / 3.0))) ** 3 if lattice[i] else int(counts[i])
        out.append((n, int(grids[i]), float(boxes[i]), bool(lattice[i])))
    return out


def _batch_catalogs(case, seed):
    out = []
    for i, (n, _, L, lattice) in enumerate(_batch_shapes(case)):
        if lattice:
            out.append(catalogs.zeldovich_torch(round(n ** (1.0 / 3.0)), L, seed=1000 * seed + i))
        else:
            out.append(catalogs.poisson_torch(n, L, seed=1000 * seed + i))
    return out


_CONTEXT = []


def _context():
    if not _CONTEXT:
        _CONTEXT.append(pkmom.Context(0))
    return _CONTEXT[0]


# ---------------------------------------------------------------------------- one pass
def prepare(case, seed):
    if case["call"] == "batch":
        params = [pkmom.params(L, ng, case["nbins"], theta_scale=THETA_SCALE) for _, ng, L, _ in _batch_shapes(case)]
        return {"call": "batch", "runner": BatchRunner(_batch_catalogs(case, seed), params)}
    pos, vel, mass = _particles(case, seed)
    if case["call"] == "estimate_host":
        pos, vel, mass = (None if t is None else t.cpu().pin_memory().numpy() for t in (pos, vel, mass))
    return {"call": case["call"], "ctx": _context(), "pos": pos, "vel": vel, "mass": mass, "p": _params(case),
            "nmu": case.get("nmu", 0)}


def run(state):
    if state["call"] == "batch":
        return state["runner"].run()
    ctx, pos, vel, mass, p = state["ctx"], state["pos"], state["vel"], state["mass"], state["p"]
    if state["call"] == "estimate_mu":
        return ctx.estimate_mu(pos, vel, p, state["nmu"], direction=(0.0, 0.0, 1.0), mass=mass)
    if state["call"] == "estimate_host":
        return ctx.estimate_host(pos, vel, p, mass=mass)
    return ctx.estimate(pos, vel, p, mass=mass)


def work(case):
    """Catalogue read once, spectra written once; the deposit's 2 * 4 * order^3 operations a
    particle, four real transforms, and about 60 operations a stored mode."""
    def one(n, ng, order, values, item, out):
        cells = float(ng) ** 3
        return (n * values * item + out * 8,
                8.0 * order ** 3 * n + 4 * 2.5 * cells * math.log2(cells) + 60.0 * 0.5 * cells)

    if case["call"] == "batch":
        parts = [one(n, ng, 4, 6, 4, 14 * case["nbins"]) for n, ng, _, _ in _batch_shapes(case)]
    else:
        out = 16 * case["nbins"] * case["nmu"] if case["call"] == "estimate_mu" else 14 * case["nbins"]
        parts = [one(case["n"], case["ng"], case["order"], 7 if case["mass"] else 6, 8 if case["fp64"] else 4, out)]
    return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}


# ---------------------------------------------------------------------------- in 64 bits
def _bspline(x, m):
    """The centred B-spline of order m at x, by truncated powers."""
    s = torch.zeros_like(x)
    for k in range(m + 1):
        s += (-1.0) ** k * math.comb(m, k) * torch.clamp(x + 0.5 * m - k, min=0.0) ** (m - 1)
    return s / math.factorial(m - 1)


def _transforms(pos, vel, mass, L, ng, order):
    """The real transforms of the four assigned grids, one after another. The grid
    coordinate is formed in the catalogue's precision; everything after it in 64 bits."""
    scale = torch.tensor(ng / L, dtype=pos.dtype, device=pos.device)
    n = pos.shape[0]
    chunk = 1 << 23
    for f in range(4):
        grid = torch.zeros(ng ** 3, dtype=torch.float64, device=pos.device)
        for i in range(0, n, chunk):
            u = (pos[i:i + chunk] * scale).double()
            q = torch.ones(u.shape[0], dtype=torch.float64, device=pos.device) if mass is None else \
                mass[i:i + chunk].double()
            if f:
                q = q * vel[i:i + chunk, f - 1].double()
            first = torch.floor(u + (0.5 if order % 2 else 0.0)) - (order - 1) // 2
            w, c = [], []
            for k in range(order):
                node = first + k
                w.append(_bspline(u - node, order))
                c.append(torch.remainder(node.long(), ng))
            for k0 in range(order):
                for k1 in range(order):
                    w01, c01 = q * w[k0][:, 0] * w[k1][:, 1], (c[k0][:, 0] * ng + c[k1][:, 1]) * ng
                    for k2 in range(order):
                        grid.index_add_(0, c01 + c[k2][:, 2], w01 * w[k2][:, 2])
        yield torch.fft.rfftn(grid.view(ng, ng, ng))
        del grid


def _axis_factors(ng, order):
    """Per frequency index 0 .. ng-1: the integer frequency, 1 / Bhat^2 and Sigma / Bhat^2."""
    i = torch.arange(ng, device="cuda")
    n = torch.where(i < ng // 2, i, i - ng)
    w = 2.0 * math.pi * n.double() / ng
    b2 = torch.special.sinc(w / (2.0 * math.pi)) ** (2 * order)
    at = torch.arange(1 - order, order, device="cuda", dtype=torch.float64)
    sigma = (_bspline(at, 2 * order)[None, :] * torch.cos(w[:, None] * at[None, :])).sum(1)
    return n, 1.0 / b2, sigma / b2


def _moments(vel, mass):
    v = vel.double()
    m = torch.ones(v.shape[0], dtype=torch.float64, device=v.device) if mass is None else mass.double()
    M, S2 = m.sum(), (m * m).sum()
    vb = (m[:, None] * v).sum(0) / M
    m2 = (m * m)[:, None]
    dv = v - vb
    return {"M": M, "S2": S2, "vb": vb, "R": (m2 * v).sum(0), "Rb": (m2 * dv).sum(0), "Q": (m2 * v).T @ v,
            "Qb": (m2 * dv).T @ dv}


def _slabs(F, ng, order, umin, umax, nbins, step):
    """Half-spectrum modes in slabs: frequencies, transforms, window factors and shell."""
    n, g, h = _axis_factors(ng, order)
    nh = ng // 2 + 1
    for a in range(0, ng, step):
        s = slice(a, min(a + step, ng))
        n0, n1 = n[s][:, None, None], n[None, :, None]
        n2 = torch.arange(nh, device="cuda")[None, None, :]
        nsq = n0 * n0 + n1 * n1 + n2 * n2
        u = torch.sqrt(nsq.double())
        b = torch.clamp(torch.floor((u - umin) * nbins / (umax - umin)), max=nbins - 1).long()
        inside = (nsq > 0) & (u >= umin) & (u <= umax)
        fields = [t[s] for t in F]
        yield (n0, n1, n2, u, b, inside, fields, g[s][:, None, None] * g[None, :, None] * g[None, None, :nh],
               h[s][:, None, None] * h[None, :, None] * h[None, None, :nh])


def _spectra64(pos, vel, mass, L, ng, nbins, order, bulk, theta_sn):
    mom = _moments(vel, mass)
    F = list(_transforms(pos, vel, mass, L, ng, order))
    kf, V = 2.0 * math.pi / L, L ** 3
    acc = torch.zeros((14, nbins), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 22) // (ng * (ng // 2 + 1)))
    for n0, n1, n2, u, b, ok, (d, *p), g, h in _slabs(F, ng, order, 1.0, ng / 2.0, nbins, step):
        wt = torch.where((n2 == 0) | (n2 == ng // 2), 1.0, 2.0).double().expand(u.shape)[ok]
        cell = b[ok]
        acc[0].index_add_(0, cell, wt * kf * u[ok])
        acc[1].index_add_(0, cell, wt)
        c = V / mom["M"] ** 2
        one = [acc[2], acc[9]]
        for row, val in zip(one, (c * g * d.abs() ** 2 - c * mom["S2"] * h, c * mom["S2"] * h)):
            row.index_add_(0, cell, wt * val[ok])
        k = [kf * n0.double(), kf * n1.double(), kf * n2.double()]
        for at, sn_at, Q, shift in ((3, 10, mom["Q"], 0.0), (6, 12, mom["Qb"], 1.0))[:2 if bulk else 1]:
            q = [p[i] - shift * mom["vb"][i] * d for i in range(3)]
            kp = k[0] * q[0] + k[1] * q[1] + k[2] * q[2]
            kqk = sum(k[i] * k[j] * Q[i, j] for i in range(3) for j in range(3)) if theta_sn == "tensor" else \
                (k[0] ** 2 + k[1] ** 2 + k[2] ** 2) * torch.trace(Q) / 3.0
            sn_pp, sn_tt = c * torch.trace(Q) * h, c * THETA_SCALE ** 2 * kqk * h
            vals = (c * g * sum(t.abs() ** 2 for t in q) - sn_pp, c * THETA_SCALE ** 2 * g * kp.abs() ** 2 - sn_tt,
                    c * THETA_SCALE * g * (d.conj() * kp).imag)
            for i, v in enumerate(vals + (sn_pp, sn_tt)):
                acc[at + i if i < 3 else sn_at + i - 3].index_add_(0, cell, wt * v[ok])
    count = acc[1].clone()
    out = acc / count
    out[1] = count
    if not bulk:
        out[6:9] = out[12:14] = math.nan
    empty = count == 0
    out[:, empty] = math.nan
    out[1, empty] = 0.0
    return out


def _spectra_mu64(pos, vel, mass, L, ng, nbins, nmu, order):
    """(|k|, mu) bins along z. A stored mode counts at mu and, mirrored (terms odd in k
    negated), at -mu; modes with a Nyquist component are left out. The mu bin is decided in
    32 bits."""
    mom = _moments(vel, mass)
    F = list(_transforms(pos, vel, mass, L, ng, order))
    kf, c, ts = 2.0 * math.pi / L, L ** 3 / mom["M"] ** 2, THETA_SCALE
    vb = mom["vb"]
    eb = vb / vb.norm()
    cells = nbins * nmu
    acc = torch.zeros((16, cells), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 22) // (ng * (ng // 2 + 1)))
    for n0, n1, n2, u, b, ok, (d, *p), g, h in _slabs(F, ng, order, 1.0, ng / 2.0, nbins, step):
        ok = ok & (n0 != -(ng // 2)) & (n1 != -(ng // 2)) & (n2 != ng // 2)
        q = [p[i] - vb[i] * d for i in range(3)]
        k = [kf * n0.double(), kf * n1.double(), kf * n2.double()]

        def dot(v):
            return k[0] * v[0] + k[1] * v[1] + k[2] * v[2]

        def quad(T):
            return sum(k[i] * k[j] * T[i, j] for i in range(3) for j in range(3))

        X, Xb = (-1j * c * ts * (g * d.conj() * dot(w) - h * dot(r)) for w, r in ((p, mom["R"]), (q, mom["Rb"])))
        sn_tt, im_sn = c * ts * ts * quad(mom["Q"]) * h, -c * ts * dot(mom["R"]) * h
        even = {0: kf * u, 2: torch.ones_like(u), 3: c * g * d.abs() ** 2 - c * mom["S2"] * h,
                4: c * g * sum(t.abs() ** 2 for t in p) - c * torch.trace(mom["Q"]) * h,
                5: c * ts * ts * g * dot(p).abs() ** 2 - sn_tt, 6: X.real,
                8: c * g * sum(t.abs() ** 2 for t in q) - c * torch.trace(mom["Qb"]) * h,
                9: c * ts * ts * (g * dot(q).abs() ** 2 - quad(mom["Qb"]) * h), 10: Xb.real,
                12: c * g * (d.conj() * sum(eb[i] * q[i] for i in range(3))).real - c * (eb @ mom["Rb"]) * h,
                13: c * mom["S2"] * h, 14: sn_tt}
        odd = {1: n2.double() / u.clamp(min=1.0), 7: X.imag, 11: Xb.imag, 15: im_sn}
        mu32 = n2.float() / torch.sqrt((n0 * n0 + n1 * n1 + n2 * n2).float()).clamp(min=1.0)
        for sign, use in ((1.0, ok), (-1.0, ok & (n2 > 0))):
            m = torch.clamp(torch.floor((sign * mu32 + 1.0) * (0.5 * nmu)), 0, nmu - 1).long()
            cell = (b * nmu + m)[use]
            for terms, s in ((even, 1.0), (odd, sign)):
                for row, v in terms.items():
                    acc[row].index_add_(0, cell, s * v.expand(u.shape)[use])
    count = acc[2].clone()
    out = acc / count
    out[2] = count
    empty = count == 0
    out[:, empty] = math.nan
    out[2, empty] = 0.0
    return out


def exact(case, seed):
    if case["call"] == "batch":
        if sum(n for n, _, _, _ in _batch_shapes(case)) > 40_000_000:
            return None
        return [_spectra64(c["pos"], c["vel"], None, L, ng, case["nbins"], 4, True, "tensor")
                for c, (_, ng, L, _) in zip(_batch_catalogs(case, seed), _batch_shapes(case))]
    pos, vel, mass = _particles(case, seed)
    if case["call"] == "estimate_mu":
        return _spectra_mu64(pos, vel, mass, case["L"], case["ng"], case["nbins"], case["nmu"], case["order"])
    out = _spectra64(pos, vel, mass, case["L"], case["ng"], case["nbins"], case["order"], case["bulk"],
                     case["theta_sn"])
    return out.cpu().numpy() if case["call"] == "estimate_host" else out
