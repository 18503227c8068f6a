"""The framework's work as its users have it do, one entry per way of use.

Every case goes through the public binding (``paper_1201_5651_gb300.oots``): a
context (or a batch of contexts, or the allocation-free trace) with its grid,
density, sources and scheme is what a program keeps; a pass hands in a state
on the device, takes one or a few substeps and reads the state back.  Sizes
and physics are those of the repository's workloads (``inputs.py``, the
benchmark and the accuracy study): Stromgren spheres, lognormal and clumpy
gas, batches of small grids, sixteen sources in a large box, the slab.

States are made as the method meets them: each source has ionised its
surroundings up to a front, found by sharing its photons out along rays from
the source; behind the front the gas sits near ionisation equilibrium, beyond
it the gas is neutral.

``exact`` repeats a pass in 64 bits with torch alone: short characteristics
shell by shell, the rates from the spectrum itself, every cell's equation by
quadrature of the time it takes to reach a state.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1201_5651_gb300 import oots

ALPHA, SIGMA, TAU0 = 2.59e-13, 6.3e-18, 0.6
X_NEUTRAL = 1.0 - 1e-6
TEMPS = (3.0e4, 3.4e4, 3.75e4, 4.0e4, 4.4e4, 5.0e4)      # blackbody sources take these in turn
A1, A2, A3 = oots.OOTS_A1, oots.OOTS_A2, oots.OOTS_A3


def _grid(name, nx, ny, nz, **kw):
    """A single grid: defaults are one blackbody source in lognormal gas, A3 under K4 = 1/4."""
    c = {"name": name, "kind": "grid", "nx": nx, "ny": ny, "nz": nz, "precision": "mixed", "scheme": A3,
         "density": "lognormal", "nsrc": 1, "spectrum": "bb", "place": "centre", "plane": -1, "box": 2.5,
         "age": 0.05, "K1": 0.0, "K3": 0.0, "K4": 0.25, "dt_trec": 0.0, "shape": -1, "steps": 1, "call": "run",
         "recombine": True}
    c.update(kw)
    return c


def listed():
    return [
        # The slab of Sect. 3.1 in FP64 under A1: 100 cells, one row, the smallest call there is.
        _grid("slab100_a1_fp64", 100, 1, 1, precision="fp64", scheme=A1, density="uniform", spectrum="mono",
              plane=0, K4=0.0, dt_trec=0.0005, recombine=False, call="advance", box=0.0, age=0.02),
        # The Stromgren sphere of Sect. 3.2 at 32^3, source in the corner, advanced by eight
        # fixed steps of t_rec/1000: launches and the wavefront's latency.
        _grid("stromgren32_advance", 32, 32, 32, density="uniform", spectrum="mono", place="corner", box=1.5,
              K4=0.0, dt_trec=0.001, steps=8, call="advance"),
        # A program with its own time loop: the step asked for, then taken, on a ragged grid
        # with the source off centre (the coupling of a hydrodynamics code).
        _grid("loop_50x41x37", 50, 41, 37, spectrum="mono", place="random", call="step"),
        # The allocation-free trace on caller-owned buffers, ragged sides.
        {"name": "trace_150x97x70", "kind": "trace", "nx": 150, "ny": 97, "nz": 70, "precision": "mixed", "box": 2.5,
         "age": 0.05},
        # The plain FP64 path, lognormal gas and a blackbody source (the reference runs of the accuracy checks).
        _grid("lognormal64_fp64", 64, 64, 64, precision="fp64"),
        # A1 on the accuracy study's 88^3 grid (cell optical depth 3): every cell integrates on the sweep's chain.
        _grid("stromgren88_a1", 88, 88, 88, scheme=A1, density="uniform", place="corner", box=1.1, K1=0.1, K4=0.0),
        # The example of the documentation: 128^3 lognormal gas, one blackbody source, nothing tuned.
        _grid("lognormal128_bb", 128, 128, 128),
        # Several sources of both kinds on an odd, non-cubic grid, first-order scheme under K3, nothing tuned.
        _grid("multi5_117x93x141_a2", 117, 93, 141, scheme=A2, nsrc=5, spectrum="both", place="random", K3=0.25, K4=0.0,
              age=0.02),
        # A plane-parallel blackbody source across a 256^3 box.
        _grid("plane256_bb", 256, 256, 256, plane=0, box=0.0, age=0.02),
        # The clumpy 256^3 box with a monochromatic source, on the tiles the tuner picks for it.
        _grid("clumpy256_mono", 256, 256, 256, density="clumpy", spectrum="mono", shape=8),
        # Sixty-four uneven grids advanced together, each with its own step.
        {"name": "batch64", "kind": "batch", "count": 64, "lo": 32, "hi": 128, "sides": 1204, "precision": "mixed",
         "scheme": A3, "K4": 0.25, "shape": 8, "box": 2.0, "age": 0.02},
        # The benchmark: 512^3 cells, sixteen blackbody sources, on the tiles the tuner picks for it.
        _grid("multisource512", 512, 512, 512, nsrc=16, place="random", shape=7, box=2.0, age=0.005),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges: sides spread over their logarithm, ragged ones among them."""
    kind = rng.choice(["single", "single", "multi", "multi", "fp64", "a1", "plane", "batch", "trace", "loop"])
    prec = rng.choice(["mixed", "mixed", "fp64"])
    seed = rng.randrange(1 << 20)                       # batches: their sides

    def sides(lo, hi):
        n = _logint(rng, lo, hi)
        return [max(lo // 2, int(n * rng.uniform(0.7, 1.0))) if rng.random() < 0.6 else n for _ in range(3)]

    if kind == "trace":
        nx, ny, nz = sides(24, 150)
        return {"kind": "trace", "nx": nx, "ny": ny, "nz": nz, "precision": prec, "box": 2.5,
                "age": round(rng.uniform(0.01, 0.2), 4)}
    if kind == "batch":
        return {"kind": "batch", "count": _logint(rng, 2, 48), "lo": 16, "hi": _logint(rng, 32, 112), "sides": seed,
                "precision": "mixed", "scheme": rng.choice([A2, A3]), "K4": rng.choice([0.25, 0.125]),
                "shape": rng.choice([-1, 7, 8]), "box": 2.0, "age": round(rng.uniform(0.01, 0.1), 4)}
    spec, age = rng.choice(["mono", "bb"]), round(rng.uniform(0.01, 0.2), 4)
    crit = rng.choice([{"K4": 0.25}, {"K4": 0.5}, {"K4": 0.0625}, {"K4": 0.0, "K3": 0.25}])
    dens = rng.choice(["lognormal", "lognormal", "uniform", "clumpy"])
    common = dict(spectrum=spec, age=age, density=dens, place=rng.choice(["centre", "corner", "random"]), **crit)
    if kind == "single":
        c = _grid("", *sides(32, 256), scheme=rng.choice([A3, A3, A2]), shape=rng.choice([-1, -1, 8, 2]),
                  call=rng.choice(["run", "run", "advance"]), **common)
    elif kind == "multi":
        c = _grid("", *sides(40, 256), nsrc=_logint(rng, 2, 16), shape=rng.choice([-1, 7, 8]), **common)
        c.update(place="random", age=round(0.2 * age, 5), spectrum=rng.choice(["bb", "bb", "both"]))
    elif kind == "fp64":
        c = _grid("", *sides(20, 72), precision="fp64", **common)
    elif kind == "a1":
        c = _grid("", *sides(16, 80), scheme=A1, **common)
        c.update(K1=rng.choice([1.0, 0.1]), K3=0.0, K4=0.0)
    elif kind == "plane":
        c = _grid("", *sides(32, 256), plane=rng.randrange(6), scheme=rng.choice([A2, A3]), **common)
        c.update(box=0.0, age=round(rng.uniform(0.01, 0.05), 4))
    else:
        c = _grid("", *sides(16, 96), call="step", precision=prec if dens == "uniform" else "mixed", **common)
    if c["call"] == "advance":
        c.update(K3=0.0, K4=0.0, dt_trec=rng.choice([0.0005, 0.001, 0.002]), steps=rng.choice([2, 4, 8]))
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda" if torch.cuda.is_available() else "cpu")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _rand(g, n, lo, hi):
    return [lo + (hi - lo) * float(v) for v in torch.rand(n, generator=g, device=g.device, dtype=torch.float64)]


def _density(kind, nz, ny, nx, g):
    """Hydrogen density (mean 100): uniform, lognormal with P(k) ~ k^-3, or lognormal with dense clumps."""
    if kind == "uniform":
        return None
    dev = g.device
    sigma = 1.5 if kind == "clumpy" else 1.0
    m = [v + (v & 1) for v in (nz, ny, nx)]
    fk = torch.fft.rfftn(torch.randn(m, generator=g, device=dev, dtype=torch.float64))
    k2 = (torch.fft.fftfreq(m[0], device=dev, dtype=torch.float64)[:, None, None] ** 2
          + torch.fft.fftfreq(m[1], device=dev, dtype=torch.float64)[None, :, None] ** 2
          + torch.fft.rfftfreq(m[2], device=dev, dtype=torch.float64)[None, None, :] ** 2)
    k2[0, 0, 0] = 1.0
    fk *= k2 ** -0.75
    fk[0, 0, 0] = 0.0
    f = torch.fft.irfftn(fk, s=m)[:nz, :ny, :nx]
    del fk, k2
    f = (f - f.mean()) / f.std()
    rho = torch.exp_(f.mul_(sigma))
    rho *= 100.0 / rho.mean()
    if kind == "clumpy":
        count = max(1, 200 * nx * ny * nz // 256 ** 3)
        zz, yy, xx = (torch.arange(n, device=dev, dtype=torch.float64) + 0.5 for n in (nz, ny, nx))
        for _ in range(count):
            cz, cy, cx, r, od = _rand(g, 5, 0.0, 1.0)
            r, od = 2.0 + 6.0 * r, 10.0 ** (1.0 + od)
            c = (cz * nz, cy * ny, cx * nx)
            lo = [max(0, int(v - r)) for v in c]
            hi = [int(v + r) + 2 for v in c]
            s = tuple(slice(a, b) for a, b in zip(lo, hi))
            d2 = ((zz[s[0]] - c[0]) ** 2)[:, None, None] + ((yy[s[1]] - c[1]) ** 2)[None, :, None] \
                + ((xx[s[2]] - c[2]) ** 2)[None, None, :]
            rho[s] = torch.where(d2 <= r * r, rho[s] * od, rho[s])
    return rho.contiguous()


def _sources(case, dims, g, qtot=1e48):
    """(vertex, Q, spectrum, T) per point source; the summed rate of several is what the box is sized by."""
    nsrc, n = case["nsrc"], dims
    out = []
    for s in range(nsrc):
        u = _rand(g, 4, 0.0, 1.0)
        if case["place"] == "corner":
            v = (0, 0, 0)
        elif case["place"] == "centre":
            v = tuple(m // 2 for m in n)
        else:
            v = tuple(min(m, 1 + int(q * (m - 1))) for q, m in zip(u[:3], n))
        bb = case["spectrum"] == "bb" or (case["spectrum"] == "both" and s % 2 == 0)
        q = qtot if nsrc == 1 else math.exp(math.log(1e47) + u[3] * math.log(100.0))
        out.append((v, q, "bb" if bb else "mono", TEMPS[(s + 3) % len(TEMPS)] if bb else 0.0))
    return out


def _strom(q, n=100.0):
    return (3.0 * q / (4.0 * math.pi * n * n * ALPHA)) ** (1.0 / 3.0)


class _Spectrum:
    """Transmitted fraction P(N) of a source's photons and its slope, from the photon spectrum itself
    (a delta at nu0, or a blackbody on [nu0, 40 nu0] with sigma ~ nu^-3)."""

    LO, HI, K = math.log(1e8), math.log(1e25), 16384
    _cache = {}

    def __init__(self, T, dev):
        self.T = T
        if not T:
            return
        x, w = np.polynomial.legendre.leggauss(16)
        e = np.linspace(0.0, math.log(40.0), 81)
        ln_nu = (0.5 * (e[1:] + e[:-1])[:, None] + 0.5 * np.diff(e)[:, None] * x).ravel()
        nu = torch.tensor(np.exp(ln_nu), device=dev)
        wt = torch.tensor((0.5 * np.diff(e)[:, None] * w).ravel(), device=dev) * nu
        phi = wt * nu * nu / torch.expm1((13.6 / 8.617333262e-5) / T * nu)
        phi = phi / phi.sum()
        sg = SIGMA / nu ** 3
        lnN = torch.linspace(self.LO, self.HI, self.K, device=dev, dtype=torch.float64)
        y, d1, z, d2 = [], [], [], []
        for part in lnN.split(2048):
            N = part.exp()
            t = -sg[None, :] * N[:, None]
            top = t.max(1, keepdim=True).values
            ex = phi * (t - top).exp()
            m0, m1, m2 = ex.sum(1), (ex * sg).sum(1), (ex * sg * sg).sum(1)
            thin = (phi * torch.expm1(t)).sum(1)
            y.append(torch.where(thin > -0.5, torch.log1p(thin.clamp(min=-0.9)), top[:, 0] + m0.log()))
            d1.append(-N * m1 / m0)
            z.append(top[:, 0] + m1.log())
            d2.append(-N * m2 / m1)
        self.h = (self.HI - self.LO) / (self.K - 1)
        self.t = [torch.cat(v) for v in (y, d1, z, d2)]
        self.s1 = float((phi * sg).sum())

    @classmethod
    def of(cls, T, dev):
        key = (T, str(dev))
        if key not in cls._cache:
            cls._cache[key] = cls(T, dev)
        return cls._cache[key]

    def _at(self, N, f, d):
        u = ((N.clamp(min=1.000001e8).log() - self.LO) / self.h).clamp(0.0, self.K - 1.000001)
        k = u.floor().long()
        t = u - k
        y0, y1, m0, m1 = f[k], f[k + 1], d[k] * self.h, d[k + 1] * self.h
        return y0 + t * (m0 + t * (3 * (y1 - y0) - 2 * m0 - m1 + t * (2 * (y0 - y1) + m0 + m1)))

    def lnP(self, N):
        if not self.T:
            return -SIGMA * N
        return torch.where(N < 1e9, torch.log1p(-self.s1 * N), self._at(N, self.t[0], self.t[1]))

    def slope(self, N):
        """-dP/dN."""
        if not self.T:
            return SIGMA * torch.exp(-SIGMA * N)
        return torch.where(N < 1e9, self.s1 + 0.0 * N, self._at(N, self.t[2], self.t[3]).exp())


def _front(v, q, T, n, dims, dx, t, alpha, dev):
    """Along rays from a vertex: how many photons it takes to ionise the gas up to a radius, over those
    sent out in time t, and the column through the gas behind the front.  Tables over (theta, phi, r)."""
    nx, ny, nz = dims
    nr = int(math.sqrt(sum(max(a, m - a) ** 2 for a, m in zip(v, dims)))) + 3
    side = max(dims)
    nth, nph = max(12, min(96, side)), max(24, min(192, 2 * side))
    th = (torch.arange(nth, device=dev) + 0.5) * (math.pi / nth)
    ph = (torch.arange(nph, device=dev) + 0.5) * (2 * math.pi / nph)
    r = torch.arange(nr, device=dev) + 0.5
    d = [th.sin()[:, None, None] * ph.cos()[None, :, None], th.sin()[:, None, None] * ph.sin()[None, :, None],
         th.cos()[:, None, None].expand(nth, nph, 1)]
    if n is None:
        nn = torch.full((nth, nph, nr), 100.0, device=dev)
    else:
        ix = [(a + e * r).floor().long() for a, e in zip(v, d)]
        ok = (ix[0] >= 0) & (ix[0] < nx) & (ix[1] >= 0) & (ix[1] < ny) & (ix[2] >= 0) & (ix[2] < nz)
        i, j, k = (m.clamp(0, s - 1) for m, s in zip(ix, dims))
        nn = torch.where(ok, n[k, j, i].float(), torch.zeros((), device=dev))
    shell = 4.0 * math.pi * (r.double() * dx) ** 2 * dx
    need = (torch.cumsum(nn.double() * (1.0 + 0.5 * alpha * nn.double() * t) * shell, 2) / (q * t)).float()
    sp = _Spectrum.of(T, dev)
    flux = q / (4.0 * math.pi * (r.double() * dx) ** 2)
    N = torch.zeros(nth, nph, nr, device=dev, dtype=torch.float64)
    for _ in range(3):
        x = (alpha * nn.double() / (flux * sp.slope(N)).clamp(min=1e-300)).clamp(max=0.5)
        N = torch.cumsum(nn.double() * x * dx, 2)
        N = torch.cat([torch.zeros_like(N[..., :1]), N[..., :-1]], 2)
    return need, N


def _developed(dims, dx, n, srcs, t, alpha, dev):
    """Neutral fraction after the sources have shone for about t: float64, (nz, ny, nx)."""
    nx, ny, nz = dims
    tabs = [_front(v, q, T, n, dims, dx, t, alpha, dev) for v, q, _, T in srcs]
    out = torch.empty(nz, ny, nx, device=dev, dtype=torch.float64)
    step = max(1, (1 << 23) // (nx * ny))
    X = torch.arange(nx, device=dev) + 0.5
    Y = torch.arange(ny, device=dev) + 0.5
    for z0 in range(0, nz, step):
        z1 = min(nz, z0 + step)
        Z = torch.arange(z0, z1, device=dev) + 0.5
        neutral = torch.ones(z1 - z0, ny, nx, device=dev)
        gamma = torch.zeros(z1 - z0, ny, nx, device=dev, dtype=torch.float64)
        for (v, q, _, T), (need, N) in zip(srcs, tabs):
            nth, nph, nr = need.shape
            px, py, pz = (X - v[0])[None, None, :], (Y - v[1])[None, :, None], (Z - v[2])[:, None, None]
            r = (px * px + py * py + pz * pz).sqrt()
            a = (torch.acos((pz / r).clamp(-1, 1)) * (nth / math.pi)).long().clamp(0, nth - 1)
            b = (torch.remainder(torch.atan2(py, px), 2 * math.pi) * (nph / (2 * math.pi))).long().clamp(0, nph - 1)
            k = r.long().clamp(0, nr - 1)
            at = (a * nph + b.expand_as(a)) * nr + k
            hi = need.view(-1)[at]
            lo = torch.where(k > 0, need.view(-1)[(at - 1).clamp(min=0)], torch.zeros_like(hi))
            neutral = torch.minimum(neutral, ((hi - 1.0) / (hi - lo).clamp(min=1e-12)).clamp(0.0, 1.0))
            slope = _Spectrum.of(T, dev).slope(N.view(-1)[at])
            gamma += q / (4.0 * math.pi * (r.double() * dx) ** 2) * slope
        c = alpha * (100.0 if n is None else n[z0:z1])
        ratio = gamma / c if alpha > 0 else gamma * 1e12
        eq = 2.0 / (2.0 + ratio + torch.sqrt(ratio * (ratio + 4.0)))       # c (1-x)^2 = gamma x
        out[z0:z1] = neutral * X_NEUTRAL + (1.0 - neutral) * eq
    return out


def _slab(dims, dx, n, code, flux, T, t, alpha, dev):
    """The same for a plane-parallel source: rows along its axis."""
    axis, back = code // 2, code & 1
    rho = torch.full((dims[2], dims[1], dims[0]), 100.0, device=dev, dtype=torch.float64) if n is None else n
    rho = rho.flip(2 - axis) if back else rho
    need = torch.cumsum(rho * (1.0 + 0.5 * alpha * rho * t) * dx, 2 - axis) / (flux * t)
    lo = need - rho * dx / (flux * t)
    neutral = ((need - 1.0) / (need - lo).clamp(min=1e-12)).clamp(0.0, 1.0)
    sp = _Spectrum.of(T, dev)
    N = torch.zeros_like(rho)
    for _ in range(3):
        gamma = flux * sp.slope(N)
        ratio = gamma / (alpha * rho) if alpha > 0 else gamma * 1e12
        eq = 2.0 / (2.0 + ratio + torch.sqrt(ratio * (ratio + 4.0)))
        N = torch.cumsum(rho * eq * dx, 2 - axis) - rho * eq * dx
    x = neutral * X_NEUTRAL + (1.0 - neutral) * eq
    return (x.flip(2 - axis) if back else x).contiguous()


def _inputs(case, seed):
    """Everything of a single grid (or of the trace), from the seed alone."""
    g = _gen(seed)
    dev = g.device
    dims = (case["nx"], case["ny"], case["nz"])
    real = torch.float64 if case["precision"] == "fp64" else torch.float32
    if case["kind"] == "trace":
        case = dict(_grid("", *dims, place="random", spectrum="mono"), **case)
    alpha = ALPHA if case["recombine"] else 0.0
    n = _density(case["density"], dims[2], dims[1], dims[0], g)
    trec = 1.0 / (ALPHA * 100.0)
    t = case["age"] * trec * _rand(g, 1, 0.8, 1.2)[0]
    p = {"dims": dims, "n": n, "alpha": alpha, "trec": trec, "plane": case["plane"], "srcs": []}
    if case["plane"] >= 0:
        # cell optical depth 10 in the uniform slab, 2 at the mean density otherwise; the front some way in
        p["dx"] = (10.0 if n is None else 2.0) / (SIGMA * 100.0)
        T = 4.0e4 if case["spectrum"] == "bb" else 0.0
        flux = dims[case["plane"] // 2] * p["dx"] * 100.0 * 0.4 / (case["age"] * trec)
        x = _slab(dims, p["dx"], n, case["plane"], flux, T, t, alpha, dev)
        p["srcs"] = [(None, flux, case["spectrum"], T)]
    else:
        p["srcs"] = _sources(case, dims, g)
        p["dx"] = case["box"] * _strom(sum(s[1] for s in p["srcs"])) / max(dims)
        x = _developed(dims, p["dx"], n, p["srcs"], t, alpha, dev)
    p["x"] = x.to(real).contiguous()
    return p


def _batch_inputs(case, seed):
    pick = np.random.default_rng(case["sides"])
    g = _gen(seed)
    real = torch.float64 if case["precision"] == "fp64" else torch.float32
    allowed = [s for s in (16, 24, 32, 48, 64, 80, 96, 112, 128) if case["lo"] <= s <= case["hi"]]
    if case["hi"] == 128:
        allowed = [32, 48, 64, 96, 128]
    out = []
    for _ in range(case["count"]):
        m = int(pick.choice(allowed))
        u = _rand(g, 6, 0.0, 1.0)
        nH, q = 10.0 * 100.0 ** u[0], 1e47 * 1000.0 ** u[1]
        v = tuple(1 + int(a * (m - 1)) for a in u[2:5])
        dx = case["box"] * _strom(q, nH) / m
        trec = 1.0 / (ALPHA * nH)
        t = case["age"] * trec * (0.8 + 0.4 * u[5])
        n = torch.full((m, m, m), nH, device=g.device, dtype=torch.float64)
        x = _developed((m, m, m), dx, n, [(v, q, "mono", 0.0)], t, ALPHA, g.device)
        out.append({"dims": (m, m, m), "dx": dx, "nH": nH, "srcs": [(v, q, "mono", 0.0)], "trec": trec,
                    "x": x.to(real).contiguous()})
    return out


def _context(p, case, n_uniform):
    c = oots.Context(0, case["precision"])
    c.set_grid(*p["dims"], p["dx"])
    c.set_physics(p.get("alpha", ALPHA), SIGMA, TAU0)
    c.set_density(n_uniform if p.get("n") is None else p["n"].cpu().numpy())
    for v, q, spec, T in p["srcs"]:
        if v is None:
            c.add_plane_source(p["plane"] // 2, -1 if p["plane"] & 1 else 1, q, spec, T)
        else:
            c.add_source([float(a) for a in v], q, spec, T)
    c.set_scheme(case["scheme"], K1=case.get("K1", 0.0), K3=case.get("K3", 0.0), K4=case["K4"],
                 dt_fixed=case.get("dt_trec", 0.0) * p["trec"])
    if case["shape"] >= 0:
        c.set_tile_shape(case["shape"])
    return c


def prepare(case, seed):
    if case["kind"] == "batch":
        ps = _batch_inputs(case, seed)
        ctxs = [_context(p, case, p["nH"]) for p in ps]
        s = {"kind": "batch", "ctxs": ctxs, "batch": oots.Batch(ctxs), "x": [p["x"] for p in ps],
             "out": [torch.empty_like(p["x"]) for p in ps], "t_end": [1e30] * len(ps)}
    elif case["kind"] == "trace":
        p = _inputs(case, seed)
        s = dict(p, kind="trace", n=p["n"].to(p["x"].dtype), out=torch.empty_like(p["x"]),
                 prec=oots.OOTS_FP64 if case["precision"] == "fp64" else oots.OOTS_MIXED)
    else:
        p = _inputs(case, seed)
        s = {"kind": case["call"], "ctx": _context(p, case, 100.0), "x": p["x"], "out": torch.empty_like(p["x"]),
             "steps": case["steps"], "t_end": case["steps"] * case["dt_trec"] * p["trec"]}
    torch.cuda.synchronize()
    return s


def run(s):
    if s["kind"] == "trace":
        x = s["x"]
        oots.oots_trace_noalloc(0, s["prec"], *s["dims"], s["dx"], s["n"].data_ptr(), 0.0, x.data_ptr(),
                                s["srcs"][0][0], SIGMA, TAU0, s["out"].data_ptr())
        return {"column": s["out"]}
    if s["kind"] == "batch":
        f32 = s["x"][0].dtype == torch.float32
        for c, x in zip(s["ctxs"], s["x"]):
            c.set_neutral_fraction_device(x.data_ptr(), f32)
            c.synchronize()                      # each context has its own stream; the batch runs on the first's
        s["batch"].run_substeps(1, s["t_end"])
        s["ctxs"][0].synchronize()
        for c, o in zip(s["ctxs"], s["out"]):
            c.get_neutral_fraction_device(o.data_ptr(), f32)
        for c in s["ctxs"]:
            c.synchronize()
        return {"x": s["out"]}
    c, x, out = s["ctx"], s["x"], s["out"]
    f32 = x.dtype == torch.float32
    c.set_neutral_fraction_device(x.data_ptr(), f32)
    if s["kind"] == "advance":
        c.set_time(0.0)
        c.advance(s["t_end"])
    elif s["kind"] == "step":
        c.step(c.compute_dt())
    else:
        c.run_substeps(s["steps"], 1e30)
    c.get_neutral_fraction_device(out.data_ptr(), f32)
    c.synchronize()                              # as a program does before it reads the copy on another stream
    return {"x": out}


def _batch_sides(case):
    pick = np.random.default_rng(case["sides"])
    allowed = [s for s in (16, 24, 32, 48, 64, 80, 96, 112, 128) if case["lo"] <= s <= case["hi"]]
    if case["hi"] == 128:
        allowed = [32, 48, 64, 96, 128]
    return [int(pick.choice(allowed)) for _ in range(case["count"])]


def work(case):
    """State in and out, and the density once (columns, half-step states and rates need not leave the
    chip); per trace and cell about 40 operations, per integration and source about 60 (FP64 and A1
    cells need no fewer)."""
    e = 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "batch":
        cells = sum(m ** 3 for m in _batch_sides(case))
        return {"bytes": 2 * e * cells, "flops": cells * (200 if case["scheme"] == A3 else 100)}
    cells = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "trace":
        return {"bytes": 3 * e * cells, "flops": 40 * cells}
    stages = 2 if case["scheme"] == A3 else 1
    return {"bytes": (2 + (case["density"] != "uniform")) * e * cells,
            "flops": cells * case["steps"] * case["nsrc"] * 100 * stages}


# ------------------------------------------------------------------------------------------------ 64-bit values
def _octants(a, v, dims, ext):
    """The eight octants of a (nz, ny, nx) array around vertex v as (8, Ex, Ey, Ez), zero beyond the grid."""
    out = torch.zeros(8, *ext, device=a.device, dtype=a.dtype)
    b = a.permute(2, 1, 0)
    for o in range(8):
        s, f = [], []
        for q in range(3):
            back = (o >> q) & 1
            s.append(slice(0, v[q]) if back else slice(v[q], dims[q]))
            if back:
                f.append(q)
        part = b[tuple(s)].flip(f) if f else b[tuple(s)]
        out[o, :part.shape[0], :part.shape[1], :part.shape[2]] = part
    return out


def _from_octants(p, v, dims):
    out = torch.zeros(dims[2], dims[1], dims[0], device=p.device, dtype=p.dtype)
    b = out.permute(2, 1, 0)
    for o in range(8):
        s, e, f = [], [], []
        for q in range(3):
            back = (o >> q) & 1
            e.append(v[q] if back else dims[q] - v[q])
            s.append(slice(0, v[q]) if back else slice(v[q], dims[q]))
            if back:
                f.append(q)
        part = p[o, :e[0], :e[1], :e[2]]
        b[tuple(s)] = part.flip(f) if f else part
    return out


class _Shells:
    """Cells of the octants around a vertex in shells max(i, j, k) = m, each from the one before."""

    def __init__(self, v, dims, dx):
        self.v, self.dims = v, dims
        self.ext = [max(a, m - a) for a, m in zip(v, dims)]
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        c = [torch.arange(e, device=self.dev, dtype=torch.float64) + 0.5 for e in self.ext]
        c = [c[0][:, None, None], c[1][None, :, None], c[2][None, None, :]]
        top = torch.maximum(torch.maximum(c[0], c[1]), c[2])
        self.r2 = c[0] ** 2 + c[1] ** 2 + c[2] ** 2
        self.sf = self.r2.sqrt() / top
        self.ties = (c[0] == top).double() + (c[1] == top).double() + (c[2] == top).double()
        self.dx = dx

    def into(self, a):
        return _octants(a, self.v, self.dims, self.ext)

    def back(self, a):
        return _from_octants(a, self.v, self.dims)

    def entry(self, m, Nout, W, Nin):
        """Entry columns of shell m, averaged over tied axes, into Nin."""
        for a in range(3):
            if m == 0 or m >= self.ext[a]:
                continue
            t = [(a + 1) % 3, (a + 2) % 3]
            order = (0, a + 1, t[0] + 1, t[1] + 1)
            r = [min(m + 1, self.ext[q]) for q in t]
            No, Wo = (q.permute(order)[:, m - 1, :r[0], :r[1]] for q in (Nout, W))
            g = [(torch.arange(k, device=self.dev, dtype=torch.float64) + 0.5) / (m + 0.5) for k in r]
            g1, g2 = g[0][:, None], g[1][None, :]
            NW = No * Wo
            num = (1 - g1) * (1 - g2) * NW
            den = (1 - g1) * (1 - g2) * Wo
            num[:, 1:] += g1[1:] * (1 - g2) * NW[:, :-1]
            den[:, 1:] += g1[1:] * (1 - g2) * Wo[:, :-1]
            num[:, :, 1:] += (1 - g1) * g2[:, 1:] * NW[:, :, :-1]
            den[:, :, 1:] += (1 - g1) * g2[:, 1:] * Wo[:, :, :-1]
            num[:, 1:, 1:] += g1[1:] * g2[:, 1:] * NW[:, :-1, :-1]
            den[:, 1:, 1:] += g1[1:] * g2[:, 1:] * Wo[:, :-1, :-1]
            share = self.ties.permute(order[1] - 1, order[2] - 1, order[3] - 1)[m, :r[0], :r[1]]
            Nin.permute(order)[:, m, :r[0], :r[1]] += torch.nan_to_num(num / den) / share

    def faces(self, m):
        """Index tuples that cover shell m once."""
        e = [min(m + 1, q) for q in self.ext]
        lo = [min(m, q) for q in self.ext]
        if m < self.ext[0]:
            yield (slice(None), m, slice(0, e[1]), slice(0, e[2]))
        if m < self.ext[1]:
            yield (slice(None), slice(0, lo[0]), m, slice(0, e[2]))
        if m < self.ext[2]:
            yield (slice(None), slice(0, lo[0]), slice(0, lo[1]), m)


def _columns(sh, n, x):
    """Entry column of every cell (nz, ny, nx)."""
    dN = sh.into(n * x) * (sh.sf * sh.dx)
    W = 1.0 / (SIGMA * dN).clamp(min=TAU0)
    Nin, Nout = torch.zeros_like(dN), torch.zeros_like(dN)
    for m in range(max(sh.ext)):
        sh.entry(m, Nout, W, Nin)
        for f in sh.faces(m):
            Nout[f] = Nin[f] + dN[f]
    return sh.back(Nin)


class _Cell:
    """F(x) = sum_s of the photons a cell takes per atom, at neutral fraction x (arrays over cells):
    A_s (P(N_s) - P(N_s + b_s x)), and its secants."""

    def __init__(self, terms, c):
        self.terms, self.c = terms, c            # terms: (A, b, N, spectrum)

    def sub(self, i):
        return _Cell([(A[i], b[i], N[i], sp) for A, b, N, sp in self.terms], self.c[i])

    def diff(self, x, d):
        """(F(x + d) - F(x)) / d, with no cancellation (x, d: (cells, nodes))."""
        out = 0.0
        for A, b, N, sp in self.terms:
            A, b, N = A[:, None], b[:, None], N[:, None]
            if not sp.T:
                z = SIGMA * b * d
                small = z.abs() < 1e-12
                q = torch.where(small, torch.ones_like(z), -torch.expm1(-z) / torch.where(small, torch.ones_like(z), z))
                big = z < -50.0                  # (1 - e^-z) / d from whole exponents
                q1 = torch.exp(-SIGMA * (N + b * x)) * SIGMA * b * torch.where(big, torch.ones_like(z), q)
                q2 = (torch.exp(-SIGMA * (N + b * x)) - torch.exp(-SIGMA * (N + b * (x + d)))) / d
                out = out + A * torch.where(big, q2, q1)
                continue
            N0, N1 = N + b * x, N + b * (x + d)
            L0, L1 = sp.lnP(N0), sp.lnP(N1)
            far = (torch.exp(L0) - torch.exp(L1)) / d
            near = 0.0
            for s, w in _G4:
                near = near + w * sp.slope(N0 + (s * b) * d)
            near = near * b
            out = out + A * torch.where((L0 - L1).abs() > 0.05, far, near)
        return out

    def f(self, x):
        """dx/dt and its slope at x (cells,)."""
        F, S = 0.0, 0.0
        for A, b, N, sp in self.terms:
            if not sp.T:
                e = torch.exp(-SIGMA * N)
                F = F - A * e * torch.expm1(-SIGMA * b * x)
                S = S + A * e * SIGMA * b * torch.exp(-SIGMA * b * x)
            else:
                F = F + A * x * _Cell([(torch.ones_like(A), b, N, sp)], None).diff(
                    torch.zeros_like(x)[:, None], x.clamp(min=1e-30)[:, None])[:, 0]
                S = S + A * b * sp.slope(N + b * x)
        return -F + self.c * (1 - x) ** 2, -S - 2 * self.c * (1 - x)


_G4 = [(0.5 + 0.5 * float(a), 0.5 * float(w)) for a, w in zip(*np.polynomial.legendre.leggauss(6))]
_G8 = np.polynomial.legendre.leggauss(8)
_EDGES = None


def _edges(last=40.0):
    global _EDGES
    if _EDGES is None:
        e, w = [0.0], 2e-4
        while e[-1] > -last:
            e.append(max(-last, e[-1] - w))
            w = min(0.25, 1.25 * w)
        _EDGES = e
    return _EDGES


def _solve(cell, x0, h, b0=None):
    """x(h) of dx/dt = f(x) from x0, and -ln of the mean of exp(-b0 x) over the step if b0 is given.
    With u = ln((x - xe)/(x0 - xe)), xe the root of f, dt = -du/D(u), D the secant slope of f at xe."""
    dev = x0.device
    lit = torch.zeros_like(x0, dtype=torch.bool)
    for A, b, N, sp in cell.terms:
        lit |= A * b * SIGMA * sp.lnP(N).exp() * h > 1e-22
    u0 = 1.0 - x0
    dark = 1.0 - u0 / (1.0 + cell.c * u0 * h)
    x = torch.where(lit, x0, dark)
    lnf = None
    if b0 is not None:
        g = torch.tensor(_G8[0], device=dev)
        w = torch.tensor(_G8[1], device=dev)
        acc = 0.0
        for lo in np.linspace(0.0, 1.0, 17)[:-1]:
            t = h * (lo + (0.5 + 0.5 * g) / 16.0)
            xt = u0[:, None] - u0[:, None] / (1.0 + (cell.c * u0)[:, None] * t)
            acc = acc + (w * torch.exp(-b0[:, None] * xt)).sum(1) / 32.0
        lnf = b0 * x0 - acc.log()
    idx = lit.nonzero()[:, 0]
    for i in idx.split(1 << 21):
        if not len(i):
            continue
        C, xs = cell.sub(i), x0[i]
        xe = torch.zeros_like(xs)
        for _ in range(200):                     # Newton from the left of the root of a convex, falling f
            F, S = C.f(xe)
            new = torch.where(S < 0, xe - F / S, xe).clamp(0.0, 1.0)
            moved = (new - xe).abs().max() > 0
            near = ((new - xe).abs() <= 1e-15 * new).all()
            xe = new
            if near or not moved:
                break
        d0 = xs - xe
        xr, lf = _march(C, xe, d0, h, None if b0 is None else b0[i])
        keep = (d0 == 0)
        x[i] = torch.where(keep, xs, xr)
        if b0 is not None:
            lnf[i] = torch.where(keep, b0[i] * xs, lf)
    return x, lnf


def _march(C, xe, d0, h, b0):
    dev, n = xe.device, len(xe)
    gx, gw = (torch.tensor(v, device=dev) for v in _G8)

    def inv(K, xe_, d0_, u):
        d = d0_[:, None] * torch.exp(u)
        tiny = d.abs() < 1e-290
        D = K.diff(xe_[:, None].expand_as(d), torch.where(tiny, torch.full_like(d, 1e-290), d))
        return 1.0 / (D + K.c[:, None] * (2.0 * (1.0 - xe_[:, None]) - d)), d

    E = _edges()
    ustar = torch.full_like(xe, E[-1])
    T = torch.zeros_like(xe)
    act = torch.arange(n, device=dev)
    K, xa, da, Ta = C, xe, d0, T
    done = torch.zeros(n, dtype=torch.bool, device=dev)
    for hi, lo in zip(E[:-1], E[1:]):
        u = 0.5 * (hi + lo) + 0.5 * (hi - lo) * gx
        v, _ = inv(K, xa, da, u[None, :].expand(len(xa), -1))
        Tn = Ta + 0.5 * (hi - lo) * (v * gw).sum(1)
        hit = (Tn >= h) & ~done
        if bool(hit.any()):
            j = hit.nonzero()[:, 0]
            Kj, xj, dj, rest = K.sub(j), xa[j], da[j], h - Ta[j]
            a, b = torch.full_like(rest, lo), torch.full_like(rest, hi)
            y = hi - (hi - lo) * rest / (Tn[j] - Ta[j])
            for _ in range(60):
                uu = 0.5 * (hi + y)[:, None] + 0.5 * (hi - y)[:, None] * gx
                vv, _ = inv(Kj, xj, dj, uu)
                gq = 0.5 * (hi - y) * (vv * gw).sum(1) - rest
                a, b = torch.where(gq > 0, y, a), torch.where(gq > 0, b, y)
                vy, _ = inv(Kj, xj, dj, y[:, None])
                yn = y + gq / vy[:, 0]
                yn = torch.where((yn >= a) & (yn <= b), yn, 0.5 * (a + b))
                if bool(((yn - y).abs() < 1e-15).all()):
                    break
                y = yn
            ustar[act[j]] = y
            done = done | hit
        Ta = Tn
        if int(done.sum()) * 4 > len(done):
            k = (~done).nonzero()[:, 0]
            if not len(k):
                break
            act, K, xa, da, Ta = act[k], K.sub(k), xa[k], da[k], Ta[k]
            done = torch.zeros(len(k), dtype=torch.bool, device=dev)
    x = xe + d0 * torch.exp(ustar)
    if b0 is None:
        return x, None
    # mean of exp(-b0 x): time spent at each u, panels graded towards both ends of [ustar, 0]
    xmin = torch.minimum(x, xe + d0)
    half, s = [0.0], 1e-6
    while half[-1] < 0.5:
        half.append(min(0.5, half[-1] + s))
        s = min(0.01, 1.3 * s)
    cut = half + [1.0 - q for q in half[-2::-1]]
    S, Tt = torch.zeros_like(x), torch.zeros_like(x)
    for lo, hi in zip(cut[:-1], cut[1:]):
        u = ustar[:, None] * (0.5 * (lo + hi) + 0.5 * (hi - lo) * gx)
        v, d = inv(C, xe, d0, u)
        wt = 0.5 * (hi - lo) * (-ustar)[:, None] * gw * v
        S += (wt * torch.exp(-b0[:, None] * (xe[:, None] + d - xmin[:, None]))).sum(1)
        Tt += wt.sum(1)
    left = (h - Tt).clamp(min=0.0) * (ustar <= E[-1])          # the rest of the step at the root
    S = S + torch.where(left > 0, left * torch.exp(-b0 * (xe - xmin)), torch.zeros_like(S))
    spent = Tt + left                                          # zero where the state hardly moves
    return x, torch.where(spent > 0, b0 * xmin - torch.log(S / spent.clamp(min=1e-300)), b0 * x)


def _plane_columns(q, code):
    axis, back = 2 - code // 2, code & 1
    q = q.flip(axis) if back else q
    c = torch.cumsum(q, axis)
    c = torch.cat([torch.zeros_like(c.narrow(axis, 0, 1)), c.narrow(axis, 0, c.shape[axis] - 1)], axis)
    return c.flip(axis) if back else c


class _Problem:
    def __init__(self, p, nH=None):
        dev = p["x"].device
        nx, ny, nz = p["dims"]
        n = p.get("n")
        self.n = torch.full((nz, ny, nx), 100.0 if nH is None else nH, device=dev, dtype=torch.float64) if n is None \
            else n.double()
        self.dx, self.alpha, self.plane = p["dx"], p.get("alpha", ALPHA), p.get("plane", -1)
        self.srcs = p["srcs"]
        self.sh = [None if s[0] is None else _Shells(s[0], p["dims"], p["dx"]) for s in self.srcs]
        self.sp = [_Spectrum.of(s[3], dev) for s in self.srcs]

    def terms(self, x):
        out = []
        for (v, q, _, T), sh, sp in zip(self.srcs, self.sh, self.sp):
            if v is None:
                N = _plane_columns(self.n * x * self.dx, self.plane)
                A, b = q / (self.n * self.dx), self.n * self.dx
            else:
                N = _columns(sh, self.n, x)
                sf, r2 = (sh.back(w.expand(8, *w.shape)) for w in (sh.sf, sh.r2))
                A = q / (4.0 * math.pi * self.dx ** 3) / (self.n * r2 * sf)
                b = self.n * self.dx * sf
            out.append((A.reshape(-1), b.reshape(-1), N.reshape(-1), sp))
        return out

    def cell(self, terms):
        return _Cell(terms, self.alpha * self.n.reshape(-1))

    def dt(self, x, terms, case):
        f, _ = self.cell(terms).f(x.reshape(-1))
        a, best = f.abs(), math.inf
        if case.get("K1", 0.0) > 0:
            best = min(best, float((case["K1"] / (self.alpha * self.n)).min()))
        if case.get("K3", 0.0) > 0:
            best = min(best, float((case["K3"] * x.reshape(-1).clamp(min=0.05) / a).min()))
        if case["K4"] > 0:
            best = min(best, float((case["K4"] / a).min()))
        return best

    def explicit(self, x, case, fixed):
        t1 = self.terms(x)
        dt = fixed if fixed > 0 else self.dt(x, t1, case)
        if case["scheme"] == A2:
            return _solve(self.cell(t1), x.reshape(-1), dt)[0].view_as(x)
        half = _solve(self.cell(t1), x.reshape(-1), 0.5 * dt)[0].view_as(x)
        return _solve(self.cell(self.terms(half)), x.reshape(-1), dt)[0].view_as(x)

    def implicit(self, x, case, fixed):
        v, q, _, T = self.srcs[0]
        sp = self.sp[0]
        dt = fixed
        if not dt:
            dt = self.dt(x, [], case) if not (case["K3"] > 0 or case["K4"] > 0) else self.dt(x, self.terms(x), case)
        out = torch.empty_like(x)
        if v is None:
            axis, back, L = 2 - self.plane // 2, self.plane & 1, x.shape[2 - self.plane // 2]
            N = torch.zeros_like(x.select(axis, 0)).reshape(-1)
            for m in range(L):
                k = L - 1 - m if back else m
                n, xs = self.n.select(axis, k).reshape(-1), x.select(axis, k).reshape(-1)
                b = n * self.dx
                xn, lf = _solve(_Cell([(q / b, b, N, sp)], self.alpha * n), xs, dt, SIGMA * b)
                out.select(axis, k).copy_(xn.view_as(out.select(axis, k)))
                N = N + lf.clamp(min=0.0) / SIGMA
            return out
        sh = self.sh[0]
        n8, x8 = sh.into(self.n), sh.into(x)
        W, Nin, Nout = torch.zeros_like(n8), torch.zeros_like(n8), torch.zeros_like(n8)
        sf, r2 = sh.sf.expand_as(n8), sh.r2.expand_as(n8)
        for m in range(max(sh.ext)):
            sh.entry(m, Nout, W, Nin)
            for f in sh.faces(m):
                ok = n8[f] > 0
                n, xs, N = n8[f][ok], x8[f][ok], Nin[f][ok]
                if not len(n):
                    continue
                b = n * self.dx * sf[f][ok]
                A = q / (4.0 * math.pi * self.dx ** 3) / (n * r2[f][ok] * sf[f][ok])
                xn, lf = _solve(_Cell([(A, b, N, sp)], self.alpha * n), xs, dt, SIGMA * b)
                lf = lf.clamp(min=0.0)
                for dst, val in ((x8, xn), (Nout, N + lf / SIGMA), (W, 1.0 / lf.clamp(min=TAU0))):
                    view = dst[f]
                    view[ok] = val
                    dst[f] = view
        return sh.back(x8)


def _affordable(case):
    """About what the 64-bit pass takes, in seconds."""
    if case["kind"] == "trace":
        return 1.0
    if case["kind"] == "batch":
        return 0.25 * case["count"]
    cells = case["nx"] * case["ny"] * case["nz"]
    stages = 2 if case["scheme"] == A3 else 1
    if case["scheme"] == A1:
        return 0.12 * max(case["nx"], case["ny"], case["nz"]) if case["plane"] < 0 else 0.05 * max(case["nx"], case["ny"], case["nz"])
    per = (3e-7 if case["spectrum"] != "mono" else 8e-8) * cells * case["nsrc"] + 0.1
    return per * stages * case["steps"]


def exact(case, seed):
    if _affordable(case) > 18.0:
        return None
    if case["kind"] == "trace":
        p = _inputs(case, seed)
        return {"column": _columns(_Shells(p["srcs"][0][0], p["dims"], p["dx"]), p["n"], p["x"].double())}
    if case["kind"] == "batch":
        return {"x": [_Problem(p, p["nH"]).explicit(p["x"].double(), case, 0.0) for p in _batch_inputs(case, seed)]}
    p = _inputs(case, seed)
    P, x = _Problem(p), p["x"].double()
    for _ in range(case["steps"]):
        fixed = case["dt_trec"] * p["trec"]
        x = P.implicit(x, case, fixed) if case["scheme"] == A1 else P.explicit(x, case, fixed)
    return {"x": x}
