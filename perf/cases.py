"""The work that a user of the library has it do, as cases that can be timed.

A case is one call (or the few calls that always go together) of the public entry points on
a cluster of the kind that paper_1603_04334_gb300.synth describes: a uniform grid with
radius-6 stencil, V_eff of erf-screened charges, s + p projectors truncated at 3 bohr, and a
block of orbitals. `listed()` gives fixed cases over the real range of sizes, `draw(rng)` more
of the same ranges; `prepare` makes what a program holds before the call, `run` makes the call
and returns its results, `work` counts the bytes and flops that the call cannot do without, and
`exact` computes the same results in 64 bits with plain torch.

Calls that overwrite their block (the filter, Rayleigh-Ritz and a CheFSI iteration) run on a
copy of the prepared block, made inside `run`, so that every pass sees the same kind of input.
"""
import math
import random

import numpy as np
import torch

from paper_1603_04334_gb300 import batching, sparc

RADIUS = 6
SIGMA, RCUT, RC_ERF = 0.8, 3.0, 1.0  # the library's defaults, written out for exact()


# ---- the cases -------------------------------------------------------------------------
def _case(kind, n, h, atoms, ncols, dtype, degree=0):
    return {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "h": h, "atoms": atoms,
            "ncols": ncols, "dtype": dtype, "degree": degree}


def listed():
    def named(name, *a, **k):
        return {"name": name, **_case(*a, **k)}

    c = []
    # H X of the smallest preset (24^3, 12 states): five short launches, all latency
    c.append(named("apply_f64_24", "apply", (24, 24, 24), 0.5, 4, 12, "f64"))
    # the spectral bounds that every solve starts with: 10 Lanczos steps on one vector
    c.append(named("bounds_64", "bounds", (64, 64, 64), 0.3, 20, 1, "f64"))
    # a filter on a grid that no tile divides, with an odd number of states
    c.append(named("filter_f64_ragged", "filter", (70, 61, 53), 0.3, 12, 33, "f64", 10))
    # the filter of the medium FP64 preset (96^3, 128 states, degree 20): the main work of a solve
    c.append(named("filter_f64_96", "filter", (96, 96, 96), 0.3, 40, 128, "f64", 20))
    # the FP32 filter where rows are not a multiple of 16 bytes
    c.append(named("filter_f32_ragged", "filter", (75, 61, 53), 0.3, 12, 40, "f32", 16))
    # the FP32 filter of the large preset (160^3, 400 atoms, degree 24), a quarter of its states
    c.append(named("filter_f32_160", "filter", (160, 160, 160), 0.25, 400, 256, "f32", 24))
    # many small clusters per launch, as the batched server runs them
    c.append(named("batch_f32_12", "batch", (32, 40, 48), 0.3, 30, 12, "f32", 16))
    # one whole iteration of the smallest preset: filter, Rayleigh-Ritz, new interval
    c.append(named("chefsi_f64_24", "chefsi", (24, 24, 24), 0.5, 4, 12, "f64", 10))
    # Rayleigh-Ritz of the medium preset (128 states)
    c.append(named("rr_f64_96", "rr", (96, 96, 96), 0.3, 40, 128, "f64"))
    # Rayleigh-Ritz of the largest request that is served (128^3, 512 states, mixed form)
    c.append(named("rr_f32_128", "rr", (128, 128, 128), 0.3, 100, 512, "f32"))
    # after the rotation: occupations, density and non-local force of the medium preset
    c.append(named("observables_f64_96", "observables", (96, 96, 96), 0.3, 40, 128, "f64"))
    # the electrostatic potential of a medium cluster's density
    c.append(named("poisson_64", "poisson", (64, 64, 64), 0.3, 20, 1, "f64"))
    return c


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["apply", "filter", "filter", "filter", "rr", "rr", "chefsi", "bounds",
                       "observables", "poisson", "batch"])
    h = rng.choice([0.25, 0.3, 0.4, 0.5])
    if kind == "batch":
        edges = sorted(rng.choice([32, 40, 48, 56, 64]) for _ in range(3))
        return _case(kind, edges, 0.3, rng.randint(2, 60), rng.randint(4, 12), "f32",
                     rng.randint(8, 16))
    dtype = rng.choice(["f64", "f64", "f32"]) if kind in ("apply", "filter", "rr",
                                                         "observables") else "f64"
    top = 96 if dtype == "f64" else 128 if kind == "rr" else 160
    n = _log(rng, 24, top)
    # half of the grids are cubes, as in the presets; the others have three ragged edges
    n = (n, n, n) if rng.random() < 0.5 else tuple(
        max(20, min(top, n + rng.randint(-9, 9))) for _ in range(3))
    nd = n[0] * n[1] * n[2]
    inner = max(0.0, (min(n) - 1) * h - 8.0)
    atoms = min(rng.randint(1, 60), int(1 + (inner / 3.0) ** 3))
    few = kind in ("apply", "filter", "observables")
    ncols = _log(rng, 1, 256) if few else _log(rng, 8, 160 if dtype == "f64" else 512)
    degree = rng.randint(4, 24) if kind in ("filter", "chefsi") else 0
    # point-orbitals of a pass: no more than those of the listed cases of the kind
    most = {"filter": 2.2e9 if dtype == "f64" else 2.5e10, "chefsi": 1.0e9}.get(
        kind, 1.1e8 if dtype == "f64" else 1.0e9)
    ncols = max(1 if few else 8, min(ncols, int(most / (nd * max(1, degree)))))
    if kind in ("bounds", "poisson"):
        ncols = 1
        if kind == "poisson":
            n = tuple(min(v, 72) for v in n)
    return _case(kind, n, h, atoms, ncols, dtype, degree)


# ---- inputs ------------------------------------------------------------------------------
def _atoms(n, h, count, seed):
    """Positions at least 2 bohr apart and 4 bohr from the walls (less in small boxes), charges
    1..4, and coefficients uniform in [-2, 2] (one for s, one for the three p)."""
    g = np.random.default_rng(seed)
    L = [(v - 1) * h for v in n]
    margin = [min(4.0, 0.35 * v) for v in L]
    lo, hi = np.array(margin), np.array([v - m for v, m in zip(L, margin)])
    R = np.zeros((0, 3))
    while R.shape[0] < count:
        c = g.uniform(lo, hi, size=(512, 3))
        d = ((c[:, None, :] - R[None, :, :]) ** 2).sum(-1)
        ok = np.nonzero((d >= 4.0).all(1))[0] if R.shape[0] else np.arange(512)
        if ok.size == 0:
            break  # the box is full
        R = np.vstack([R, c[ok[0]]])
    k = R.shape[0]
    Z = g.integers(1, 5, size=k).astype(np.float64)
    gl = g.uniform(-2.0, 2.0, size=(k, 2))
    gamma = np.column_stack([gl[:, 0], gl[:, 1], gl[:, 1], gl[:, 1]]) if k else np.zeros((0, 4))
    return np.ascontiguousarray(R), Z, np.ascontiguousarray(gamma)


def _dims(case):
    return case["nx"], case["ny"], case["nz"]


def _dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.float64


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _random_block(n, ncols, seed, dtype):
    """A start block: uniform in (-0.5, 0.5)."""
    nd = n[0] * n[1] * n[2]
    X = torch.empty((ncols, nd), dtype=dtype, device="cuda")
    return X.uniform_(-0.5, 0.5, generator=_gen(seed))


def _smooth_block(n, ncols, seed, dtype):
    """A block like a filtered one: random combinations of the box's low sine modes, weights
    falling with the mode's kinetic energy."""
    g = _gen(seed)
    m = 2
    while m ** 3 < 4 * ncols and m < min(n) // 2:
        m += 1
    modes, sines = [], []
    for v in n:
        k = torch.arange(1, m + 1, dtype=torch.float64, device="cuda")
        x = torch.arange(1, v + 1, dtype=torch.float64, device="cuda") / (v + 1)
        modes.append(k)
        sines.append(torch.sin(math.pi * k[:, None] * x[None, :]) * math.sqrt(2.0 / (v + 1)))
    e = (modes[2][:, None, None] ** 2 + modes[1][None, :, None] ** 2
         + modes[0][None, None, :] ** 2) / (3.0 * m * m)
    X = torch.empty((ncols, n[0] * n[1] * n[2]), dtype=dtype, device="cuda")
    for c in range(0, ncols, 64):
        k = min(64, ncols - c)
        a = torch.randn((k, m, m, m), dtype=torch.float64, device="cuda", generator=g)
        a = a / (1.0 + 3.0 * e)
        a = torch.matmul(a, sines[0])                                          # k, z, y, x
        a = torch.matmul(a.transpose(2, 3), sines[1]).transpose(2, 3)
        a = torch.matmul(a.permute(0, 2, 3, 1), sines[2]).permute(0, 3, 1, 2)
        X[c:c + k] = a.reshape(k, -1).to(dtype)
    return X


def _outward(lo, hi):
    """The filter interval a, b, a0 from the spectral bounds, rounded outward to sixteenths:
    the cutoff a quarter of the way up, as in a first iteration."""
    a0, b = math.floor(16.0 * lo) / 16.0, math.ceil(16.0 * hi) / 16.0
    return a0 + 0.25 * (b - a0), b, a0


def _batch_members(case):
    """(n, atoms, states) of each cluster of a batch: edges in turn, 16 to 160 states."""
    g = np.random.default_rng([case["atoms"], case["ncols"]])
    out = []
    for i in range(case["ncols"]):
        v = _dims(case)[i % 3]
        out.append(((v, v, v), int(g.integers(2, case["atoms"] + 1)), int(g.integers(16, 161))))
    return out


def _context(n, h, atoms, seed):
    R, Z, gamma = _atoms(n, h, atoms, seed)
    return sparc.Context(n, h, R, Z, gamma)


def _levels(ncols, seed):
    g = np.random.default_rng([seed, 7])
    # about 55 per cent of the levels filled, the topmost one in part
    return np.sort(g.uniform(-1.0, 0.5, ncols)), 2.0 * (int(0.55 * ncols) + 0.37)


def _density(n, h, R, Z):
    """Electrons: a Gaussian cloud of Z_J electrons around each atom."""
    x = [torch.arange(v, dtype=torch.float64, device="cuda") * h for v in n]
    rho = torch.zeros((n[2], n[1], n[0]), dtype=torch.float64, device="cuda")
    w = 1.2
    for (rx, ry, rz), z in zip(R.tolist(), Z.tolist()):
        f = [torch.exp(-((t - r) / w) ** 2) for t, r in zip(x, (rx, ry, rz))]
        rho += z / (math.pi ** 1.5 * w ** 3) * (f[2][:, None, None] * f[1][None, :, None]
                                                * f[0][None, None, :])
    return rho.reshape(-1)


def prepare(case, seed):
    n, h, kind = _dims(case), case["h"], case["kind"]
    s = {"kind": kind, "degree": case["degree"]}
    if kind == "batch":
        s["ctx"], s["X0"], s["bounds"] = [], [], []
        for i, (m, atoms, ns) in enumerate(_batch_members(case)):
            ctx = _context(m, h, atoms, [seed, i])
            s["ctx"].append(ctx)
            s["X0"].append(_random_block(m, ns, 1000 * seed + i, torch.float32))
            s["bounds"].append(_outward(*ctx.lanczos_bounds(10, 0)))
        s["X"] = [torch.empty_like(x) for x in s["X0"]]
        s["W"] = [torch.empty_like(x) for x in s["X0"]]
        s["batch"] = batching.Batch(s["ctx"])
        return s
    ctx = s["ctx"] = _context(n, h, case["atoms"], seed)
    if kind == "bounds":
        s["seed"] = seed
        return s
    if kind == "poisson":
        R, Z, _ = _atoms(n, h, case["atoms"], seed)
        s["rho"] = _density(n, h, R, Z)
        s["phi"] = torch.empty_like(s["rho"])
        return s
    make = _smooth_block if kind in ("rr", "observables") else _random_block
    s["X0"] = make(n, case["ncols"], seed, _dtype(case))
    s["X"] = torch.empty_like(s["X0"])
    if kind == "observables":
        s["X0"] /= s["X0"].norm(dim=1, keepdim=True)
        s["lam"], s["nelec"] = _levels(case["ncols"], seed)
        s["rho"] = torch.empty(s["X0"].shape[1], dtype=torch.float64, device="cuda")
    if kind in ("filter", "chefsi"):
        s["W"] = torch.empty_like(s["X0"])
        s["bounds"] = _outward(*ctx.lanczos_bounds(10, 0))
    return s


# ---- one pass ------------------------------------------------------------------------------
def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "apply":
        ctx.apply_H(s["X0"], s["X"])
        return s["X"]
    if kind == "bounds":
        return ctx.first_bounds(10, s["seed"])
    if kind == "filter":
        s["X"].copy_(s["X0"])
        ctx.cheb_filter(s["X"], s["W"], s["degree"], *s["bounds"])
        return s["X"]
    if kind == "batch":
        for x, x0 in zip(s["X"], s["X0"]):
            x.copy_(x0)
        s["batch"].filter(s["X"], s["W"], s["degree"], s["bounds"])
        return s["X"]
    if kind == "rr":
        s["X"].copy_(s["X0"])
        ritz, resid = ctx.orth_rr(s["X"])
        return {"X": s["X"], "ritz": ritz, "resid": resid}
    if kind == "chefsi":
        s["X"].copy_(s["X0"])
        ritz, resid, bounds = ctx.chefsi_step(s["X"], s["W"], s["degree"], s["bounds"])
        return {"X": s["X"], "ritz": ritz, "resid": resid, "bounds": bounds}
    if kind == "observables":
        mu, g = ctx.occupations(s["lam"], s["nelec"])
        rho = ctx.density(s["X0"], g, s["rho"])
        return {"mu": mu, "g": g, "rho": rho, "force": ctx.nonlocal_force(s["X0"], g)}
    # the tolerance of the library's accuracy tests; the solver's iteration count and its final
    # residual are reports on how it got there, not results
    phi, _, _, b = ctx.poisson(s["rho"], s["phi"], tol=1e-12, want_b=True)
    return {"phi": phi, "b": b}


# ---- what a pass cannot do without ----------------------------------------------------------
def _support(h, atoms):
    return atoms * 4.0 / 3.0 * math.pi * (RCUT / h) ** 3


def work(case):
    """Bytes: inputs read once, outputs written once. Flops: 47 per point-orbital and
    application of H for stencil, potential and recurrence, 16 per (support entry, orbital)
    for the projectors; 2 K M N for the contractions."""
    n, h, kind, nc = _dims(case), case["h"], case["kind"], case["ncols"]
    nd, e = n[0] * n[1] * n[2], 4 if case["dtype"] == "f32" else 8

    def h_flops(nd, atoms, nc):
        return nc * (47.0 * nd + 16.0 * _support(h, atoms))

    if kind == "batch":
        b = f = 0.0
        for m, atoms, ns in _batch_members(case):
            b += 4.0 * m[0] ** 3 * (2 * ns + 1)
            f += case["degree"] * h_flops(m[0] ** 3, atoms, ns)
        return {"bytes": b, "flops": f}
    block = float(e) * nd * nc
    hx = h_flops(nd, case["atoms"], nc)
    if kind == "apply":
        return {"bytes": 2 * block + e * nd, "flops": hx}
    if kind == "bounds":
        return {"bytes": 8.0 * nd, "flops": 10 * (hx + 10.0 * nd)}
    if kind == "filter":
        return {"bytes": 2 * block + e * nd, "flops": case["degree"] * hx}
    # M_s, H_s (symmetric), X Q and H X Q
    dense = 6.0 * nd * nc * nc + 10.0 * nc ** 3
    if kind == "rr":
        return {"bytes": 2 * block + 8.0 * nd, "flops": hx + dense}
    if kind == "chefsi":
        return {"bytes": 2 * block + 8.0 * nd, "flops": (case["degree"] + 1) * hx + dense}
    if kind == "observables":
        return {"bytes": block + 8.0 * nd,
                "flops": 3.0 * nd * nc + 104.0 * _support(h, case["atoms"]) * nc}
    # Poisson: at least the sweep of a direct solve, one pass per dimension and back
    return {"bytes": 3 * 8.0 * nd, "flops": 4.0 * nd * sum(n)}


# ---- the same results in 64 bits, with torch -----------------------------------------------
def _weights():
    w = [-2.0 * sum(1.0 / q ** 2 for q in range(1, RADIUS + 1))]  # one dimension's centre
    for p in range(1, RADIUS + 1):
        r = math.factorial(RADIUS) ** 2 / (math.factorial(RADIUS - p) * math.factorial(RADIUS + p))
        w.append(2.0 * (-1.0) ** (p + 1) / p ** 2 * r)
    return w  # times 1 / h^2


def _shifted_sum(Y, p, dim):
    """Y(. + p) + Y(. - p) along dim, zero outside the grid."""
    out = torch.zeros_like(Y)
    v = Y.shape[dim]
    if p < v:
        out.narrow(dim, 0, v - p).add_(Y.narrow(dim, p, v - p))
        out.narrow(dim, p, v - p).add_(Y.narrow(dim, 0, v - p))
    return out


def _erf_potential(xyz, R, Z):
    V = torch.zeros(xyz[0].numel() * xyz[1].numel() * xyz[2].numel(), dtype=torch.float64,
                    device=xyz[0].device).reshape(xyz[2].numel(), xyz[1].numel(), -1)
    for r, z in zip(R.tolist(), Z.tolist()):
        d = ((xyz[2] - r[2]) ** 2)[:, None, None] + ((xyz[1] - r[1]) ** 2)[None, :, None] \
            + ((xyz[0] - r[0]) ** 2)[None, None, :]
        d = d.sqrt()
        V -= z * torch.where(d > 1e-12, torch.erf(d / RC_ERF) / d.clamp_min(1e-300),
                             torch.full_like(d, 2.0 / (math.sqrt(math.pi) * RC_ERF)))
    return V


class _Exact:
    """H of one cluster on blocks of shape (columns, nz, ny, nx)."""

    def __init__(self, n, h, R, Z, gamma):
        self.n, self.h, self.gamma = n, h, gamma
        self.shape = (n[2], n[1], n[0])
        self.w = [v / h ** 2 for v in _weights()]
        x = [torch.arange(v, dtype=torch.float64, device="cuda") * h for v in n]
        self.V = _erf_potential(x, R, Z)
        self.atoms = []
        for r in R.tolist():
            dx, dy, dz = x[0] - r[0], x[1] - r[1], x[2] - r[2]
            d2 = ((dx ** 2)[None, None, :] + (dy ** 2)[None, :, None]) + (dz ** 2)[:, None, None]
            idx = torch.nonzero(d2.reshape(-1) <= RCUT * RCUT).reshape(-1)
            k, j, i = idx // (n[0] * n[1]), idx // n[0] % n[1], idx % n[0]
            e = torch.exp(-d2.reshape(-1)[idx] / (2.0 * SIGMA ** 2))
            p = math.sqrt(0.75 / math.pi) * e
            chi = torch.stack([math.sqrt(0.25 / math.pi) * e, p * dx[i], p * dy[j], p * dz[k]], 1)
            self.atoms.append((idx, chi))

    def apply(self, Y, out=None):
        out = torch.empty_like(Y) if out is None else out
        step = max(1, int(2.5e8 / self.V.numel()))  # columns at a time: temporaries of 2 GB
        for c in range(0, Y.shape[0], step):
            y = Y[c:c + step].reshape(-1, *self.shape)
            o = y * (self.V - 1.5 * self.w[0])
            for p in range(1, RADIUS + 1):
                t = _shifted_sum(y, p, 1)
                t += _shifted_sum(y, p, 2)
                t += _shifted_sum(y, p, 3)
                o.add_(t, alpha=-0.5 * self.w[p])
            o, y = o.reshape(o.shape[0], -1), y.reshape(o.shape[0], -1)
            for (idx, chi), g in zip(self.atoms, self.gamma):
                C = y[:, idx] @ chi * (self.h ** 3 * torch.as_tensor(g, device=y.device))
                o[:, idx] += C @ chi.T
            out[c:c + step] = o.reshape(out[c:c + step].shape)
        return out

    def bounds(self, steps, seed):
        """Lanczos from the library's start vector: SplitMix64 of (seed xor node)."""
        nd = self.V.numel()
        z = np.arange(nd, dtype=np.uint64) ^ np.uint64(seed)
        with np.errstate(over="ignore"):
            z = z + np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z = z ^ (z >> np.uint64(31))
        v = (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53 - 0.5
        v = torch.from_numpy(v).to("cuda").reshape(1, -1)
        v = v / v.norm()
        vp, beta, al, be = torch.zeros_like(v), 0.0, [], []
        for _ in range(steps):
            w = self.apply(v)
            al.append(float((w * v).sum()))
            w = w - al[-1] * v - beta * vp
            beta = float(w.norm())
            be.append(beta)
            vp, v = v, w / beta
        T = np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1)
        ev, Q = np.linalg.eigh(T)
        return float(ev[0]), float(max(1.01 * ev[-1], ev[-1] + abs(be[-1] * Q[-1, -1])))

    def filter(self, X, degree, a, b, a0):
        e, c = (b - a) / 2.0, (b + a) / 2.0
        out = torch.empty(X.shape, dtype=torch.float64, device="cuda")
        for q in range(0, X.shape[0], 64):
            y0 = X[q:q + 64].double()
            s1 = sigma = e / (a0 - c)
            y1 = (self.apply(y0) - c * y0) * (s1 / e)
            for _ in range(2, degree + 1):
                sn = 1.0 / (2.0 / s1 - sigma)
                y2 = self.apply(y1)
                y2.add_(y1, alpha=-c).mul_(2.0 * sn / e).add_(y0, alpha=-sigma * sn)
                y0, y1, sigma = y1, y2, sn
            out[q:q + 64] = y1
        return out

    def rayleigh_ritz(self, Y):
        HY = self.apply(Y)
        L = torch.linalg.cholesky(Y @ Y.T)
        Hs = Y @ HY.T
        A = torch.linalg.solve_triangular(L, 0.5 * (Hs + Hs.T), upper=False)
        A = torch.linalg.solve_triangular(L, A.T.contiguous(), upper=False)
        ritz, Q = torch.linalg.eigh(0.5 * (A + A.T))
        at = Q.abs().argmax(dim=0, keepdim=True)
        Q = Q * torch.sign(Q.gather(0, at))
        C = torch.linalg.solve_triangular(L.T.contiguous(), Q, upper=True)
        X = C.T @ Y
        return X, ritz, (C.T @ HY - ritz[:, None] * X).norm(dim=1)


def _force(H, X, g):
    """f_J = -(4 / h^3) sum_n g_n sum_l gamma_Jl Y_l W_l with Y = h^3 sum x chi, W = h^3 sum
    (grad x) chi over the support."""
    n, h = H.n, H.h
    wg = [0.0] + [(-1.0) ** (p + 1) / (h * p) * math.factorial(RADIUS) ** 2
                  / (math.factorial(RADIUS - p) * math.factorial(RADIUS + p))
                  for p in range(1, RADIUS + 1)]
    f = torch.zeros((len(H.atoms), 3), dtype=torch.float64, device="cuda")
    gam = torch.as_tensor(H.gamma, device="cuda")
    for c in range(0, X.shape[0], 16):
        x = X[c:c + 16].reshape(-1, *H.shape)
        gr = []
        for dim, v in ((3, n[0]), (2, n[1]), (1, n[2])):
            o = torch.zeros_like(x)
            for p in range(1, min(RADIUS, v - 1) + 1):
                o.narrow(dim, 0, v - p).add_(x.narrow(dim, p, v - p), alpha=wg[p])
                o.narrow(dim, p, v - p).add_(x.narrow(dim, 0, v - p), alpha=-wg[p])
            gr.append(o.reshape(o.shape[0], -1))
        x = x.reshape(x.shape[0], -1)
        for J, (idx, chi) in enumerate(H.atoms):
            y = x[:, idx] @ chi * g[c:c + 16, None] * gam[J]
            for d in range(3):
                f[J, d] += (y * (gr[d][:, idx] @ chi)).sum()
    return -4.0 * h ** 3 * f


def _harmonics(x, y, z):
    """Real solid harmonics, l <= 6, orthonormal on the unit sphere: {(l, m): values}."""
    r2 = x * x + y * y + z * z
    A, B, out = torch.ones_like(x), torch.zeros_like(x), {}
    for m in range(7):
        if m:
            A, B = A * x - B * y, A * y + B * x
        P = {m: torch.full_like(x, float(np.prod(np.arange(1, 2 * m, 2))) if m else 1.0)}
        for l in range(m + 1, 7):
            P[l] = (2 * l - 1) * z * P[l - 1]
            if l > m + 1:
                P[l] = P[l] - (l + m - 1) * r2 * P[l - 2]
            P[l] = P[l] / (l - m)
        for l in range(m, 7):
            N = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m)
                          * (2 if m else 1))
            out[l, m] = N * P[l] * A
            if m:
                out[l, -m] = N * P[l] * B
    return out


def _poisson(n, h, R, Z, rho):
    """phi and the pseudocharges: the multipole boundary values enter the right-hand side,
    and the separable operator is inverted in the eigenvectors of its three factors."""
    w = [v / h ** 2 for v in _weights()]
    shape = (n[2], n[1], n[0])
    P = RADIUS
    xe = [(torch.arange(v + 2 * P, dtype=torch.float64, device="cuda") - P) * h for v in n]
    Ve = _erf_potential(xe, R, Z)
    core = [slice(P, P + v) for v in shape]

    def laplacian(F):
        out = 3.0 * w[0] * F[core[0], core[1], core[2]]
        for p in range(1, P + 1):
            for dim in range(3):
                for s in (-p, p):
                    at = list(core)
                    at[dim] = slice(P + s, P + s + shape[dim])
                    out = out + w[p] * F[at[0], at[1], at[2]]
        return out

    b = -laplacian(Ve) / (4.0 * math.pi)
    total = b + rho.reshape(shape)
    c = [0.5 * (v - 1) * h for v in n]
    Xg, Yg, Zg = (xe[0] - c[0])[None, None, :], (xe[1] - c[1])[None, :, None], (xe[2] - c[2])[:, None, None]
    X, Y, Zz = (t.expand(*[v + 2 * P for v in shape]).contiguous() for t in (Xg, Yg, Zg))
    S = _harmonics(X, Y, Zz)
    r = (X * X + Y * Y + Zz * Zz).sqrt()
    ext = torch.zeros_like(r)
    for (l, m), v in S.items():
        q = h ** 3 * (total * v[core[0], core[1], core[2]]).sum()
        ext += 4.0 * math.pi / (2 * l + 1) * q * v / r.clamp_min(1e-300) ** (2 * l + 1)
    ext[core[0], core[1], core[2]] = 0.0
    rhs = total + laplacian(ext) / (4.0 * math.pi)
    vec, val = [], []
    for v in n:
        i = torch.arange(v, device="cuda")
        d = (i[:, None] - i[None, :]).abs()
        T = torch.zeros((v, v), dtype=torch.float64, device="cuda")
        for p in range(P + 1):
            T[d == p] = w[p]
        a, q = torch.linalg.eigh(-T / (4.0 * math.pi))
        val.append(a)
        vec.append(q)
    t = torch.einsum("zyx,xa,yb,zc->cba", rhs, *vec)
    t = t / (val[2][:, None, None] + val[1][None, :, None] + val[0][None, None, :])
    return torch.einsum("cba,xa,yb,zc->zyx", t, *vec).reshape(-1), b.reshape(-1)


def exact(case, seed):
    n, h, kind = _dims(case), case["h"], case["kind"]
    if kind == "batch":
        out = []
        for i, (m, atoms, ns) in enumerate(_batch_members(case)):
            H = _Exact(m, h, *_atoms(m, h, atoms, [seed, i]))
            X = _random_block(m, ns, 1000 * seed + i, torch.float32)
            out.append(H.filter(X, case["degree"], *_outward(*H.bounds(10, 0))))
        return out
    R, Z, gamma = _atoms(n, h, case["atoms"], seed)
    if kind == "poisson":
        phi, b = _poisson(n, h, R, Z, _density(n, h, R, Z))
        return {"phi": phi, "b": b}
    H = _Exact(n, h, R, Z, gamma)
    if kind == "bounds":
        lo, hi = H.bounds(10, seed)
        return [lo + 0.25 * (hi - lo), hi, lo]
    if kind in ("rr", "observables"):
        X = _smooth_block(n, case["ncols"], seed, _dtype(case))
        if kind == "observables":
            X /= X.norm(dim=1, keepdim=True)
        X = X.double()
    else:
        X = _random_block(n, case["ncols"], seed, _dtype(case)).double()
    if kind == "apply":
        return H.apply(X)
    if kind == "observables":
        lam, nelec = _levels(case["ncols"], seed)
        lo, hi = lam[0] - 1.0, lam[-1] + 1.0
        for _ in range(200):
            mu = 0.5 * (lo + hi)
            g = 1.0 / (1.0 + np.exp(np.clip((lam - mu) / 1e-3, -700.0, 700.0)))
            lo, hi = (mu, hi) if 2.0 * g.sum() < nelec else (lo, mu)
        gt = torch.from_numpy(g).to("cuda")
        rho = torch.zeros(X.shape[1], dtype=torch.float64, device="cuda")
        for c in range(X.shape[0]):
            rho += g[c] * X[c] ** 2
        return {"mu": float(mu), "g": g, "rho": 2.0 / h ** 3 * rho, "force": _force(H, X, gt)}
    if kind in ("filter", "chefsi"):
        a, b, a0 = _outward(*H.bounds(10, 0))
        X = H.filter(X, case["degree"], a, b, a0)
        if kind == "filter":
            return X
    X, ritz, resid = H.rayleigh_ritz(X)
    out = {"X": X, "ritz": ritz, "resid": resid}
    if kind == "chefsi":
        out["bounds"] = [float(ritz[-1]), b, float(ritz[0])]
    return out
