"""The calls whose speed matters to a user of the library, as measurable cases.

A case describes one ensemble (lattice, coupling, precision, system sizes,
Landau coefficients, relaxation times, sampling schedule) and one pass over it:
advance the ensemble by ``steps`` time steps and read what the run is for (the
block observables, the structure factor, the momentum spectra, the histograms,
a snapshot of the first system's populations).  ``listed`` holds the workloads
themselves, ``draw`` gives others of the same ranges, ``exact`` the same
outputs from a plain FP64 torch implementation of the method.

Outputs of a float32 run are handed over as float32 (the populations are
float32; their FP64 sums carry the accuracy of that storage); a float64 run
hands over float64.
"""
import math

import numpy as np
import torch

import paper_1202_4748_gb300 as lb


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def case(name=None, **kw):
    """One case; ``sides`` is a comma-separated list of system sizes XxYxZ.
    Every size runs ``n_a`` values of a in [a0, a1] with ``replicas`` seeds."""
    c = dict(lattice="D3Q19", coupling="guo", precision="fp32", sides="64x64x64", n_a=1, a0=0.0, a1=0.0,
             replicas=1, b=0.1, kappa=0.01, kT=1e-4, tau="one", steps=100, obs=100, sk=0, jk=False, hist=0,
             chunk=100, field=True)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def cubes(*sides):
    return ",".join("%dx%dx%d" % (n, n, n) for n in sides)


def squares(*sides):
    return ",".join("%dx%dx1" % (n, n) for n in sides)


def listed():
    fss = dict(n_a=8, a0=-0.004, a1=0.004, replicas=4)
    return [
        # The smallest call: one 16^3 system at the critical point, sampled every
        # 10 steps; launches and latency count, the device is nearly idle.
        case("single_16", sides=cubes(16), steps=1000, obs=10),
        # One 64^3 system just below the critical point, sampled every 100 steps
        # with its structure factor: an ordinary single run.
        case("single_64", sides=cubes(64), a0=-0.002, a1=-0.002, steps=400, sk=100, field=False),
        # The finite-size-scaling ensemble of 160 systems, one sampling interval:
        # the production run of the library.
        case("fss_160", sides=cubes(16, 24, 32, 48, 64), **fss),
        # The same on the paper's own lattice and coupling.
        case("fss_160_d2q9", lattice="D2Q9", coupling="modeq", sides=squares(64, 120, 184, 336, 512), **fss),
        # The same with the paper's coupling carried to three dimensions.
        case("fss_160_modeq", coupling="modeq", sides=cubes(16, 24, 32, 48, 64), **fss),
        # The largest single lattice, the bandwidth case.
        case("large_256", sides=cubes(256), field=False),
        # Statics of the Guo form at the paper's 2-D parameters: 16 replicas of
        # 64^2, structure factor and momentum spectra every 20 steps.
        case("statics_2d", lattice="D2Q9", sides=squares(64), a0=1e-3, a1=1e-3, replicas=16, b=2.8e-2, kappa=9.6e-5,
             kT=1e-7, steps=1000, obs=0, sk=20, jk=True, field=False),
        # The 3-D comparison of the couplings: 8 replicas of 32^3, the modified
        # equilibrium, spectra every 20 steps.
        case("statics_3d", coupling="modeq", sides=cubes(32), a0=1e-2, a1=1e-2, replicas=8, b=2.8e-2, kappa=1e-3,
             kT=1e-6, steps=1000, obs=0, sk=20, jk=True, field=False),
        # The accuracy study's FP64 arm: the 16^3 and 24^3 members of the
        # ensemble in FP64, sampled every 10 steps.
        case("fss_fp64", precision="fp64", sides=cubes(16, 24), steps=50, obs=10, sk=50, chunk=0, **fss),
        # FP64 on the paper's lattice with order-parameter histograms: one 512^2
        # system below the critical point.
        case("histogram_fp64", lattice="D2Q9", coupling="modeq", precision="fp64", sides=squares(512), a0=-0.002,
             a1=-0.002, steps=100, obs=10, hist=512, chunk=0),
        # Sides of no convenient factor (odd, ragged against any tile), as a user
        # who sizes the box by the physics has them.
        case("odd_sides", sides="45x50x37,61x33x70,27x27x27,99x20x41", n_a=2, a0=-0.002, a1=0.002, replicas=4,
             steps=100, obs=50),
        # Transport study: a separate bulk rate, so every mode relaxes at its own.
        case("mode_rates", sides=cubes(64), a0=0.1, a1=0.1, replicas=4, tau="modes", steps=100, obs=50),
    ]


def draw(rng):
    """One more case: any lattice, coupling, precision and relaxation setting,
    sizes spread over the range of the listed ones, odd sides among them."""
    lattice = rng.choice(["D3Q19", "D3Q19", "D2Q9"])
    coupling = rng.choice(["guo", "modeq"])
    precision = "fp64" if rng.random() < 0.3 else "fp32"
    tau = rng.choice(["one", "one", "one", "one", "single", "modes"])
    # site updates of a pass: about what the largest listed cases take in time
    budget = 2e7 if precision == "fp64" else (7e8 if tau == "one" else 1.2e8)
    budget = math.exp(rng.uniform(math.log(budget / 64), math.log(budget)))
    steps = rng.choice([20, 50, 100, 100, 200, 500])
    sites = max(2000.0, budget / steps)
    n_sizes = rng.choice([1, 1, 2, 3, 4])
    replicas = rng.choice([1, 2, 4, 8])
    per = max(1000.0, sites / (n_sizes * replicas))
    spectra = rng.random() < 0.35
    sizes = []
    for _ in range(n_sizes):
        v = per * math.exp(rng.uniform(-0.7, 0.3))
        # sides in use: multiples of 8 (as the ensembles have), of 4, or any number
        step = rng.choice([8, 8, 4, 1])

        def side(x, lo=6):
            return max(lo, int(round(x / step)) * step if step > 1 else int(x))

        if lattice == "D2Q9":
            nx = min(1448, side(math.sqrt(v)))
            ny, nz = (nx, 1) if spectra or rng.random() < 0.5 else (min(1448, side(v / nx)), 1)
        else:
            nx = min(160, side(v ** (1.0 / 3.0)))
            ny = nz = nx
            if not spectra and rng.random() < 0.5:
                ny = min(160, side(nx * rng.uniform(0.6, 1.4)))
                nz = min(160, side(v / (nx * ny)))
        sizes.append("%dx%dx%d" % (nx, ny, nz))
    obs = rng.choice([10, steps // 2, steps])
    a0 = rng.uniform(-0.004, 0.004)
    return case(lattice=lattice, coupling=coupling, precision=precision, sides=",".join(sizes), a0=a0, a1=a0,
                replicas=replicas, tau=tau, steps=steps, obs=obs, sk=steps if spectra else 0,
                jk=spectra and rng.random() < 0.5, hist=256 if precision == "fp64" and rng.random() < 0.3 else 0,
                chunk=rng.choice([0, steps]), field=math.prod(int(v) for v in sizes[0].split("x")) <= 50000)


# ---------------------------------------------------------------------------
# the run
# ---------------------------------------------------------------------------
def taus(c):
    """Relaxation times per mode: all 1 (the workloads), one other rate, or bulk,
    shear and ghost rates of their own."""
    q, nc = (9, 3) if c["lattice"] == "D2Q9" else (19, 4)
    if c["tau"] == "one":
        return [1.0] * q
    if c["tau"] == "single":
        return [1.0] * nc + [0.8] * (q - nc)
    n_shear = 2 if q == 9 else 5
    return [1.0] * nc + [1.2] + [0.8] * n_shear + [1.1] * (q - nc - 1 - n_shear)


def systems_of(c, seed):
    out = []
    for size in c["sides"].split(","):
        nx, ny, nz = (int(v) for v in size.split("x"))
        for k in range(c["n_a"]):
            a = c["a0"] + (c["a1"] - c["a0"]) * k / max(1, c["n_a"] - 1)
            for r in range(c["replicas"]):
                out.append(dict(lattice=c["lattice"], coupling=c["coupling"], nx=nx, ny=ny, nz=nz, rho_c=1.0, a=a,
                                b=c["b"], kappa=c["kappa"], kT=c["kT"], tau=taus(c), seed=int(seed) + r,
                                system_id=len(out)))
    return out


def density_of(systems, seed, device):
    """The quench: density 1 + U(-0.01, 0.01), each system's mean removed; one
    flat float64 tensor, systems concatenated."""
    gen = torch.Generator(device="cpu").manual_seed(int(seed))
    n = sum(s["nx"] * s["ny"] * s["nz"] for s in systems)
    d = (torch.rand(n, generator=gen, dtype=torch.float64) - 0.5).to(device) * 0.02
    at = 0
    for s in systems:
        k = s["nx"] * s["ny"] * s["nz"]
        d[at:at + k] += 1.0 - d[at:at + k].mean()
        at += k
    return d


def prepare(case, seed):
    c = case
    systems = systems_of(c, seed)
    opts = dict(precision=c["precision"], obs_every=c["obs"], sk_every=c["sk"], jk_spectra=c["jk"],
                graph_chunk=c["chunk"])
    if c["hist"]:
        opts.update(hist_bins=c["hist"], hist_range=0.1)
    ens = lb.Ensemble(systems, **opts)
    ens.init(rho_device=density_of(systems, seed, "cuda"))
    return dict(case=dict(c), ens=ens)


LEVEL = np.dtype([("block", "i4", 4), ("n", "f8"), ("sum_m", "f8"), ("sum_m2", "f8"), ("sum_abs_m", "f8"),
                  ("sum_m4", "f8"), ("sum_e", "f8"), ("sum_e2", "f8")])
GLOBAL = np.dtype([("step", "i8"), ("n_samples", "i8"), ("mass0", "f8"), ("mass", "f8"), ("momentum", "f8", 3),
                   ("rho_mean", "f8")])


def nbins_of(system):
    return max(2, system["nx"] // 2)


def run(state):
    c, ens = state["case"], state["ens"]
    real = np.float32 if c["precision"] == "fp32" else np.float64
    out = {}
    ens.step(c["steps"])
    if c["obs"]:
        levels, first, glob = ens.observables_all_raw()
        L, G = np.frombuffer(levels, dtype=LEVEL), np.frombuffer(glob, dtype=GLOBAL)
        out["n"] = L["n"].astype(np.int64)
        out["m"] = np.stack([L["sum_m"], L["sum_abs_m"]]).astype(real)
        for f in ("m2", "m4", "e", "e2"):
            out[f] = L["sum_" + f].astype(real)
        out["conserved"] = np.concatenate([G["mass"][:, None], G["momentum"]], axis=1).astype(real)
        if c["hist"]:
            # every block level below the whole system, whose order parameter is
            # zero by conservation (its bin would record rounding alone)
            out["hist"] = np.concatenate([ens.histogram(k, l)[0] for k in range(len(ens.systems))
                                          for l in range(1, first[k + 1] - first[k])]).astype(np.int64)
    if c["sk"]:
        sk = [ens.structure_factor(k, nbins_of(s)) for k, s in enumerate(ens.systems)]
        out["sk"] = np.concatenate([v[0] for v in sk]).astype(real)
        out["sk_points"] = np.concatenate([v[1] for v in sk])
        if c["jk"]:
            out["jk"] = np.concatenate([ens.momentum_spectra(k, nbins_of(s))[0].ravel()
                                        for k, s in enumerate(ens.systems)]).astype(real)
    if c["field"]:
        out["field"] = ens.read_fields(0).astype(real, copy=False)
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: every step reads and writes each population once; a sample reads
    them once more.  Operations: about 250 (D2Q9) or 600 (D3Q19) per site
    update for moments, equilibrium, noise and back-transform."""
    c = case
    systems = systems_of(c, 0)
    n = sum(s["nx"] * s["ny"] * s["nz"] for s in systems)
    q, es = (9 if c["lattice"] == "D2Q9" else 19), (4 if c["precision"] == "fp32" else 8)
    samples = (c["steps"] // c["obs"] if c["obs"] else 0) + (c["steps"] // c["sk"] if c["sk"] else 0)
    return {"bytes": float(n) * q * es * (2 * c["steps"] + samples),
            "flops": float(n) * c["steps"] * (250 if q == 9 else 600)}


# ---------------------------------------------------------------------------
# the same outputs in plain FP64 torch
# ---------------------------------------------------------------------------
EXACT_SITE_STEPS = 1.8e9          # about 20 s of a GB300


def velocities(lattice):
    if lattice == "D2Q9":
        return [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
                (-1, 1, 0)]
    faces = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
    edges = [(1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
             (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
    return [(0, 0, 0)] + faces + edges


class Model:
    """Tables of one lattice, coupling and set of relaxation times, as matrices
    on the features (conserved fields and their products) of a site."""

    def __init__(self, c, device):
        self.d2 = c["lattice"] == "D2Q9"
        self.vel = velocities(c["lattice"])
        v = np.array(self.vel, dtype=np.float64)
        x, y, z = v.T
        n2 = (v * v).sum(1)
        if self.d2:
            t = np.where(n2 == 0, 4 / 9, np.where(n2 == 1, 1 / 9, 1 / 36))
            T = [n2 * 0 + 1, x, y, 3 * n2 - 2, x * x - y * y, x * y, (3 * n2 - 4) * x, (3 * n2 - 4) * y,
                 9 * n2 * n2 - 15 * n2 + 2]
            self.nc, self.pair, shear, B = 3, (3, 8), 4, 3.0
        else:
            t = np.where(n2 == 0, 1 / 3, np.where(n2 == 1, 1 / 18, 1 / 36))
            T = [n2 * 0 + 1, x, y, z, n2 - 1, 3 * x * x - n2, y * y - z * z, x * y, y * z, z * x, (3 * n2 - 5) * x,
                 (3 * n2 - 5) * y, (3 * n2 - 5) * z, (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z,
                 3 * n2 * n2 - 6 * n2 + 1, (2 * n2 - 3) * (3 * x * x - n2), (2 * n2 - 3) * (y * y - z * z)]
            self.nc, self.pair, shear, B = 4, (4, 16), 6, 4.5
        T = np.array(T)
        N = (T * T * t).sum(1)
        Tinv = (t[:, None] * T.T) / N
        q = len(t)
        tau = np.array(taus(c))
        lam = 1.0 / tau
        lam[:self.nc] = 0.0
        gam = 1.0 - lam
        self.g = 1.0 - gam[:, None] * gam[None, :]
        self.N, self.T0, self.q, self.t = N, T[:, 0], q, t
        self.nu = (tau[shear] - 0.5) / 3.0
        self.guo = c["coupling"] == "guo"
        # features of the equilibrium: rho, iso, j (3), X (xx yy zz xy yz zx), K (the same six)
        six = [(0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (2, 0)]
        M = np.zeros((q, 17))
        for i in range(1, q):
            ci = v[i]
            M[i, 1] = 3 * t[i]
            M[i, 2:5] = 3 * t[i] * ci
            for k, (a, b) in enumerate(six):
                mult = 1.0 if a == b else 2.0
                M[i, 5 + k] = 4.5 * t[i] * mult * (ci[a] * ci[b] - (a == b) / 3.0)
                M[i, 11 + k] = t[i] * (4.5 * mult * ci[a] * ci[b] + (a == b) * (B - 4.5 * n2[i]))
        M[0] = -M[1:].sum(0)
        M[0, 0] += 1.0
        # features of the Guo source: F (3), u F symmetrised (xx yy zz xy yz zx)
        W = np.zeros((q, 9))
        for i in range(q):
            W[i, 0:3] = 3 * t[i] * v[i]
            for k, (a, b) in enumerate(six):
                W[i, 3 + k] = t[i] * (9.0 * v[i, a] * v[i, b] - 3.0 * (a == b))
        dev = dict(dtype=torch.float64, device=device)
        # f' = keep f + eq features + src features + back xi
        self.keep = torch.tensor(Tinv @ np.diag(1 - lam) @ T, **dev)
        self.eq = torch.tensor(Tinv @ np.diag(lam) @ T @ M, **dev)
        self.src = torch.tensor(Tinv @ np.diag(1 - lam / 2) @ T @ W, **dev)
        self.back = torch.tensor(Tinv[:, self.nc:], **dev)
        self.rest = torch.tensor(M, **dev)
        self.cvec = torch.tensor(v.T.copy(), **dev)


def at(s, c):
    """s(r + c) on the periodic lattice (last axes z, y, x)."""
    return torch.roll(s, shifts=(-c[2], -c[1], -c[0]), dims=(-3, -2, -1))


def gradient(s, m):
    g = [0.0, 0.0, 0.0]
    for i in range(1, m.q):
        v = at(s, m.vel[i])
        for a in range(3):
            if m.vel[i][a]:
                g[a] = g[a] + 3.0 * m.t[i] * m.vel[i][a] * v
    return [x if torch.is_tensor(x) else torch.zeros_like(s) for x in g]


def laplacian(s, m):
    out = torch.zeros_like(s)
    for i in range(1, m.q):
        out += 6.0 * m.t[i] * (at(s, m.vel[i]) - s)
    return out


def philox(ctr, key):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    mask = 0xFFFFFFFF
    c0, c1, c2, c3 = ctr
    k0, k1 = key
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        pa, pb = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((pb >> 32) & mask) ^ c1 ^ k0, pb & mask, ((pa >> 32) & mask) ^ c3 ^ k1, pa & mask
    return c0, c1, c2, c3


def normals(n_sys, n_sites, ids, seeds, step, count, device):
    """(count, systems, sites) standard normals of one step, in draw order."""
    site = torch.arange(n_sites, dtype=torch.int64, device=device)[None, :].expand(n_sys, -1)
    zero = torch.zeros_like(site)
    key = ((seeds & 0xFFFFFFFF)[:, None], (seeds >> 32)[:, None])
    out = torch.empty((count, n_sys, n_sites), dtype=torch.float64, device=device)
    for d in range((count + 3) // 4):
        w = philox((site, zero + (step & 0xFFFFFFFF), zero + (step >> 32), zero + (ids[:, None] * 256 + d)), key)
        for h in (0, 2):
            k = 4 * d + h
            if k >= count:
                continue
            r = torch.sqrt(-2.0 * torch.log((w[h].double() + 0.5) * 2.0 ** -32))
            ang = (2.0 * math.pi) * ((w[h + 1].double() + 0.5) * 2.0 ** -32)
            out[k] = r * torch.cos(ang)
            if k + 1 < count:
                out[k + 1] = r * torch.sin(ang)
    return out


def products(p, q_):
    """p_a q_b symmetrised: xx yy zz xy yz zx."""
    return [p[0] * q_[0], p[1] * q_[1], p[2] * q_[2]] + [0.5 * (p[a] * q_[b] + p[b] * q_[a])
                                                         for a, b in ((0, 1), (1, 2), (2, 0))]


def thermo(rho, A, b):
    phi = rho - 1.0
    p0 = rho * (A * phi + b * phi ** 3) - (0.5 * A * phi ** 2 + 0.25 * b * phi ** 4)
    return p0, rho * (A + 3.0 * b * phi ** 2)


def step_exact(f, t, m, c, A, ids, seeds):
    """One time step of every system of a size class, f (q, systems, z, y, x)."""
    rho = f.sum(0)
    j = list(torch.tensordot(m.cvec, f, dims=1))
    lap = laplacian(rho, m)
    p0, cs2 = thermo(rho, A, c["b"])
    zero = torch.zeros_like(rho)
    new = torch.tensordot(m.keep, f, dims=1)
    if m.guo:
        F = [c["kappa"] * rho * g for g in gradient(lap, m)]
        u = [(j[a] + 0.5 * F[a]) / rho for a in range(3)]
        feats = [rho, p0] + [rho * ua for ua in u] + [rho * w for w in products(u, u)] + [zero] * 6
        new += torch.tensordot(m.src, torch.stack(F + [w if k < 3 else 2.0 * w
                                                       for k, w in enumerate(products(u, F))]), dims=1)
    else:
        g = gradient(rho, m)
        u = [x / rho for x in j]
        udg = u[0] * g[0] + u[1] * g[1] + u[2] * g[2]
        ug = products(u, g)
        X = [rho * w + m.nu * (2.0 * ug[k] + (udg if k < 3 else 0.0)) for k, w in enumerate(products(u, u))]
        if m.d2:
            X[2] = zero                                # no z components in two dimensions
        feats = [rho, p0 - c["kappa"] * rho * lap] + j + X + [c["kappa"] * w for w in products(g, g)]
    new += torch.tensordot(m.eq, torch.stack(feats), dims=1)
    if c["kT"] > 0:
        K = m.q - m.nc
        n = normals(rho.shape[0], rho[0].numel(), ids, seeds, t, K, f.device).reshape((K,) + tuple(rho.shape))
        scale = torch.sqrt(3.0 * rho * c["kT"])
        P, R = m.pair
        om = 1.0 - 3.0 * cs2
        mpp = (m.N[P] + om * m.T0[P] ** 2) * m.g[P, P]
        mrr = (m.N[R] + om * m.T0[R] ** 2) * m.g[R, R]
        mpr = om * m.T0[P] * m.T0[R] * m.g[P, R]
        l11 = torch.sqrt(mpp)
        l21 = mpr / l11
        l22 = torch.sqrt(mrr - l21 * l21)
        nP = n[P - m.nc].clone()
        n[R - m.nc] = l21 * nP + l22 * n[R - m.nc]
        n[P - m.nc] = l11 * nP
        for a in range(m.nc, m.q):
            if a not in (P, R):
                n[a - m.nc] *= math.sqrt(m.N[a] * m.g[a, a])
        new += torch.tensordot(m.back, n * scale, dims=1)
    for i in range(m.q):
        cx, cy, cz = m.vel[i]
        f[i] = torch.roll(new[i], shifts=(cz, cy, cx), dims=(-3, -2, -1))
    return f


def rest_state(rho, m, c, A):
    """f^eq(rho, u = 0, grad rho)."""
    p0, _ = thermo(rho, A, c["b"])
    zero = torch.zeros_like(rho)
    if m.guo:
        feats = [rho, p0] + [zero] * 15
    else:
        g = gradient(rho, m)
        feats = [rho, p0 - c["kappa"] * rho * laplacian(rho, m)] + [zero] * 9 + [c["kappa"] * w
                                                                                 for w in products(g, g)]
    return torch.tensordot(m.rest, torch.stack(feats), dims=1)


def block_dims(nx, ny, nz, d2):
    out, k = [], 1
    while nx % k == 0 and ny % k == 0 and (d2 or nz % k == 0):
        out.append((nx // k, ny // k, 1 if d2 else nz // k))
        if out[-1] == (1, 1, 1):
            return out
        k *= 2
    return out + [(1, 1, 1)]


def block_sums(phi, dims):
    """Per system (m, |m|, m^2, m^4, e, e^2) sums over the blocks of one level."""
    s, (nz, ny, nx), (bx, by, bz) = phi.shape[0], phi.shape[1:], dims
    v = phi.reshape(s, nz // bz, bz, ny // by, by, nx // bx, bx)
    m = v.mean(dim=(2, 4, 6)).reshape(s, -1)
    e = 0.5 * (v * v).mean(dim=(2, 4, 6)).reshape(s, -1)
    return torch.stack([m.sum(1), m.abs().sum(1), (m * m).sum(1), (m ** 4).sum(1), e.sum(1), (e * e).sum(1)], 1)


def shells(shape, d2, device):
    """Shell index of every k point: the integer nearest |n|, 0 at k = 0."""
    n2 = 0
    for ax, n in zip((0, 1, 2), shape):
        if d2 and ax == 0:
            continue
        k = torch.arange(n, device=device)
        k = torch.where(2 * k < n, k, k - n)
        n2 = n2 + (k * k).reshape([-1 if a == ax else 1 for a in range(3)])
    n2 = n2.expand(shape) if n2.dim() == 3 else n2
    j = torch.floor(torch.sqrt(n2.double())).long()
    j = torch.where(j * (j + 1) < n2, j + 1, j)
    return torch.where(j * (j - 1) >= n2, j - 1, j).clamp_min(0)


def binned(spec, shell, nbins):
    """Shell sums (systems, nbins) of (systems, z, y, x) spectra."""
    s = spec.shape[0]
    out = torch.zeros((s, int(shell.max()) + 1), dtype=torch.float64, device=spec.device)
    out.index_add_(1, shell.reshape(-1), spec.reshape(s, -1))
    return out[:, 1:nbins + 1]


def momentum_spectra(f, m, c, d2):
    rho = f.sum(0)
    j = list(torch.tensordot(m.cvec, f, dims=1))
    if m.guo:
        g = gradient(laplacian(rho, m), m)
        j = [j[a] + 0.5 * c["kappa"] * rho * g[a] for a in range(3)]
    d = 2 if d2 else 3
    shape, N = tuple(rho.shape[1:]), float(rho[0].numel())
    J = [torch.fft.fftn(j[a], dim=(-3, -2, -1)) for a in range(d)]
    nv = []
    for ax, n in ((2, shape[2]), (1, shape[1]), (0, shape[0])):
        k = torch.arange(n, device=f.device)
        k = torch.where(2 * k < n, k, k - n).double()
        nv.append(k.reshape([-1 if a == ax else 1 for a in range(3)]))
    nn = torch.sqrt(sum(v * v for v in nv[:d]))
    safe = torch.where(nn > 0, nn, torch.ones_like(nn))
    p2 = sum((nv[a] / safe) * J[a] for a in range(d)).abs() ** 2
    tot = sum(x.abs() ** 2 for x in J)
    nonzero = (nn > 0).double()
    return [J[0].abs() ** 2 / N, nonzero * p2 / N, nonzero * (tot - p2) / (N * (d - 1))]


def exact(case, seed):
    c = case
    systems = systems_of(c, seed)
    sites = sum(s["nx"] * s["ny"] * s["nz"] for s in systems)
    if sites * c["steps"] > EXACT_SITE_STEPS:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    d2 = c["lattice"] == "D2Q9"
    m = Model(c, dev)
    rho_all = density_of(systems, seed, dev)
    per = c["n_a"] * c["replicas"]                     # systems of one size are consecutive
    rows, at_site, field = [], 0, None
    for first in range(0, len(systems), per):
        group = systems[first:first + per]
        nx, ny, nz = (group[0][k] for k in ("nx", "ny", "nz"))
        n = nx * ny * nz
        rho = rho_all[at_site:at_site + n * per].reshape(per, nz, ny, nx)
        at_site += n * per
        A = torch.tensor([s["a"] for s in group], dtype=torch.float64, device=dev).reshape(-1, 1, 1, 1)
        ids = torch.tensor([s["system_id"] for s in group], dtype=torch.int64, device=dev)
        seeds = torch.tensor([s["seed"] for s in group], dtype=torch.int64, device=dev)
        f = rest_state(rho, m, c, A)
        dims = block_dims(nx, ny, nz, d2)
        acc = [0.0] * len(dims)
        sk = jk = cons = None
        nb = nbins_of(group[0])
        shell = shells((nz, ny, nx), d2, dev) if c["sk"] else None
        for t in range(c["steps"]):
            f = step_exact(f, t, m, c, A, ids, seeds)
            obs_due = c["obs"] and (t + 1) % c["obs"] == 0
            sk_due = c["sk"] and (t + 1) % c["sk"] == 0
            if not (obs_due or sk_due):
                continue
            r = f.sum(0)
            mean = r.mean(dim=(1, 2, 3), keepdim=True)
            phi = (r - mean) / mean
            if obs_due:
                acc = [x + block_sums(phi, b) for x, b in zip(acc, dims)]
                cons = torch.cat([r.sum(dim=(1, 2, 3))[:, None],
                                  torch.tensordot(m.cvec, f, dims=1).sum(dim=(2, 3, 4)).T], 1)
            if sk_due:
                s_ = binned(torch.fft.fftn(phi, dim=(-3, -2, -1)).abs() ** 2 / n, shell, nb)
                sk = s_ if sk is None else sk + s_
                if c["jk"]:
                    j_ = torch.stack([binned(x, shell, nb) for x in momentum_spectra(f, m, c, d2)], 1)
                    jk = j_ if jk is None else jk + j_
        if first == 0 and c["field"]:
            field = f[:, 0].cpu().numpy()
        rows.append((per, dims, acc, cons, sk, jk))
    out = {}
    if c["obs"]:
        L = torch.stack([acc[l][k] for per, dims, acc, *_ in rows for k in range(per)
                         for l in range(len(dims))]).cpu().numpy()
        out["n"] = None
        out["m"] = np.stack([L[:, 0], L[:, 1]])
        out.update(m2=L[:, 2], m4=L[:, 3], e=L[:, 4], e2=L[:, 5])
        out["conserved"] = torch.cat([r[3] for r in rows]).cpu().numpy()
        if c["hist"]:
            out["hist"] = None
    if c["sk"]:
        out["sk"] = torch.cat([r[4].reshape(-1) for r in rows]).cpu().numpy()
        out["sk_points"] = None
        if c["jk"]:
            out["jk"] = torch.cat([r[5].reshape(-1) for r in rows]).cpu().numpy()
    if c["field"]:
        out["field"] = field
    return out
