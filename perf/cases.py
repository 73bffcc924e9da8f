"""The work that users of this library have it do, as measurable cases.

Four kinds of case, each through the public Python binding:

lattice   one periodic lattice: a run from initial fields to final moments (or from given
          populations to final populations), `steps` time steps in one lbm_step call.
batch     many independent small lattices with Fourier probes: initial fields, `steps`
          steps, the probe series and the final moments.
eigs      von Neumann eigenvalues of many parameter points.
limit     the linear-stability limit over a (viscosity, angle) table for all equilibria.

`listed` names the cases, `draw` samples the same ranges, `prepare` makes the inputs (from
the seed alone) and the object a program keeps, `run` is one pass, `work` the bytes and
operations a pass cannot do without and `exact` the same outputs in FP64 torch / NumPy
arithmetic written out from the formulas, without the library.
"""
import math

import numpy as np
import torch

from paper_2303_08163_gb300 import inputs, lbm

EQS = {"entropic": lbm.ENTROPIC, "poly2": lbm.POLY2, "product": lbm.PRODUCT}
PRECS = {"f64": lbm.F64, "f32": lbm.F32, "f16s": lbm.F16S}
ESIZE = {"f64": 8, "f32": 4, "f16s": 2}
DEV = "cuda"


# ---------------------------------------------------------------------------------- cases

def _lattice(D, nx, ny, nz, prec, flow, tau, steps, eq="entropic", bulk=0, diag=0, io="fields"):
    return {"kind": "lattice", "D": D, "nx": nx, "ny": ny, "nz": nz, "prec": prec, "flow": flow,
            "tau": tau, "steps": steps, "eq": eq, "bulk": bulk, "diag": diag, "io": io}


def _re1600_tau(n):
    """Relaxation time of the vortex at Re = 1600 (u0 = 0.1) on n cells per side."""
    return 0.5 + 3 * 0.1 * n / (2 * math.pi) / 1600.0


def listed():
    return [
        # the small FP64 validation run: a 64^2 vortex, 1000 steps, energy decay checked after
        dict(_lattice(2, 64, 64, 1, "f64", "vortex", 0.8, 1000), name="tgv2d-64-f64"),
        # a small 3-D run in the production precision, as in parameter studies and tests
        dict(_lattice(3, 32, 32, 32, "f16s", "vortex", 0.6, 500, bulk=1), name="tgv3d-32-f16s"),
        # an odd-sized 2-D lattice (rows of no 16-byte multiple), comparison equilibrium
        dict(_lattice(2, 509, 381, 1, "f32", "shear", 0.51, 200, eq="poly2"), name="shear2d-ragged-f32"),
        # the 4096^2 double shear layer with its fused diagnostics every 10 steps
        dict(_lattice(2, 4096, 4096, 1, "f32", "shear", 0.5 + 3e-5, 50, diag=10), name="shear2d-4096-f32"),
        # a ragged 3-D box of decaying turbulence, binary16 storage
        dict(_lattice(3, 250, 131, 67, "f16s", "modes", 0.52, 50), name="turb3d-ragged-f16s"),
        # a mid-sized 3-D run in FP32 storage with the bulk correction
        dict(_lattice(3, 256, 256, 256, "f32", "vortex", _re1600_tau(256), 20, bulk=1), name="tgv3d-256-f32-bulk"),
        # FP64 storage in 3-D resumed from and saved to populations, an odd number of steps
        dict(_lattice(3, 128, 128, 128, "f64", "vortex", 0.6, 11, io="populations"), name="tgv3d-128-f64-pop"),
        # the headline run: 512^3 Taylor-Green vortex, binary16 storage, diagnostics every 10
        dict(_lattice(3, 512, 512, 512, "f16s", "vortex", _re1600_tau(512), 20, diag=10), name="tgv3d-512-f16s"),
        # the linear-mode sweep: thousands of small FP64 lattices, probes every 10 steps
        {"name": "batch-sweep-4096", "kind": "batch", "count": 4096, "nmin": 16, "nmax": 256, "flat": False,
         "steps": 20, "every": 10, "eq": "entropic", "bulk": 0, "table": 2303},
        # the pressure-wave experiment: a few one-dimensional lattices, many steps
        {"name": "batch-wave-1d", "kind": "batch", "count": 28, "nmin": 128, "nmax": 128, "flat": True,
         "steps": 1000, "every": 10, "eq": "entropic", "bulk": 1, "table": 7},
        # dispersion / dissipation of the sweep's instances from the linear theory
        {"name": "vn-eigs-4096", "kind": "eigs", "count": 4096, "eq": "entropic", "bulk": 0},
        # the stability-domain figure: the three equilibria over 6 viscosities x 9 angles
        {"name": "vn-limit-table", "kind": "limit", "pairs": 54, "nk": 25, "iterations": 14},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


MOST_UPDATES = 512 ** 3 * 20


def draw(rng):
    """A case of the listed ranges: any size between the smallest and the largest, odd and
    ragged ones among them, every precision, equilibrium, option and direction."""
    kind = rng.choice(["lattice2", "lattice2", "lattice2", "lattice3", "lattice3", "lattice3", "batch", "batch",
                       "eigs", "limit"])
    eq = rng.choice(["entropic", "entropic", "poly2", "product"])
    bulk = rng.choice([0, 1])
    if kind.startswith("lattice"):
        D = int(kind[-1])
        prec = rng.choice(["f16s", "f32", "f64"] if D == 2 else ["f16s", "f16s", "f32", "f32", "f64"])
        # side lengths around a common log-uniform size; half of the rows 16-byte multiples
        top = 4096 if D == 2 else 512
        n = _logint(rng, 64 if D == 2 else 32, top)
        if prec == "f64":
            n = min(n, 2048 if D == 2 else 192)
        side = [max(8, min(top, int(n * rng.uniform(0.7, 1.4)))) for _ in range(D)]
        side[0] = max(8, side[0] // 8 * 8) if rng.random() < 0.5 else side[0] | 1 if rng.random() < 0.5 else side[0]
        cells = math.prod(side)
        most = MOST_UPDATES // (16 if prec == "f64" else 2 if prec == "f32" else 1)
        steps = max(1, min(_logint(rng, 10, 1000), most // (4 * cells)))
        flow = rng.choice(["vortex", "modes"] if D == 3 else ["vortex", "shear"])
        io = rng.choice(["fields", "fields", "fields", "populations"])
        diag = rng.choice([0, 0, 10]) if io == "fields" else 0
        tau = 0.5 + math.exp(rng.uniform(math.log(0.005), math.log(0.5)))
        return _lattice(D, side[0], side[1], side[2] if D == 3 else 1, prec, flow, tau, steps, eq, bulk, diag, io)
    if kind == "batch":
        if rng.random() < 0.4:
            return {"kind": "batch", "count": rng.randint(4, 64), "nmin": 64, "nmax": rng.choice([64, 128, 200]),
                    "flat": True, "steps": _logint(rng, 100, 2000), "every": rng.choice([1, 10]), "eq": eq,
                    "bulk": bulk, "table": rng.randint(1, 10000)}
        count = _logint(rng, 16, 4096)
        return {"kind": "batch", "count": count, "nmin": 16, "nmax": rng.choice([96, 160, 256]), "flat": False,
                "steps": max(10, min(200, 81920 // count)), "every": rng.choice([5, 10]), "eq": eq, "bulk": bulk,
                "table": rng.randint(1, 10000)}
    if kind == "eigs":
        return {"kind": "eigs", "count": _logint(rng, 64, 65536), "eq": eq, "bulk": bulk}
    return {"kind": "limit", "pairs": rng.randint(1, 54), "nk": rng.choice([17, 25, 33]),
            "iterations": rng.randint(8, 20)}


# --------------------------------------------------------------------------------- inputs

def _dims(case):
    return case["nx"], case["ny"], case["nz"]


def _fields(case, seed):
    """Initial rho (ncell,) and u (D, ncell) of a lattice case in FP64, on the GPU: a
    vortex, a double shear layer or a few solenoidal Fourier modes, with seeded phases."""
    nx, ny, nz = _dims(case)
    D = case["D"]
    r = np.random.default_rng([seed, 11])
    t = [2 * math.pi * torch.arange(n, device=DEV, dtype=torch.float64) / n for n in (nx, ny, nz)]
    ph = r.uniform(0, 2 * math.pi, 3)
    X, Y, Z = t[0][None, None, :] + ph[0], t[1][None, :, None] + ph[1], t[2][:, None, None] + (ph[2] if D == 3 else 0.0)
    shape = (nz, ny, nx)
    u = torch.zeros((D,) + shape, device=DEV, dtype=torch.float64)
    rho = torch.ones(shape, device=DEV, dtype=torch.float64)
    if case["flow"] == "vortex":
        u0 = 0.1 if D == 3 else 0.05
        cz = torch.cos(Z) if D == 3 else 1.0
        u[0] = u0 * torch.sin(X) * torch.cos(Y) * cz
        u[1] = -u0 * torch.cos(X) * torch.sin(Y) * cz
        if D == 3:
            rho += u0 * u0 * 3.0 / 16.0 * (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2.0)
    elif case["flow"] == "shear":
        y = torch.remainder(Y / (2 * math.pi), 1.0)
        u[0] = torch.where(y <= 0.5, 0.1 * torch.tanh(80 * (y - 0.25)), 0.1 * torch.tanh(80 * (0.75 - y)))
        u[1] = 0.005 * torch.sin(X)
    else:
        for _ in range(6):
            k = r.integers(1, 5, 3)
            kk = k * 2 * math.pi / np.array([nx, ny, nz])
            a = np.cross(kk, r.normal(size=3))
            a *= 0.03 / max(float(np.linalg.norm(a)), 1e-30)
            w = torch.cos(int(k[0]) * X + int(k[1]) * Y + int(k[2]) * Z + r.uniform(0, 2 * math.pi))
            for c in range(3):
                u[c] += float(a[c]) * w
    return rho.reshape(-1), u.reshape(D, -1)


def _io_dtype(case):
    return (torch.float64, np.float64) if case["prec"] == "f64" else (torch.float32, np.float32)


def _populations(case, seed):
    """Given canonical populations: the equilibrium of the fields with 0.1 % of seeded
    noise, in the type that they are handed over in."""
    rho, u = _fields(case, seed)
    td, _ = _io_dtype(case)
    f = torch.stack([v.to(td) for v in _equilibrium(case["D"], case["eq"], rho, u)])
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    f *= 1 + 1e-3 * (torch.rand(f.shape, generator=gen, device=DEV, dtype=torch.float32).to(td) - 0.5)
    return f


def _table(case, seed):
    """Instance table of a batch: sizes and wavenumbers from the case, the rest seeded."""
    t = inputs.linear_mode_batch(count=case["count"], seed=case["table"], nmin=case["nmin"], nmax=case["nmax"])
    r = np.random.default_rng([seed, 12])
    n = case["count"]
    if case["flat"]:
        t["ny"] = np.ones(n, dtype=np.int32)
        t["nmode"] = np.ones(n, dtype=np.int32)
        t["kind"] = np.ones(n, dtype=np.int32)
        t["U0"] = np.linspace(-0.3, 0.3, n)
        t["tau"] = np.full(n, 0.65)
        t["amp"] = 1e-3
    t["phase"] = r.uniform(0, 2 * math.pi, n)
    return t


def _cells(t):
    """Per packed cell of a batch: instance, x, y (device), and the instance offsets."""
    n = torch.from_numpy((t["nx"].astype(np.int64) * t["ny"])).to(DEV)
    start = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(n, 0)])
    inst = torch.repeat_interleave(torch.arange(len(n), device=DEV), n)
    nx = torch.from_numpy(t["nx"].astype(np.int64)).to(DEV)
    local = torch.arange(int(start[-1]), device=DEV) - start[inst]
    return inst, local % nx[inst], local // nx[inst], local, start, nx


def _batch_fields(t):
    """rho (total,) and the two velocity components (total,) of a batch, FP64."""
    inst, x, _, _, _, nx = _cells(t)
    d = {k: torch.from_numpy(np.asarray(t[k], dtype=np.float64)).to(DEV) for k in ("nmode", "U0", "phase", "kind")}
    wave = t["amp"] * torch.sin(2 * math.pi * d["nmode"][inst] * x / nx[inst] + d["phase"][inst])
    sound = d["kind"][inst] == 1
    rho = torch.where(sound, 1.0 + wave, torch.ones_like(wave))
    return rho, d["U0"][inst].clone(), torch.where(sound, torch.zeros_like(wave), wave)


def _pack(t, ux, uy):
    """Per-instance [2][cells] packing of two velocity components."""
    inst, _, _, local, start, _ = _cells(t)
    n = start[1:] - start[:-1]
    out = torch.empty(2 * len(ux), device=DEV, dtype=ux.dtype)
    out[2 * start[inst] + local] = ux
    out[2 * start[inst] + n[inst] + local] = uy
    return out


def _eig_params(case, seed):
    r = np.random.default_rng([seed, 13])
    n = case["count"]
    um = 0.3
    return np.stack([0.5 + np.exp(r.uniform(math.log(5e-4), 0.0, n)), r.uniform(0.9, 1.1, n),
                     r.uniform(-um, um, n), r.uniform(-um, um, n),
                     r.uniform(0, math.pi, n), r.uniform(0, math.pi, n)], axis=1)


def _limit_pairs(case, seed):
    r = np.random.default_rng([seed, 14])
    n = case["pairs"]
    nus = 10.0 ** (np.linspace(-6, 0.08, n) + r.uniform(-0.05, 0.05, n))
    return nus, r.permutation(np.linspace(0, math.pi / 2, n)) if n > 1 else r.uniform(0, math.pi / 2, 1)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        td, nd = _io_dtype(case)
        lat = lbm.Lattice(lbm.D2Q9 if case["D"] == 2 else lbm.D3Q27, _dims(case), case["tau"], EQS[case["eq"]],
                          case["bulk"], PRECS[case["prec"]])
        if case["diag"]:
            lat.set_option(lbm.OPT_DIAG_EVERY, case["diag"])
        s = {"case": case, "lat": lat, "nd": nd}
        n = lat.ncell
        if case["io"] == "populations":
            s["f"] = _populations(case, seed)
            s["out"] = torch.empty((lat.Q, n), device=DEV, dtype=td)
        else:
            rho, u = _fields(case, seed)
            s["rho"], s["u"] = rho.to(td), u.to(td).contiguous()
            s["out"] = (torch.empty(n, device=DEV, dtype=td), torch.empty((lat.D, n), device=DEV, dtype=td))
        return s
    if kind == "batch":
        t = _table(case, seed)
        dims = np.stack([t["nx"], t["ny"], np.ones(case["count"], dtype=np.int32)], axis=1)
        b = lbm.Batch(lbm.D2Q9, dims, t["tau"], EQS[case["eq"]], case["bulk"])
        kvec = np.stack([t["nmode"], 0 * t["nmode"], 0 * t["nmode"]], axis=1)
        b.set_probe(kvec, case["every"])
        rho, ux, uy = _batch_fields(t)
        u = _pack(t, ux, uy)
        return {"case": case, "batch": b, "rho": rho, "u": u, "out": (torch.empty_like(rho), torch.empty_like(u))}
    if kind == "eigs":
        return {"case": case, "params": _eig_params(case, seed)}
    nu, theta = _limit_pairs(case, seed)
    return {"case": case, "nu": nu, "theta": theta}


# ----------------------------------------------------------------------------------- pass

def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "lattice":
        lat = s["lat"]
        if case["io"] == "populations":
            lat.set_populations(s["f"], dtype=s["nd"])
            lat.step(case["steps"])
            return lat.get_populations(dtype=s["nd"], out=s["out"])
        lat.init_fields(s["rho"], s["u"], dtype=s["nd"])
        lat.step(case["steps"])
        rho, u = lat.moments(dtype=s["nd"], out=s["out"])
        got = {"rho": rho, "u": u}
        if case["diag"]:
            h = lat.diag_history()
            got["diag"] = np.array([[d["mass"], *d["momentum"], d["kinetic"], d["max_u"]] for d in h])
        return got
    if kind == "batch":
        b = s["batch"]
        b.init_fields(s["rho"], s["u"])
        b.step(case["steps"])
        series = b.probe_series()
        rho, u = b.moments(out=s["out"])
        return {"series": series, "rho": rho, "u": u}
    if kind == "eigs":
        return lbm.vn_eigenvalues(EQS[case["eq"]], case["bulk"], s["params"])
    return {name: lbm.vn_stability_limit(eq, s["nu"], s["theta"], nk=case["nk"], u_hi=0.95,
                                         iterations=case["iterations"]) for name, eq in EQS.items()}


# ----------------------------------------------------------------------------------- work

def _cell_flops(D, eq, bulk):
    """Floating-point operations of one cell update (an FMA is two, a division or a square
    root one): the moments, the equilibrium's factors, two FMAs and one product a direction."""
    base = {("entropic", 2): 116, ("poly2", 2): 107, ("product", 2): 100,
            ("entropic", 3): 309, ("poly2", 3): 310, ("product", 3): 284}[(eq, D)]
    return base + (6 if bulk else 0)


def work(case):
    """Inputs read once, outputs and the updated state written once; the collisions' flops."""
    kind = case["kind"]
    if kind == "lattice":
        cells, D = math.prod(_dims(case)), case["D"]
        Q, io = 3 ** D, 8 if case["prec"] == "f64" else 4
        ends = 2 * cells * io * (Q if case["io"] == "populations" else D + 1)
        return {"bytes": ends + cells * Q * ESIZE[case["prec"]],
                "flops": cells * case["steps"] * _cell_flops(D, case["eq"], case["bulk"])}
    if kind == "batch":
        t = _table(case, 0)
        cells = int((t["nx"].astype(np.int64) * t["ny"]).sum())
        samples = -(-case["steps"] // case["every"])
        return {"bytes": cells * (2 * 3 * 8 + 9 * 8) + case["count"] * samples * 64,
                "flops": cells * (case["steps"] * _cell_flops(2, case["eq"], case["bulk"]) + samples * 24)}
    # complex 9 x 9 eigenvalues: about 10 n^3 complex operations of 8 flops
    one = 10 * 9 ** 3 * 8
    if kind == "eigs":
        return {"bytes": case["count"] * (6 + 18) * 8, "flops": case["count"] * one}
    # the search's result needs at least one spectrum per wave vector of each stable bound
    return {"bytes": case["pairs"] * 3 * 8, "flops": 3 * case["pairs"] * case["nk"] ** 2 * one}


# ---------------------------------------------------------------- the same in 64 bits, plain

W1 = {-1: 1 / 6, 0: 2 / 3, 1: 1 / 6}


def _velocities(D):
    return [((i % 3) - 1, (i // 3) % 3 - 1, (i // 9) - 1 if D == 3 else 0) for i in range(3 ** D)]


def _factors(eq, u):
    """1-D factors a(c) with f^eq = rho prod_a a_a(c_a): a(0), a(+1), a(-1) as c -> tensor."""
    if eq == "entropic":
        S = torch.sqrt(1 + 3 * u * u)
        Z = (2 * u + S) / (1 - u)
        return {0: 2 / 3 * (2 - S), 1: (2 - S) * Z / 6, -1: (2 - S) / Z / 6}
    return {0: 2 / 3 - u * u, 1: 1 / 6 + u / 2 + u * u / 2, -1: 1 / 6 - u / 2 + u * u / 2}


def _equilibrium(D, eq, rho, u):
    """f^eq_i(rho, u) of every direction, one at a time (u: D tensors)."""
    if eq == "poly2":
        uu = sum(u[a] * u[a] for a in range(D))
        for c in _velocities(D):
            cu = sum((c[a] * u[a] for a in range(D) if c[a]), torch.zeros_like(rho))
            w = math.prod(W1[c[a]] for a in range(D))
            yield w * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)
        return
    fac = [_factors(eq, u[a]) for a in range(D)]
    for c in _velocities(D):
        v = rho
        for a in range(D):
            v = v * fac[a][c[a]]
        yield v


def _rate(eq, bulk, tau, u):
    """2 beta: 1 / tau, or with the local correction of the bulk viscosity."""
    if not bulk:
        return 1.0 / tau
    umax = u[0].abs()
    for v in u[1:]:
        umax = torch.maximum(umax, v.abs())
    nu = (tau - 0.5) / 3.0
    if eq == "entropic":
        S = torch.sqrt(1 + 3 * umax * umax)
        A = (2 - S) / (S * S)
    else:
        A = 1 - 4.5 * umax * umax
    return 2 / (6 * nu / A + 1)


def _moments(D, f):
    rho = f[0].clone()
    for v in f[1:]:
        rho += v
    j = [torch.zeros_like(rho) for _ in range(D)]
    for c, v in zip(_velocities(D), f):
        for a in range(D):
            if c[a]:
                j[a] += c[a] * v
    return rho, [v / rho for v in j]


def _exact_lattice(case, seed):
    D, (nx, ny, nz) = case["D"], _dims(case)
    td, _ = _io_dtype(case)
    shape = (nz, ny, nx)
    if case["io"] == "populations":
        f = [v.double().reshape(shape) for v in _populations(case, seed)]
    else:
        rho, u = _fields(case, seed)
        rho, u = rho.to(td).double().reshape(shape), [v.to(td).double().reshape(shape) for v in u]
        f = [v.clone() for v in _equilibrium(D, case["eq"], rho, u)]
        del rho, u
    diags = []
    for t in range(case["steps"]):
        rho, u = _moments(D, f)
        if case["diag"] and t % case["diag"] == 0:
            ke = sum((rho * v * v).sum() for v in u) / 2
            j = [float((rho * v).sum()) for v in u] + [0.0] * (3 - D)
            diags.append([float(rho.sum()), *j, float(ke), max(float(v.abs().max()) for v in u)])
        om = _rate(case["eq"], case["bulk"], case["tau"], u)
        for i, (c, e) in enumerate(zip(_velocities(D), _equilibrium(D, case["eq"], rho, u))):
            f[i] = torch.roll(f[i] + om * (e - f[i]), (c[2], c[1], c[0]), (0, 1, 2))
        del rho, u, om
    if case["io"] == "populations":
        return torch.stack([v.reshape(-1) for v in f])
    rho, u = _moments(D, f)
    got = {"rho": rho.reshape(-1), "u": torch.stack([v.reshape(-1) for v in u])}
    if case["diag"]:
        got["diag"] = np.array(diags)
    return got


def _exact_batch(case, seed):
    t = _table(case, seed)
    inst, x, y, _, start, nxs = _cells(t)
    nys = torch.from_numpy(t["ny"].astype(np.int64)).to(DEV)
    nx, ny, base = nxs[inst], nys[inst], start[inst]
    src = [base + (x - c[0]) % nx + nx * ((y - c[1]) % ny) for c in _velocities(2)]
    tau = torch.from_numpy(np.asarray(t["tau"], dtype=np.float64)).to(DEV)[inst]
    kx = 2 * math.pi * torch.from_numpy(t["nmode"].astype(np.float64)).to(DEV)[inst] * x / nx
    rho, ux, uy = _batch_fields(t)
    f = [v.clone() for v in _equilibrium(2, case["eq"], rho, [ux, uy])]
    series = []
    for n in range(case["steps"]):
        rho, u = _moments(2, f)
        if n % case["every"] == 0:
            one = torch.zeros((case["count"], 4, 2), device=DEV, dtype=torch.float64)
            for q, v in enumerate([rho, rho * u[0], rho * u[1]]):
                one[:, q, 0].index_add_(0, inst, v * torch.cos(kx))
                one[:, q, 1].index_add_(0, inst, -v * torch.sin(kx))
            series.append(one)
        om = _rate(case["eq"], case["bulk"], tau, u)
        f = [(v + om * (e - v))[s] for v, e, s in zip(f, _equilibrium(2, case["eq"], rho, u), src)]
    rho, u = _moments(2, f)
    return {"series": torch.view_as_complex(torch.stack(series, 1).contiguous()), "rho": rho,
            "u": _pack(t, u[0], u[1])}


def _vn_matrices(eq, bulk, p):
    """Amplification matrices (count, 9, 9) of parameter points (tau, rho, u_x, u_y, k_x, k_y):
    E (1 + 2 beta (d f^eq / d f - 1)), the derivatives by automatic differentiation."""
    p = torch.from_numpy(p)
    rho, ux, uy = (p[:, i].clone().requires_grad_() for i in (1, 2, 3))
    c = np.array(_velocities(2), dtype=np.float64)
    rows = []
    for e in _equilibrium(2, eq, rho, [ux, uy]):
        g = torch.autograd.grad(e.sum(), (rho, ux, uy), retain_graph=True)
        rows.append(torch.stack([g[0] + (g[1] * (c[j, 0] - ux) + g[2] * (c[j, 1] - uy)) / rho for j in range(9)], 1))
    J = torch.stack(rows, 1).detach()
    om = _rate(eq, bulk, p[:, 0], [p[:, 2], p[:, 3]])
    eye = torch.eye(9, dtype=torch.float64)
    om = torch.as_tensor(om).reshape(-1, 1, 1)
    A = eye + om * (J - eye)
    ph = -(p[:, 4:5] * torch.from_numpy(c[:, 0]) + p[:, 5:6] * torch.from_numpy(c[:, 1]))
    return (torch.polar(torch.ones_like(ph), ph)[:, :, None] * A).numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        return _exact_lattice(case, seed)
    if kind == "batch":
        return _exact_batch(case, seed)
    if kind == "eigs":
        lam = np.linalg.eigvals(_vn_matrices(case["eq"], case["bulk"], _eig_params(case, seed)))
        return np.take_along_axis(lam, np.argsort(-np.abs(lam), axis=1, kind="stable"), axis=1)
    # the search over every wave vector takes minutes in NumPy
    return None
