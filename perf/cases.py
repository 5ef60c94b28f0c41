"""Timed cases of the framework: what a user's program has it do.

A simulation case is one restart of a prepared magnet: m is written (device
tensor), the clock is set back, the magnet is advanced a stated number of
steps by the adaptive solver with its usual cap on the step size, and m (and
the table of energies, where the case samples it) is read back.  The other
cases are the stray field alone, a batch of independent simulations and the
learned demag surrogate's inference and training gradient.

Sizes are those of the repository's own workloads and tests (the 64 x 16
film, the 256 x 256 grain film, the 128 x 128 x 32 ellipsoid, the 68 x 78 x 32
and ragged parity grids, the batched grids, the 512 x 512 surrogate film) and
the next sizes a user reaches for (a ragged 500 x 387 film, a 256 x 256 x 64
block).  ``draw`` spreads the same families over their ranges.

``exact`` restates the method in float64 with plain torch: Newell's cell
averaged demag tensor, an FFT convolution, exchange, anisotropy, interfacial
DMI, Zeeman, the Zhang-Li torque, Dormand-Prince and Bogacki-Shampine steps
with step control, and the Fourier neural operator with autograd.
"""
import itertools
import math

import numpy as np
import torch

from paper_1406_7635_gb300 import mm

MU0 = 4e-7 * math.pi
GAMMA = 1.7595e11
MU_B = 9.2740100783e-24
E_CHARGE = 1.602176634e-19


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: a muMag-style film sampled every 20 steps; launches and latency count
        {"name": "film_64x16", "kind": "film", "nx": 64, "ny": 16, "nz": 1, "steps": 20},
        # a polycrystalline film under a time-dependent field (the paper's grain film)
        {"name": "grains_256x256", "kind": "grains", "nx": 256, "ny": 256, "nz": 1, "steps": 10},
        # a skyrmion-type film of ragged size: interfacial DMI, perpendicular anisotropy
        {"name": "dmi_film_500x387", "kind": "dmi", "nx": 500, "ny": 387, "nz": 1, "steps": 5},
        # the 3-D flagship: vortex in an ellipsoid
        {"name": "ellipsoid_128x128x32", "kind": "ellipsoid", "nx": 128, "ny": 128, "nz": 32, "steps": 5},
        # a ragged 3-D part of several materials with holes
        {"name": "parts_77x93x21", "kind": "parts", "nx": 77, "ny": 93, "nz": 21, "steps": 8},
        # the largest simulation: a block beyond the fused layouts
        {"name": "block_256x256x64", "kind": "ellipsoid", "nx": 256, "ny": 256, "nz": 64, "steps": 2},
        # a racetrack: periodic along the wire, Zhang-Li torque, ragged width
        {"name": "racetrack_256x63", "kind": "wire", "nx": 256, "ny": 63, "nz": 1, "steps": 10},
        # energy minimisation dynamics: third-order solver, precession off, a thin layer stack
        {"name": "relax_96x96x4", "kind": "relax", "nx": 96, "ny": 96, "nz": 4, "steps": 12},
        # the stray field alone, of a magnetisation a program holds on the device
        {"name": "stray_field_128x128x32", "kind": "stray", "nx": 128, "ny": 128, "nz": 32},
        # many small simulations of uneven grids advanced together
        {"name": "batch_64", "kind": "batch", "instances": 64, "ps": 1.0},
        # the learned demag field of one film, as inside an RK stage
        {"name": "fno_forward_512", "kind": "fno", "ny": 512, "nx": 512, "modes": 24, "samples": 1},
        # loss and gradient of one training batch of the surrogate
        {"name": "fno_grad_512x4", "kind": "fno_grad", "ny": 512, "nx": 512, "modes": 24, "samples": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["film", "film", "grains", "dmi", "ellipsoid", "ellipsoid", "parts", "parts", "wire", "relax",
                       "stray", "batch", "fno", "fno_grad"])
    if kind in ("film", "grains", "dmi"):
        nx, ny = _log_int(rng, 20, 640), _log_int(rng, 8, 500)
        return {"kind": kind, "nx": nx, "ny": ny, "nz": 1, "steps": 5 + rng.randrange(8)}
    if kind in ("ellipsoid", "parts", "stray"):
        big = kind == "ellipsoid"
        nx, ny = _log_int(rng, 24, 224 if big else 140), _log_int(rng, 12, 224 if big else 140)
        nz = _log_int(rng, 2, 56 if big else 32)
        c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz}
        if kind != "stray":
            c["steps"] = max(2, min(2 + rng.randrange(4), 8000000 // (nx * ny * nz)))
        return c
    if kind == "wire":
        return {"kind": kind, "nx": 1 << rng.randrange(6, 10), "ny": _log_int(rng, 10, 200), "nz": 1,
                "steps": 4 + rng.randrange(8)}
    if kind == "relax":
        return {"kind": kind, "nx": _log_int(rng, 24, 160), "ny": _log_int(rng, 16, 160), "nz": 1 + rng.randrange(6),
                "steps": 6 + rng.randrange(8)}
    if kind == "batch":
        return {"kind": kind, "instances": _log_int(rng, 8, 64), "ps": round(rng.uniform(0.4, 0.95), 2)}
    ny, nx = _log_int(rng, 96, 512), _log_int(rng, 96, 512)
    if kind == "fno":
        return {"kind": kind, "ny": ny, "nx": nx, "modes": rng.choice([12, 16, 24]), "samples": 1 + rng.randrange(2)}
    return {"kind": kind, "ny": ny, "nx": nx, "modes": rng.choice([12, 16, 24]), "samples": 1 + rng.randrange(4)}


# ---------------------------------------------------------------------------
# inputs, from the seed alone
# ---------------------------------------------------------------------------
def _unit(v, keep):
    n = np.sqrt((v * v).sum(axis=0))
    return np.where(keep & (n > 0), v / np.where(n > 0, n, 1.0), 0.0)


def _magnet(case, seed):
    """Grid, materials by region, start state and solver of a simulation."""
    rng = np.random.default_rng(seed)
    kind, nx, ny, nz = case["kind"], case["nx"], case["ny"], case["nz"]
    shape = (nz, ny, nx)
    p = {"nx": nx, "ny": ny, "nz": nz, "d": (4e-9, 4e-9, 3e-9), "mask": np.ones(shape, np.uint8),
         "region": np.zeros(shape, np.uint8), "anis": False, "zeeman": True, "freq": 0.0, "pbc": (0, 0, 0),
         "precession": True, "method": "rk45", "zhang_li": False, "dt": 1e-13, "scale": None}
    mat = {"msat": 8e5, "aex": 1.3e-11, "alpha": 0.02, "ku1": 0.0, "u": (1.0, 0.0, 0.0), "dind": 0.0,
           "jcur": (0.0, 0.0, 0.0), "xi": 0.0, "b0": (0.0, 0.0, 0.0), "b1": (0.0, 0.0, 0.0)}
    mats = [mat]
    noise = rng.standard_normal((3,) + shape)
    if kind == "film":
        mat["b0"] = (-24.6e-3, 4.3e-3, 0.0)
        m = np.array([1.0, 1.0, 0.1])[:, None, None, None] + 0.05 * noise
    elif kind == "grains":
        p["d"], p["anis"], p["freq"], p["dt"] = (2e-9, 2e-9, 1e-9), True, 1e9, 4e-14
        n = 64
        cx, cy = rng.uniform(0, nx, n), rng.uniform(0, ny, n)
        d2 = ((np.arange(nx)[None, :, None] - cx) ** 2 + (np.arange(ny)[:, None, None] - cy) ** 2)
        p["region"] = np.argmin(d2, axis=2).astype(np.uint8)[None]
        phi, ku = rng.uniform(0, 2 * np.pi, n), rng.uniform(0.5e5, 1.5e5, n)
        mats = [dict(mat, msat=1e6, aex=1.5e-11, alpha=0.1, ku1=ku[i], u=(math.cos(phi[i]), math.sin(phi[i]), 0.0),
                     b1=(10e-3, 0.0, 0.0)) for i in range(n)]
        s = rng.uniform(0.8, 1.0, (n, n))
        p["scale"] = np.triu(s, 1) + np.triu(s, 1).T + np.eye(n)
        m = noise
    elif kind == "dmi":
        p["d"], p["anis"] = (2e-9, 2e-9, 1e-9), True
        mat.update(msat=5.8e5, aex=1.5e-11, alpha=0.3, ku1=7e5, u=(0.0, 0.0, 1.0), dind=3e-3, b0=(0.0, 0.0, 0.05))
        x = np.arange(nx)[None, None, :] + np.zeros(shape)
        a = 2 * np.pi * x / 40.0
        m = np.stack([np.sin(a), np.zeros(shape), np.cos(a)]) + 0.1 * noise
        p["dt"] = 2e-14
    elif kind in ("ellipsoid", "stray"):
        p["d"], p["zeeman"], p["dt"] = (3e-9, 3e-9, 3e-9), False, 5e-14
        mat["alpha"] = 0.01
        z, y, x = np.meshgrid(*[(np.arange(k) + 0.5) / k * 2 - 1 for k in shape], indexing="ij")
        p["mask"] = (x * x + y * y + z * z <= 1.0).astype(np.uint8)
        p["mask"][nz // 2, ny // 2, nx // 2] = 1
        m = np.stack([-y * ny, x * nx, np.full(shape, 4.0)])
        m = m / np.sqrt((m * m).sum(axis=0)) + 0.02 * noise
    elif kind == "parts":
        p["d"], p["anis"], p["dt"] = (2e-9, 2e-9, 2e-9), True, 2e-14
        p["region"] = ((np.arange(nx) * 3) // nx).astype(np.uint8)[None, None, :] + np.zeros(shape, np.uint8)
        p["mask"] = (rng.uniform(size=shape) > 0.05).astype(np.uint8)
        mats = []
        for _ in range(3):
            u = rng.standard_normal(3)
            mats.append(dict(mat, msat=rng.uniform(6e5, 1.1e6), aex=rng.uniform(1.0e-11, 1.6e-11),
                             alpha=rng.uniform(0.05, 0.3), ku1=rng.uniform(0, 3e5), u=tuple(u / np.linalg.norm(u)),
                             b0=tuple(rng.uniform(-0.03, 0.03, 3))))
        m = np.array([0.3, 1.0, 0.2])[:, None, None, None] + 0.3 * noise
    elif kind == "wire":
        p["pbc"], p["zhang_li"], p["zeeman"] = (1, 0, 0), True, False
        mat.update(jcur=(-1e13, 0.0, 0.0), xi=0.05)
        a = np.pi * np.tanh((np.arange(nx) - nx / 3.0) / 5.0) - np.pi * np.tanh((np.arange(nx) - 2 * nx / 3.0) / 5.0)
        a = a / 2 + np.zeros(shape)
        m = np.stack([np.cos(a), np.sin(a), np.full(shape, 0.1)]) + 0.05 * noise
    else:   # relax
        p["precession"], p["method"], p["dt"] = False, "rk23", 1e-13
        mat.update(alpha=1.0, b0=(10e-3, 20e-3, 0.0))
        m = np.array([1.0, 0.5, 0.2])[:, None, None, None] + 0.2 * noise
    p["mats"] = mats
    p["m0"] = _unit(m, p["mask"] != 0).astype(np.float32)
    return p


_BATCH_GRIDS = ((32, 32, 1), (64, 32, 1), (128, 64, 2), (96, 96, 4))


def _batch(case, seed):
    """The batched workload: grids in equal shares, materials, fields, m."""
    rng = np.random.default_rng(seed)
    specs, m0s = [], []
    for i in range(case["instances"]):
        nx, ny, nz = _BATCH_GRIDS[i % len(_BATCH_GRIDS)]
        d = rng.standard_normal(3)
        specs.append({"nx": nx, "ny": ny, "nz": nz, "dx": 4e-9, "dy": 4e-9, "dz": 4e-9,
                      "msat": rng.uniform(4e5, 1.2e6), "aex": rng.uniform(0.8e-11, 2e-11),
                      "alpha": rng.uniform(0.005, 0.5), "bext": list(d / np.linalg.norm(d) * rng.uniform(0, 50e-3))})
        m = np.array([1.0, 0.2, 0.3])[:, None, None, None] + 0.3 * rng.standard_normal((3, nz, ny, nx))
        m0s.append(_unit(m, np.ones((nz, ny, nx), bool)).astype(np.float32))
    return specs, m0s


_WIDTH, _LAYERS = 32, 4


def _network(case, seed):
    """Parameters in the documented flat order P, p, {W, b, R}, Q, q; inputs
    u of a magnetised film and the field-like targets y."""
    rng = np.random.default_rng(seed)
    C, k, S, H, W = _WIDTH, case["modes"], case["samples"], case["ny"], case["nx"]
    prm = [rng.standard_normal(3 * C) / math.sqrt(3), 0.1 * rng.standard_normal(C)]
    for _ in range(_LAYERS):
        prm += [rng.standard_normal(C * C) / math.sqrt(C), 0.1 * rng.standard_normal(C),
                rng.standard_normal(2 * C * C * 2 * k * k) / C]
    prm += [rng.standard_normal(3 * C) / math.sqrt(C), 0.1 * rng.standard_normal(3)]
    g = torch.Generator().manual_seed(int(seed))
    u = torch.randn((S, 3, H, W), generator=g)
    u = 0.3 * u + torch.randn((S, 3, 1, 1), generator=g)
    u = u / u.square().sum(dim=1, keepdim=True).sqrt()
    y = -0.3 * u + 0.05 * torch.randn((S, 3, H, W), generator=g)
    return np.concatenate(prm).astype(np.float32), u.float(), y.float()


# ---------------------------------------------------------------------------
# the program: contexts, plans and device tensors it keeps; one pass
# ---------------------------------------------------------------------------
def _context(p):
    ctx = mm.Context(p["nx"], p["ny"], p["nz"], *p["d"])
    if any(p["pbc"]):
        ctx.set_pbc(*p["pbc"])
    ctx.set_geometry(p["mask"])
    ctx.set_regions(p["region"])
    for r, a in enumerate(p["mats"]):
        ctx.set_material(r, a["msat"], a["aex"], a["alpha"], GAMMA, a["ku1"], 0.0, a["u"], a["dind"], a["jcur"], a["xi"])
        ctx.set_bext(r, a["b0"], a["b1"])
    if p["scale"] is not None:
        for i, j in itertools.combinations(range(len(p["mats"])), 2):
            ctx.set_exchange_scale(i, j, p["scale"][i, j])
    ctx.set_bext_timefn(p["freq"], 0.0)
    ctx.enable_terms(True, True, p["anis"], p["zeeman"], p["precession"])
    if p["zhang_li"]:
        ctx.enable_stt(True, False)
    ctx.set_integrator(p["method"])
    ctx.set_solver(1e-5, 0.8, p["dt"], 1e-20, p["dt"])
    return ctx


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        specs, m0s = _batch(case, seed)
        return {"kind": kind, "batch": mm.Batch(specs), "m0": m0s, "t": 0.0, "span": case["ps"] * 1e-12}
    if kind in ("fno", "fno_grad"):
        prm, u, y = _network(case, seed)
        net = mm.FNO(case["ny"], case["nx"], width=_WIDTH, layers=_LAYERS, modes_x=case["modes"],
                     modes_y=case["modes"], max_batch=case["samples"])
        net.set_params(prm)
        u, y = u.cuda(), y.cuda()
        return {"kind": kind, "net": net, "u": u, "y": y, "out": torch.empty_like(y), "samples": case["samples"]}
    p = _magnet(case, seed)
    m0 = torch.from_numpy(p["m0"]).cuda()
    s = {"kind": kind, "ctx": _context(p), "m0": m0, "out": torch.empty_like(m0), "dt": p["dt"],
         "steps": case.get("steps", 0)}
    return s


def run(s):
    kind = s["kind"]
    if kind == "stray":
        s["ctx"].demag_apply(s["m0"], s["out"])
        return s["out"]
    if kind == "fno":
        s["net"].forward(s["u"], s["out"], s["samples"])
        return s["out"]
    if kind == "fno_grad":
        grad, loss = s["net"].grad(s["u"], s["y"], s["samples"])
        return {"grad": grad, "loss": loss}
    if kind == "batch":
        b = s["batch"]
        for i, m in enumerate(s["m0"]):
            b.set_m(i, m)
        b.set_solver(dt0=2e-14, dt_max=5e-14)
        s["t"] += s["span"]
        b.run(s["t"])
        return np.concatenate([b.get_m(i).ravel() for i in range(b.n)])
    ctx = s["ctx"]
    ctx.set_m_device(s["m0"])
    ctx.set_time(0.0, s["dt"])
    if kind in ("film", "grains"):
        ctx.run(s["steps"] * s["dt"])
        ctx.get_m_device(s["out"])
        e = ctx.get_energies()
        return {"m": s["out"], "energies": [e[k] for k in ("demag", "exch", "anis", "zeeman")]}
    ctx.step(s["steps"])
    ctx.get_m_device(s["out"])
    return {"m": s["out"]}


# ---------------------------------------------------------------------------
# work: what a pass cannot do without
# ---------------------------------------------------------------------------
def _conv_work(nx, ny, nz, pbc=(0, 0, 0)):
    """(bytes, flops) of one demag field: m in, the kernel octant in, B out;
    pruned transforms of the padded lines, 30 flops per frequency point."""
    px, py, pz = (1 if n == 1 else (n if q else 2 * n) for n, q in zip((nx, ny, nz), pbc))
    hx = px // 2 + 1
    lg = lambda v: math.log2(v) if v > 1 else 0.0  # noqa: E731
    one_way = (2.5 * px * lg(px) * 3 * ny * nz + 5 * py * lg(py) * 3 * hx * nz + 5 * pz * lg(pz) * 3 * hx * py)
    flops = 2 * one_way + 30.0 * hx * py * pz
    octant = hx * (py // 2 + 1) * (pz // 2 + 1) * (24 if nz > 1 else 16)
    return 24.0 * nx * ny * nz + octant, flops


def work(case):
    kind = case["kind"]
    if kind == "batch":
        by, fl = 0.0, 0.0
        for i in range(case["instances"]):
            nx, ny, nz = _BATCH_GRIDS[i % len(_BATCH_GRIDS)]
            b, f = _conv_work(nx, ny, nz)
            evals = 6 * math.ceil(case["ps"] * 1e-12 / 5e-14) + 1
            by += evals * (24.0 * nx * ny * nz) + b
            fl += evals * (f + 150.0 * nx * ny * nz)
        return {"bytes": by, "flops": fl}
    if kind in ("fno", "fno_grad"):
        C, k, S, H, W, L = _WIDTH, case["modes"], case["samples"], case["ny"], case["nx"], _LAYERS
        n = H * W
        spectral = 2 * (2.0 * C * H * W * 2 * k + 8.0 * C * H * 2 * k * k) + 8.0 * C * C * 2 * k * k
        flops = S * (12.0 * C * n + L * (spectral + 2.0 * C * C * n + 10.0 * C * n))
        prm = 4.0 * (6 * C + 3 + L * (C * C + C + 4 * C * C * k * k))
        if kind == "fno":
            return {"bytes": S * 24.0 * n + prm, "flops": flops}
        return {"bytes": S * 24.0 * n + 2 * prm, "flops": 3 * flops}
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    by, fl = _conv_work(nx, ny, nz, (1, 0, 0) if kind == "wire" else (0, 0, 0))
    if kind == "stray":
        return {"bytes": by, "flops": fl}
    evals = (3 if kind == "relax" else 6) * case["steps"] + 1
    return {"bytes": evals * by, "flops": evals * (fl + 150.0 * nx * ny * nz)}


# ---------------------------------------------------------------------------
# float64 restatement
# ---------------------------------------------------------------------------
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _newell_f(x, y, z):
    R = torch.sqrt(x * x + y * y + z * z)
    xz, xy = torch.sqrt(x * x + z * z), torch.sqrt(x * x + y * y)
    o = torch.zeros_like(R)
    a = torch.where(xz > 0, 0.5 * y * (z * z - x * x) * torch.asinh(y / torch.where(xz > 0, xz, 1.0)), o)
    b = torch.where(xy > 0, 0.5 * z * (y * y - x * x) * torch.asinh(z / torch.where(xy > 0, xy, 1.0)), o)
    c = torch.where(x * R != 0, x * y * z * torch.atan(y * z / torch.where(x * R != 0, x * R, 1.0)), o)
    return a + b - c + (2 * x * x - y * y - z * z) * R / 6


def _newell_g(x, y, z):
    R = torch.sqrt(x * x + y * y + z * z)
    o = torch.zeros_like(R)

    def ash(u, v, w):   # asinh(u / sqrt(v^2 + w^2)), 0 where the root is 0 (its factor vanishes too)
        q = torch.sqrt(v * v + w * w)
        return torch.where(q > 0, torch.asinh(u / torch.where(q > 0, q, 1.0)), o)

    def at(u, v, w):    # atan(u v / (w R)), its factor w vanishes where w R = 0
        q = w * R
        return torch.where(q != 0, torch.atan(u * v / torch.where(q != 0, q, 1.0)), o)

    return (x * y * z * ash(z, x, y) + y / 6 * (3 * z * z - y * y) * ash(x, y, z) +
            x / 6 * (3 * z * z - x * x) * ash(y, x, z) - z ** 3 / 6 * at(x, y, z) - z * y * y / 2 * at(x, z, y) -
            z * x * x / 2 * at(y, z, x) - x * y * R / 3)


def _tensor(X, Y, Z, d):
    """N (six components) of cell offsets X, Y, Z (float64 tensors, in cells):
    exact within eight largest edges, the tent-weighted dipole beyond."""
    d0, d1, d2 = (v / max(d) for v in d)
    x, y, z = (a.reshape(-1) * e for a, e in zip((X, Y, Z), (d0, d1, d2)))
    out = torch.zeros((6, x.numel()), dtype=torch.float64, device=x.device)
    near = (x * x + y * y + z * z) < 64.0
    xn, yn, zn = x[near], y[near], z[near]
    acc = torch.zeros((6, xn.numel()), dtype=torch.float64, device=x.device)
    for i, j, k in itertools.product((-1, 0, 1), repeat=3):
        w = (2.0 if i == 0 else -1.0) * (2.0 if j == 0 else -1.0) * (2.0 if k == 0 else -1.0)
        a, b, c = xn + i * d0, yn + j * d1, zn + k * d2
        acc[0] += w * _newell_f(a, b, c)
        acc[1] += w * _newell_f(b, a, c)
        acc[2] += w * _newell_f(c, b, a)
        acc[3] += w * _newell_g(a, b, c)
        acc[4] += w * _newell_g(a, c, b)
        acc[5] += w * _newell_g(b, c, a)
    out[:, near] = acc / (4 * math.pi * d0 * d1 * d2)
    far = ~near
    if bool(far.any()):
        xf, yf, zf = x[far], y[far], z[far]
        g, wg = np.polynomial.legendre.leggauss(3)
        pts = [(s * (0.5 + 0.5 * t), 0.5 * w * (0.5 - 0.5 * t)) for t, w in zip(g, wg) for s in (-1, 1)]
        acc = torch.zeros((6, xf.numel()), dtype=torch.float64, device=x.device)
        for (p, wp), (q, wq), (r, wr) in itertools.product(pts, repeat=3):
            a, b, c = xf + p * d0, yf + q * d1, zf + r * d2
            i2 = 1.0 / (a * a + b * b + c * c)
            i3 = i2 * i2.sqrt() * (wp * wq * wr)
            i5 = 3.0 * i3 * i2
            acc[0] += i3 - i5 * a * a
            acc[1] += i3 - i5 * b * b
            acc[2] += i3 - i5 * c * c
            acc[3] -= i5 * a * b
            acc[4] -= i5 * a * c
            acc[5] -= i5 * b * c
        out[:, far] = acc * (d0 * d1 * d2 / (4 * math.pi))
    return out.reshape((6,) + X.shape)


class _Demag:
    """B = -mu0 N * M by a zero-padded (or, along x with one image on each
    side, cyclic) FFT in float64."""

    def __init__(self, n, d, pbc):
        self.n = n
        self.pad = tuple(1 if k == 1 else (k if q else 2 * k) for k, q in zip(n, pbc))
        ax = [torch.arange(k, dtype=torch.float64, device=_dev()) for k in n]
        Z, Y, X = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
        N = _tensor(X, Y, Z, d)
        signs = ((1, 1, 1, -1, -1, 1), (1, 1, 1, -1, 1, -1), (1, 1, 1, 1, -1, -1))   # parity in x, y, z
        if pbc[0]:
            other = _tensor(X - n[0], Y, Z, d)
            other[..., 0] = 0.0
            N = N + other
        for axis in range(3):   # mirror into the padded box: index p - i holds offset -i
            dim, k, p = 3 - axis, n[axis], self.pad[axis]
            if p == 2 * k:
                full = torch.zeros(N.shape[:dim] + (p,) + N.shape[dim + 1:], dtype=torch.float64, device=N.device)
                full.narrow(dim, 0, k).copy_(N)
                if k > 1:
                    sg = torch.tensor(signs[axis], dtype=torch.float64, device=N.device).view(6, 1, 1, 1)
                    full.narrow(dim, k + 1, k - 1).copy_((N.narrow(dim, 1, k - 1) * sg).flip(dim))
                N = full
        self.K = torch.stack([torch.fft.rfftn(N[c]) for c in range(6)])

    def __call__(self, M):
        s = (self.pad[2], self.pad[1], self.pad[0])
        F = [torch.fft.rfftn(M[c], s=s) for c in range(3)]
        nz, ny, nx = M.shape[1:]
        out = []
        for row in ((0, 3, 4), (3, 1, 5), (4, 5, 2)):
            h = torch.fft.irfftn(sum(self.K[k] * f for k, f in zip(row, F)), s=s)
            out.append(-MU0 * h[:nz, :ny, :nx])
        return torch.stack(out)


def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])


_RK = {
    "rk45": ((0, 1 / 5, 3 / 10, 4 / 5, 8 / 9, 1, 1),
             ((), (1 / 5,), (3 / 40, 9 / 40), (44 / 45, -56 / 15, 32 / 9),
              (19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729),
              (9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656),
              (35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84)),
             (71 / 57600, 0, -71 / 16695, 71 / 1920, -17253 / 339200, 22 / 525, -1 / 40), 0.2),
    "rk23": ((0, 0.5, 0.75, 1), ((), (0.5,), (0, 0.75), (2 / 9, 1 / 3, 4 / 9)),
             (-5 / 72, 1 / 12, 1 / 9, -1 / 8), 1 / 3),
}


class _Magnet:
    """Fields, torque and steps of one magnet in float64."""

    def __init__(self, p, demag=None):
        dev = _dev()
        self.p, self.d = p, p["d"]
        reg = torch.from_numpy(p["region"].astype(np.int64)).to(dev)
        self.mag = torch.from_numpy(p["mask"] != 0).to(dev)
        tab = lambda k: torch.tensor([a[k] for a in p["mats"]], dtype=torch.float64, device=dev)  # noqa: E731
        cell = lambda k: tab(k)[reg]                                                             # noqa: E731
        vec = lambda k: tab(k)[reg].permute(3, 0, 1, 2)                                          # noqa: E731
        self.ms = cell("msat") * self.mag
        self.safe = cell("msat")
        self.alpha, self.k1, self.u = cell("alpha"), 2 * cell("ku1") / self.safe, vec("u")
        self.b0, self.b1, self.has_anis = vec("b0"), vec("b1"), p["anis"]
        a = tab("aex") / tab("msat")
        s = torch.ones((len(a), len(a)), dtype=torch.float64, device=dev)
        if p["scale"] is not None:
            s = torch.tensor(p["scale"], dtype=torch.float64, device=dev)
        lut = 2 * s * 2 * a[:, None] * a[None, :] / (a[:, None] + a[None, :])
        self.dind, self.aex = cell("dind"), cell("aex")
        self.own = lut[reg, reg]
        per = p["pbc"]
        self.nb = []   # (tensor dim of m, step, cell size, present, coupling)
        for axis, delta in ((0, self.d[0]), (1, self.d[1]), (2, self.d[2])):
            dim = 2 - axis
            n = reg.shape[dim]
            idx = torch.arange(n, device=dev)
            for step in (1, -1):
                valid = torch.ones(n, dtype=torch.bool, device=dev) if per[axis] else ((idx + step >= 0) & (idx + step < n))
                view = [1, 1, 1]
                view[dim] = n
                present = self.mag.roll(-step, dim) & valid.view(view) & self.mag
                self.nb.append((dim, step, delta, axis, present, lut[reg, reg.roll(-step, dim)]))
        if p["zhang_li"]:
            xi = cell("xi")
            self.zu = MU_B * vec("jcur") / (2 * E_CHARGE * self.safe * (1 + xi * xi))
            self.zc = (1 + xi * self.alpha) / (1 + self.alpha ** 2), (xi - self.alpha) / (1 + self.alpha ** 2)
        self.dmi = bool((self.dind != 0).any())
        self.demag = demag or _Demag((p["nx"], p["ny"], p["nz"]), self.d, per)
        m = torch.from_numpy(p["m0"]).to(dev).double()
        self.m = self._unit(m)

    def _unit(self, m):
        n = m.square().sum(dim=0).sqrt()
        return torch.where(self.mag & (n > 0), m / torch.where(n > 0, n, 1.0), 0.0)

    def parts(self, m, t):
        ex = torch.zeros_like(m)
        values = {}
        for dim, step, delta, axis, present, lut in self.nb:
            v = m.roll(-step, 1 + dim)
            if self.dmi:
                c = step * delta * self.dind / (2 * self.aex)
                ghost = m.clone()
                if axis == 0:
                    ghost[0], ghost[2] = m[0] - c * m[2], m[2] + c * m[0]
                elif axis == 1:
                    ghost[1], ghost[2] = m[1] - c * m[2], m[2] + c * m[1]
                v = torch.where(present, v, ghost)
                ex += torch.where(present, lut, self.own) * (v - m) / delta ** 2
            else:
                v = torch.where(present, v, m)
                ex += lut * (v - m) / delta ** 2
            values[(axis, step)] = v
        f = {"demag": self.demag(self.ms * m), "exch": ex * self.mag}
        f["anis"] = self.k1 * (self.u * m).sum(dim=0) * self.u if self.has_anis else torch.zeros_like(m)
        s = math.sin(2 * math.pi * self.p["freq"] * t)
        f["zeeman"] = (self.b0 + s * self.b1) if self.p["zeeman"] else torch.zeros_like(m)
        if self.dmi:
            gx = (values[(0, 1)] - values[(0, -1)]) / (2 * self.d[0])
            gy = (values[(1, 1)] - values[(1, -1)]) / (2 * self.d[1])
            f["dmi"] = 2 * self.dind / self.safe * torch.stack([gx[2], gy[2], -gx[0] - gy[1]])
        self.values = values
        return f

    def torque(self, m, t):
        B = sum(self.parts(m, t).values())
        mB = _cross(m, B)
        mmB = _cross(m, mB)
        pre = mB if self.p["precession"] else 0.0
        tq = -GAMMA / (1 + self.alpha ** 2) * (pre + self.alpha * mmB)
        if self.p["zhang_li"]:
            h = sum(self.zu[a] * (self.values[(a, 1)] - self.values[(a, -1)]) / (2 * self.d[a]) for a in range(3))
            mh = _cross(m, h)
            tq = tq - (self.zc[0] * _cross(m, mh) + self.zc[1] * mh)
        return tq * self.mag

    def advance(self, steps, t_end, dt0, dt_max, max_err=1e-5):
        c, a, e, ex = _RK[self.p["method"]]
        t, dt, done = 0.0, dt0, 0
        k = [self.torque(self.m, t)]
        while (t < t_end) if t_end is not None else (done < steps):
            h = min(dt, t_end - t) if t_end is not None else dt
            k = k[:1]
            for s in range(1, len(c)):
                y = self.m + sum(h * w * q for w, q in zip(a[s], k) if w)
                k.append(self.torque(y, t + c[s] * h))
            err = sum(h * w * q for w, q in zip(e, k) if w)
            eps = float(err.square().sum(dim=0).sqrt()[self.mag].max())
            factor = 5.0 if eps == 0 else min(5.0, max(0.2, 0.8 * (max_err / eps) ** ex))
            dt = min(h * factor, dt_max)
            if eps <= max_err:
                self.m, t, done, k = self._unit(y), t + h, done + 1, [k[-1]]
                if t_end is not None and t + 1e-6 * h >= t_end:
                    t = t_end
        self.t = t

    def energies(self):
        f = self.parts(self.m, self.t)
        V = self.d[0] * self.d[1] * self.d[2]
        return [float(-(1.0 if k == "zeeman" else 0.5) * (self.ms * self.m * f[k]).sum() * V)
                for k in ("demag", "exch", "anis", "zeeman")]


def _fno(case, seed):
    C, k, S, H, W = _WIDTH, case["modes"], case["samples"], case["ny"], case["nx"]
    flat, u, y = _network(case, seed)
    prm = torch.from_numpy(flat).double().to(_dev()).requires_grad_(True)
    pos = 0

    def take(*shape):
        nonlocal pos
        n = math.prod(shape)
        v = prm[pos:pos + n].view(*shape)
        pos += n
        return v

    def channels(A, v):
        return (A @ v.reshape(S, A.shape[1], H * W)).view(S, A.shape[0], H, W)

    u, y = u.double().to(_dev()), y.double().to(_dev())
    P, p = take(C, 3), take(C)
    v = channels(P, u) + p.view(1, C, 1, 1)
    rows = torch.cat([torch.arange(k), torch.arange(H - k, H)]).to(_dev())
    for l in range(_LAYERS):
        A, b, R = take(C, C), take(C), torch.view_as_complex(take(C, C, 2 * k, k, 2).contiguous())
        F = torch.fft.fft2(v)[:, :, rows, :k]
        O = torch.einsum("oijk,sijk->sojk", R, F)
        wgt = torch.full((k,), 2.0, dtype=torch.float64, device=v.device)
        wgt[0] = 1.0
        full = torch.zeros((S, C, H, W), dtype=torch.complex128, device=v.device)
        full[:, :, rows, :k] = O * wgt
        z = channels(A, v) + b.view(1, C, 1, 1) + torch.fft.ifft2(full).real
        v = torch.nn.functional.gelu(z) if l < _LAYERS - 1 else z
    Q, q = take(3, C), take(3)
    return prm, channels(Q, v) + q.view(1, 3, 1, 1), y


def exact(case, seed):
    kind = case["kind"]
    if kind in ("fno", "fno_grad"):
        if kind == "fno":
            with torch.no_grad():
                return _fno(case, seed)[1]
        prm, out, y = _fno(case, seed)
        loss = (out - y).square().sum() / y.square().sum()
        loss.backward()
        return {"grad": prm.grad, "loss": loss.detach().reshape(())}
    if kind == "batch":
        specs, m0s = _batch(case, seed)
        if len(specs) > 96:
            return None
        kernels, out = {}, []
        for s, m0 in zip(specs, m0s):
            shape = m0.shape[1:]
            p = {"nx": s["nx"], "ny": s["ny"], "nz": s["nz"], "d": (s["dx"], s["dy"], s["dz"]),
                 "mask": np.ones(shape, np.uint8), "region": np.zeros(shape, np.uint8), "anis": False, "zeeman": True,
                 "freq": 0.0, "pbc": (0, 0, 0), "precession": True, "method": "rk45", "zhang_li": False, "scale": None,
                 "mats": [{"msat": s["msat"], "aex": s["aex"], "alpha": s["alpha"], "ku1": 0.0, "u": (1.0, 0.0, 0.0),
                           "dind": 0.0, "jcur": (0.0, 0.0, 0.0), "xi": 0.0, "b0": tuple(s["bext"]),
                           "b1": (0.0, 0.0, 0.0)}], "m0": m0}
            if shape not in kernels:
                kernels[shape] = _Demag((p["nx"], p["ny"], p["nz"]), p["d"], p["pbc"])
            g = _Magnet(p, kernels[shape])
            g.advance(None, case["ps"] * 1e-12, 2e-14, 5e-14)
            out.append(g.m.reshape(-1))
        return torch.cat(out)
    p = _magnet(case, seed)
    g = _Magnet(p)
    if kind == "stray":   # (m is read as it is: the start state is of unit length up to float32 rounding)
        return g.demag(g.ms * torch.from_numpy(p["m0"]).to(_dev()).double())
    if kind in ("film", "grains"):
        g.advance(None, case["steps"] * p["dt"], p["dt"], p["dt"])
        return {"m": g.m, "energies": g.energies()}
    g.advance(case["steps"], None, p["dt"], p["dt"])
    return {"m": g.m}
