"""What a user of the library has it do, as cases that can be timed and compared.

Every case goes through the Python binding of the C ABI (`rrmhd.Context`, `rrmhd.Server`).  The
states are synthetic, with the ranges of the paper's tests and of `workloads.py`: Riemann problems
with densities over three decades, Lorentz factors up to 10, opacities over six decades and free
streaming up to 0.99; a magnetised 2D blast; a smooth 3D turbulent box.  Grid sizes belong to the
case, states to the seed.
"""
import math
import random

import numpy as np
import torch

from paper_2212_00370_gb300 import rrmhd

GAMMA = 4.0 / 3.0


def listed():
    return [
        # one small solve: the radiative shock tube of the paper (400 cells), the smallest call
        {"name": "shock_tube_fp64", "kind": "tube", "n": 400, "precision": "fp64", "steps": 3},
        # a handful of 1D problems, as in a parameter study's first look
        {"name": "riemann_64_fp64", "kind": "riemann", "n_inst": 64, "precision": "fp64",
         "solver": "pvm", "recon": "vanleer", "steps": 2},
        # an ordinary study in full precision, an uneven number of ragged instances
        {"name": "riemann_1001_fp64", "kind": "riemann", "n_inst": 1001, "precision": "fp64",
         "solver": "pvm", "recon": "vanleer", "steps": 2},
        # the whole batch in the fast form: what the benchmark times
        {"name": "riemann_4096_bulk", "kind": "riemann", "n_inst": 4096, "precision": "fp32_bulk",
         "solver": "pvm", "recon": "vanleer", "steps": 2},
        # the paper's comparison solver and another limiter
        {"name": "riemann_500_radhll", "kind": "riemann", "n_inst": 500, "precision": "fp64",
         "solver": "radhll", "recon": "minmod", "steps": 2},
        # 2D magnetised blast with constrained transport, fast form
        {"name": "blast_2d_bulk", "kind": "blast", "nx": 1024, "ny": 1024, "precision": "fp32_bulk",
         "steps": 2},
        # 3D turbulent box with constrained transport, full precision, odd sides
        {"name": "box_3d_fp64", "kind": "box", "nx": 97, "ny": 101, "nz": 103, "precision": "fp64",
         "steps": 1},
        # a caller with its own time stepping: the fluxes of one direction of a 2D grid
        {"name": "flux_sweep_fp64", "kind": "sweep", "nx": 513, "ny": 767, "dir": 1,
         "precision": "fp64"},
        # ... the implicit radiation-matter solve of its own explicit states
        {"name": "implicit_source", "kind": "implicit", "n": 300007},
        # ... primitives from conserved states, and back
        {"name": "con2prim", "kind": "con2prim", "n": 2000003},
        {"name": "prim2con", "kind": "prim2con", "n": 8000001},
        # a stream of solve requests, 1D and planar 2D, through the serving loop
        {"name": "serving_bulk", "kind": "serve", "n_req": 20, "t_end": 0.004},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tube", "riemann", "riemann", "blast", "box", "sweep", "implicit", "con2prim",
                       "prim2con", "serve"])
    precision = rng.choice(["fp64", "fp32_bulk"])
    if kind == "tube":
        return {"kind": kind, "n": _log_int(rng, 100, 4000), "precision": precision,
                "steps": rng.randint(1, 4)}
    if kind == "riemann":
        top = 1000 if precision == "fp64" else 4000
        return {"kind": kind, "n_inst": _log_int(rng, 16, top), "precision": precision,
                "solver": rng.choice(["pvm", "pvm", "radhll"]),
                "recon": rng.choice(["vanleer", "minmod", "mc", "godunov"]), "steps": rng.randint(1, 2)}
    if kind == "blast":
        top = 500 if precision == "fp64" else 1000
        return {"kind": kind, "nx": _log_int(rng, 64, top), "ny": _log_int(rng, 64, top),
                "precision": precision, "steps": rng.randint(1, 2)}
    if kind == "box":
        return {"kind": kind, "nx": _log_int(rng, 16, 100), "ny": _log_int(rng, 16, 100),
                "nz": _log_int(rng, 16, 100), "precision": precision, "steps": 1}
    if kind == "sweep":
        return {"kind": kind, "nx": _log_int(rng, 64, 700), "ny": _log_int(rng, 64, 700),
                "dir": rng.randint(0, 1), "precision": precision}
    if kind == "implicit":
        return {"kind": kind, "n": _log_int(rng, 1000, 300000)}
    if kind == "serve":
        return {"kind": kind, "n_req": rng.randint(4, 20), "t_end": rng.choice([0.002, 0.003, 0.004])}
    top = 2000000 if kind == "con2prim" else 8000000
    return {"kind": kind, "n": _log_int(rng, 1000, top)}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uni(g, n, lo, hi):
    return lo + (hi - lo) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _log(g, n, lo, hi):
    return 10.0 ** _uni(g, n, lo, hi)


def _direction(g, n):
    d = torch.randn(3, n, generator=g, device="cuda", dtype=torch.float64)
    return d / d.norm(dim=0)


def _states(g, n, Bx=None):
    """n primitive states of the Riemann distribution, with kappa and sigma."""
    V = torch.empty(12, n, device="cuda", dtype=torch.float64)
    V[0] = _log(g, n, -2, 1)
    W = _uni(g, n, 1, 10)
    V[1:4] = torch.sqrt(1 - 1 / W ** 2) * _direction(g, n)
    V[4] = _log(g, n, -3, 1)
    V[5] = _uni(g, n, -1, 1) if Bx is None else Bx
    V[6] = _uni(g, n, -1, 1)
    V[7] = _uni(g, n, -1, 1)
    V[8] = _log(g, n, -3, 1)
    V[9:] = _uni(g, n, 0, 0.99) * V[8] * _direction(g, n)
    return V, _log(g, n, -3, 3), _log(g, n, -3, 2)


def _sizes(n_inst):
    r = random.Random(n_inst)
    return [r.randint(128, 2048) for _ in range(n_inst)]


def _riemann(g, sizes):
    """Ragged 1D Riemann problems, packed: left state in the first half of each instance."""
    m = len(sizes)
    Bx = _uni(g, m, -1, 1)
    VL, kL, sL = _states(g, m, Bx)
    VR, kR, sR = _states(g, m, Bx)
    n = torch.tensor(sizes, device="cuda")
    inst = torch.repeat_interleave(torch.arange(m, device="cuda"), n)
    off = torch.cumsum(n, 0) - n
    pos = torch.arange(inst.numel(), device="cuda") - off[inst]
    left = (2 * pos + 1) < n[inst]

    def pick(a, b):
        return torch.where(left, a[..., inst], b[..., inst]).contiguous()

    return pick(VL, VR), pick(kL, kR), pick(sL, sR)


def _smooth(g, shape, modes=6, kmax=3):
    """Random Fourier modes on the unit periodic box, zero mean and unit deviation (array [z][y][x])."""
    axes = [((torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n) for n in shape]
    k = torch.randint(1, kmax + 1, (modes, len(shape)), generator=g, device="cuda").tolist()
    ph = (2 * math.pi * torch.rand(modes, generator=g, device="cuda", dtype=torch.float64)).tolist()
    f = torch.zeros(*shape, device="cuda", dtype=torch.float64)
    for m in range(modes):
        a = ph[m]
        for d, x in enumerate(axes):
            view = [1] * len(shape)
            view[d] = -1
            a = a + 2 * math.pi * k[m][d] * x.view(view)
        f += torch.cos(a)
    f -= f.mean()
    return f / f.std()


def _blast(g, nx, ny):
    x = (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5) / nx - 0.5
    y = (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5) / ny - 0.5
    hot = (x[None, :] ** 2 + y[:, None] ** 2 < 0.01).reshape(-1)
    V = torch.zeros(12, nx * ny, device="cuda", dtype=torch.float64)
    V[0] = 1.0
    vx, vy = _smooth(g, (ny, nx)).reshape(-1), _smooth(g, (ny, nx)).reshape(-1)
    s = 0.05 / torch.sqrt(vx ** 2 + vy ** 2).max()
    V[1], V[2] = vx * s, vy * s
    V[4] = torch.where(hot, 100.0, 0.1).to(torch.float64)
    V[5] = 0.5
    V[8] = (V[4] / V[0]) ** 4
    kappa = 10.0 ** (1.5 * _smooth(g, (ny, nx)).reshape(-1))
    grid = rrmhd.make_grid(2, (nx, ny), (1.0 / nx, 1.0 / ny), ("periodic", "periodic"))
    return grid, V, kappa, torch.zeros_like(kappa)


def _box(g, nx, ny, nz):
    sh = (nz, ny, nx)
    V = torch.zeros(12, nx * ny * nz, device="cuda", dtype=torch.float64)
    V[0] = torch.exp(0.5 * _smooth(g, sh)).reshape(-1)
    v = torch.stack([_smooth(g, sh) for _ in range(3)])
    V[1:4] = (v * (0.3 / torch.sqrt((v ** 2).sum(0).mean()))).reshape(3, -1)
    vm = V[1:4].norm(dim=0)
    V[1:4] *= torch.clamp(0.95 / vm, max=1.0)
    V[4] = 1.0
    A = [_smooth(g, sh) for _ in range(3)]

    def d(f, ax):  # derivative along x, y, z = array axis 2, 1, 0
        return (torch.roll(f, -1, 2 - ax) - torch.roll(f, 1, 2 - ax)) * (0.5 * (nx, ny, nz)[ax])

    B = torch.stack([d(A[2], 1) - d(A[1], 2), d(A[0], 2) - d(A[2], 0), d(A[1], 0) - d(A[0], 1)])
    V[5:8] = (B * (0.3 / torch.sqrt((B ** 2).sum(0).mean()))).reshape(3, -1)
    V[8] = (V[4] / V[0]) ** 4
    kappa = 10.0 ** (1.0 + _smooth(g, sh)).reshape(-1)
    grid = rrmhd.make_grid(3, (nx, ny, nz), (1.0 / nx, 1.0 / ny, 1.0 / nz), ("periodic",) * 3)
    return grid, V, kappa, 0.1 * kappa


def _conserved(V):
    """(D, S, tau_e, B, E_r, F_r) of primitives, by the textbook formulas in 64 bits."""
    rho, v, p, B = V[0], V[1:4], V[4], V[5:8]
    W = 1 / torch.sqrt(1 - (v ** 2).sum(0))
    vB = (v * B).sum(0)
    b0 = W * vB
    b = B / W + b0 * v
    bsq = (B ** 2).sum(0) / W ** 2 + vB ** 2
    w = rho + GAMMA / (GAMMA - 1) * p + bsq
    U = V.clone()
    U[0] = rho * W
    U[1:4] = w * W ** 2 * v - b0 * b
    U[4] = (rho * (W - 1) * W + (GAMMA / (GAMMA - 1) * p + bsq) * W ** 2) - (p + 0.5 * bsq) - b0 ** 2
    return U


def _context(grids, V, kappa, sigma, **opts):
    ctx = rrmhd.Context(grids, **opts)
    ctx.set_opacity(kappa, sigma)
    ctx.set_state(V)
    return ctx


def _requests(case, g):
    """Host arrays of the requests: 70 % 1D with 256..4096 cells, 30 % planar 2D with sides 128..256."""
    r = random.Random(case["n_req"])
    out = []
    Bx = _uni(g, case["n_req"], -1, 1)
    VL, kL, sL = _states(g, case["n_req"], Bx)
    VR, kR, sR = _states(g, case["n_req"], Bx)
    for i in range(case["n_req"]):
        two_d = i % 10 in (3, 6, 9)
        n = r.randint(128, 256) if two_d else r.randint(256, 4096)
        left = (2 * torch.arange(n, device="cuda") + 1) < n
        if two_d:
            left = left.repeat(n)
            grid = rrmhd.make_grid(2, (n, n), (1.0 / n, 1.0 / n))
        else:
            grid = rrmhd.make_grid(1, (n,), (1.0 / n,))
        V = torch.where(left, VL[:, i:i + 1], VR[:, i:i + 1])
        out.append((grid, V.cpu().numpy(), torch.where(left, kL[i], kR[i]).cpu().numpy(),
                    torch.where(left, sL[i], sR[i]).cpu().numpy()))
    return out


# ------------------------------------------------------------------ cases
def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = {"case": case}
    if kind == "tube":
        n = case["n"]
        left = (2 * torch.arange(n, device="cuda") + 1) < n
        dens, pres, kappa = [float(x) for x in _uni(g, 3, 0.5, 1.5)]
        V = torch.zeros(12, n, device="cuda", dtype=torch.float64)
        V[0] = torch.where(left, dens, 0.125 * dens)
        V[4] = torch.where(left, pres, 0.1 * pres)
        V[8] = (V[4] / V[0]) ** 4
        k = torch.full((n,), kappa, device="cuda", dtype=torch.float64)
        s["V"] = V
        s["ctx"] = _context([rrmhd.make_grid(1, (n,), (1.0 / n,))], V, k, torch.zeros_like(k),
                            gamma=5.0 / 3.0, precision=case["precision"])
    elif kind == "riemann":
        sizes = _sizes(case["n_inst"])
        s["V"], k, sg = _riemann(g, sizes)
        s["ctx"] = _context([rrmhd.make_grid(1, (n,), (1.0 / n,)) for n in sizes], s["V"], k, sg,
                            gamma=GAMMA, precision=case["precision"], solver=case["solver"],
                            recon=case["recon"])
    elif kind == "blast":
        grid, s["V"], k, sg = _blast(g, case["nx"], case["ny"])
        s["ctx"] = _context([grid], s["V"], k, sg, gamma=GAMMA, precision=case["precision"], ct=1)
    elif kind == "box":
        grid, s["V"], k, sg = _box(g, case["nx"], case["ny"], case["nz"])
        s["ctx"] = _context([grid], s["V"], k, sg, gamma=GAMMA, precision=case["precision"], ct=1)
    elif kind == "sweep":
        grid, V, k, sg = _blast(g, case["nx"], case["ny"])
        s["ctx"] = _context([grid], V, k, sg, gamma=GAMMA, precision=case["precision"])
    elif kind == "implicit":
        n = case["n"]
        V, k, sg = _states(g, n)
        s["ctx"] = _context([rrmhd.make_grid(1, (n,), (1.0 / 512,))], V, k, sg, gamma=GAMMA)
        s["U"], s["Z"] = _conserved(V), s["ctx"].prim_z(V)  # warm start: the state before the source
    elif kind == "serve":
        s["req"] = _requests(case, g)
        s["srv"] = rrmhd.Server(max_resident_cells=1000000, gamma=GAMMA, precision="fp32_bulk", ct=1)
    else:
        n = case["n"]
        V, _, _ = _states(g, n)
        s["ctx"] = rrmhd.Context([rrmhd.make_grid(1, (64,), (1.0 / 64,))], gamma=GAMMA)
        if kind == "con2prim":  # warm start 1 % away, as from a neighbouring state
            s["U"], s["Z"] = _conserved(V), s["ctx"].prim_z(V) * _uni(g, n, 0.99, 1.01)
        else:
            s["V"] = V
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "sweep":
        return s["ctx"].flux_sweep(case["dir"])
    if kind == "implicit":
        return s["ctx"].implicit_source(1e-3, s["U"], s["Z"])
    if kind == "con2prim":
        return s["ctx"].con2prim(s["U"], s["Z"])
    if kind == "prim2con":
        return s["ctx"].prim2con(s["V"])
    if kind == "serve":
        ids = [s["srv"].submit(grid, V, k, sg, case["t_end"]) for grid, V, k, sg in s["req"]]
        s["srv"].wait_idle(120.0)
        got = {r["id"]: (V, r["status"], r["steps"], r["t"]) for r, V in s["srv"].poll()}
        got = [got[i] for i in ids]
        return {"V": [x[0] for x in got], "status": np.array([x[1] for x in got]),
                "steps": np.array([x[2] for x in got]), "t": np.array([x[3] for x in got])}
    # a solve from a given state: a new state starts with an empty solver cache
    s["ctx"].set_state(s["V"])
    s["ctx"].imex_step(case["steps"])
    return s["ctx"].get_state()


def _cells(case):
    kind = case["kind"]
    if kind == "riemann":
        return sum(_sizes(case["n_inst"]))
    if kind in ("blast", "sweep"):
        return case["nx"] * case["ny"]
    if kind == "box":
        return case["nx"] * case["ny"] * case["nz"]
    if kind == "serve":
        r = random.Random(case["n_req"])
        return sum(r.randint(128, 256) ** 2 if i % 10 in (3, 6, 9) else r.randint(256, 4096)
                   for i in range(case["n_req"]))
    return case["n"]


def work(case):
    """Bytes: primitives and opacities in, results out, once.  Operations (an addition, product,
    quotient or root is one): about 2000 for a PVM-int-8 face (9 recoveries, 11 fluxes), 400 for a
    Rad-HLL face, 1500 for an implicit solve of a cell, 60 for one conversion, 200 for one recovery."""
    kind, n = case["kind"], _cells(case)
    if kind == "prim2con":
        return {"bytes": 192 * n, "flops": 60 * n}
    if kind == "con2prim":
        return {"bytes": 204 * n, "flops": 200 * n}
    if kind == "implicit":
        return {"bytes": (96 + 24 + 192 + 4) * n, "flops": 1500 * n}
    if kind == "sweep":
        return {"bytes": (96 + 24 + 96) * n, "flops": 2000 * n}
    face = 400 if case.get("solver") == "radhll" else 2000
    dims = {"blast": 2, "box": 3}.get(kind, 1)
    steps = case.get("steps", 1)
    if kind == "serve":  # the 1D and 2D requests take about 0.8 t_end n steps of 2 n^2 faces
        dims, steps = 2, max(1, int(200 * case["t_end"] * 2 / 0.4))
    return {"bytes": (96 + 16 + 192) * n, "flops": 3 * steps * (dims * face + 1500) * n}


def exact(case, seed):
    """The conversions have a closed form; a step, a sweep or a solve is an iteration whose value is
    defined by its own finite differences, so it has none here."""
    kind = case["kind"]
    if kind not in ("con2prim", "prim2con"):
        return None
    V, _, _ = _states(_gen(seed), case["n"])
    return _conserved(V) if kind == "prim2con" else (V, None)
