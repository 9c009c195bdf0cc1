"""Performance cases of the solver: what a user has it do, through the public
entry points of paper_1509_00680_gb300.gps, over the range of grids, boundary
conditions, problems and precisions that it serves.

A case is a dict of plain values.  listed() gives the fixed ones, draw(rng)
one more of the same ranges, prepare(case, seed) the inputs and handles that a
program has in hand before the call, run(state) one pass and its outputs,
work(case) the bytes and operations that a pass cannot do without, and
exact(case, seed) the outputs as plain torch gives them in 64 bits.

Fields of a case: op (what is called), bc, nx, ny, nz, h (bohr), charges, and
for solves problem, precision and conc (mol/L of a 1:1 electrolyte).
"""
import math
import random

import numpy as np
import torch

from paper_1509_00680_gb300 import gps

EPS0 = 78.36
DELTA = 0.5                     # width of the cavity switching function, bohr
BC = {"free": gps.GPS_BC_FREE, "periodic": gps.GPS_BC_PERIODIC, "surface": gps.GPS_BC_SURFACE,
      "wire": gps.GPS_BC_WIRE}
# Spectrum precisions.  The mixed ones go to the FP32 spectrum four decades
# below the first residual, as a program does that wants its potentials within
# about 1e-10 of the FP64 ones (at the default of two decades: about 1e-8).
SWITCH = 1e-4
PRECISION = {"fp64": gps.GPS_FP64, "mixed": gps.GPS_MIXED, "df64": gps.GPS_DF64,
             "mixed_df64": gps.GPS_MIXED_DF64}


def _case(name, op, bc, n, h=0.3, charges=20, **kw):
    return dict(name=name, op=op, bc=bc, nx=n[0], ny=n[1], nz=n[2], h=h, charges=charges, **kw)


def listed():
    return [
        # one vacuum solve of a small cell, as a plugin calls it every step: launch latency
        _case("vacuum_periodic_30x24x20_fp64", "vacuum", "periodic", (30, 24, 20), h=0.4, charges=4),
        # the preconditioner on a molecule's odd-sized box (padded lengths 150, 180, 128)
        _case("precondition_free_75x90x64_fp64", "precondition", "free", (75, 90, 64), precision="fp64"),
        # the same step on a large slab with the double-float spectrum
        _case("precondition_surface_160x160x256_df64", "precondition", "surface", (160, 160, 256), charges=64,
              precision="df64"),
        # a single cavity in a 64^3 box, arrays in host memory, the default precision
        _case("gpe_free_64_fp64_host", "solve", "free", (64, 64, 64), charges=1, problem="gpe", precision="fp64",
              conc=0.0, host=True),
        # a cluster in a periodic cell: the default precision, and the fast one
        _case("gpe_periodic_128_fp64", "solve", "periodic", (128, 128, 128), problem="gpe", precision="fp64",
              conc=0.0, host=False),
        _case("gpe_periodic_128_mixed_df64", "solve", "periodic", (128, 128, 128), problem="gpe",
              precision="mixed_df64", conc=0.0, host=False),
        # electrolyte over a slab with a planar interface
        _case("lpb_surface_160x160x256_fp64", "solve", "surface", (160, 160, 256), charges=64, problem="lpb",
              precision="fp64", conc=0.1, host=False),
        # a chain periodic along z in an odd-sized box, FP64 then FP32 spectrum
        _case("lpb_wire_90x80x150_mixed", "solve", "wire", (90, 80, 150), h=0.35, charges=6, problem="lpb",
              precision="mixed", conc=0.3, host=False),
        # a solute in 0.5 M electrolyte, nonlinear: many inner solves
        _case("nlpb_free_128_mixed_df64", "solve", "free", (128, 128, 128), charges=20, problem="nlpb",
              precision="mixed_df64", conc=0.5, host=False),
        # a large solute of 200 charges
        _case("gpe_free_256_mixed_df64", "solve", "free", (256, 256, 256), charges=200, problem="gpe",
              precision="mixed_df64", conc=0.0, host=False),
        # what a DFT code takes after each solve: cavity, polarization charge, v_eps, energies
        _case("dft_periodic_128", "dft", "periodic", (128, 128, 128)),
        # requests of mixed sizes, boundary conditions and problems in flight at the same time
        _case("serve_16_mixed_df64", "serve", "mixed", (96, 96, 96), precision="mixed_df64", conc=0.1, requests=16),
    ]


def _smooth(n):
    for p in (2, 3, 5):
        while n % p == 0:
            n //= p
    return n == 1


# 5-smooth edges; a padded (free) axis takes the odd ones too
_EVEN = [n for n in range(16, 257, 2) if _smooth(n)]
_ANY = [n for n in range(15, 257) if _smooth(n)]


def _free_axes(bc):
    """Axes (x, y, z) that are free, i.e. zero-padded to twice their length."""
    return {"free": (1, 1, 1), "periodic": (0, 0, 0), "surface": (0, 0, 1), "wire": (1, 1, 0)}[bc]


def draw(rng):
    op = rng.choice(["vacuum", "precondition", "precondition", "solve", "solve", "solve", "solve", "dft", "serve"])
    if op == "serve":
        return dict(op=op, bc="mixed", nx=96, ny=96, nz=96, h=0.3, charges=rng.randrange(6, 41),
                    precision=rng.choice(["mixed_df64", "fp64"]), conc=round(10 ** rng.uniform(-2, 0), 4),
                    requests=rng.randrange(2, 13))
    bc = rng.choice(["free", "periodic", "surface", "wire"] if op != "dft" else ["free", "periodic", "surface"])
    problem = rng.choice(["gpe", "gpe", "lpb", "lpb", "nlpb"]) if op == "solve" else None
    # grid points: from the smallest cells to the cases' own sizes, by their logarithm
    lo, hi = {"vacuum": (4e3, 4e6), "precondition": (4e3, 4e6), "dft": (3e4, 4e6)}.get(op, (5e4, 2e6))
    if problem == "nlpb":
        hi = 5e5
    edge = math.exp(rng.uniform(math.log(lo), math.log(hi))) ** (1.0 / 3.0)
    n = []
    for free in _free_axes(bc):
        want = edge * rng.uniform(0.8, 1.25)
        pool = _ANY if free else _EVEN
        n.append(min(pool, key=lambda m: abs(math.log(m / want))))
    case = dict(op=op, bc=bc, nx=n[0], ny=n[1], nz=n[2], h=round(rng.uniform(0.28, 0.4), 3),
                charges=2 * rng.randrange(1, 21))
    if op == "precondition":
        case["precision"] = rng.choice(["fp64", "df64"])
    if op == "solve":
        case.update(problem=problem, precision=rng.choice(["fp64", "mixed", "df64", "mixed_df64"]),
                    conc=round(10 ** rng.uniform(-2, 0), 4) if problem != "gpe" else 0.0,
                    host=rng.random() < 0.25)
    return case


# --------------------------------------------------------------- inputs --

def _charges(case, rng):
    """Gaussian charges (q, sigma, centre) and cavity spheres (radius, centre):
    neutral sets of q in {+-1, +-2}, sigma in [0.8, 1.5], cavities of radius
    1.2 x [2.5, 3.5] that end three widths inside the free faces and leave
    solvent around the solute.  Surface grids hold the charges in a slab below
    the interface, wire grids around the axis."""
    bc, h = case["bc"], case["h"]
    n = (case["nx"], case["ny"], case["nz"])
    free = _free_axes(bc)
    length = [m * h for m in n]
    span = [(m - 1) * h for m in n]
    dmax = 4.2
    for a in range(3):
        if free[a] and not (bc == "surface"):
            dmax = min(dmax, 0.45 * span[a] - 3.0 * DELTA)
    dmax = max(dmax, 0.5)
    lo, hi = [0.0] * 3, list(length)
    for a in range(3):
        if free[a]:
            lo[a], hi[a] = dmax + 3.0 * DELTA, span[a] - dmax - 3.0 * DELTA
            if hi[a] <= lo[a]:
                lo[a] = hi[a] = 0.5 * span[a]
    if bc == "surface":
        lo[2], hi[2] = 0.16 * length[2], 0.26 * length[2]
    count = max(1, case["charges"])
    if bc != "surface":
        volume = length[0] * length[1] * length[2]
        fill = int(0.35 * volume / (4.0 / 3.0 * math.pi * min(3.6, dmax) ** 3))
        count = max(1, min(count, fill))
    if count > 1:
        count -= count % 2
    width = [hi[a] - lo[a] for a in range(3)]
    apart, pos = min(2.5, 0.5 * max(width)) if count > 1 else 0.0, []
    while len(pos) < count:
        for _ in range(200):
            p = [lo[a] + width[a] * rng.random() for a in range(3)]
            if count == 1:
                p = [0.5 * (lo[a] + hi[a]) if free[a] else p[a] for a in range(3)]
            if all(sum((p[a] - o[a]) ** 2 for a in range(3)) >= apart * apart for o in pos):
                pos.append(p)
                break
        else:
            apart *= 0.8
    q = [1.0] if count == 1 else [float(rng.choice((1, 2))) for _ in range(count // 2)]
    if count > 1:
        q = q + [-v for v in q]
        rng.shuffle(q)
    sigma = [rng.uniform(0.8, 1.5) for _ in pos]
    radius = [min(1.2 * rng.uniform(2.5, 3.5), dmax) for _ in pos]
    return list(zip(q, sigma, pos)), list(zip(radius, pos))


def _axis(n, h):
    return torch.arange(n, dtype=torch.float64, device="cuda") * h


def _fields(case, seed):
    """Charge density and dielectric function on the grid, shape (nz, ny, nx)."""
    rng = random.Random(int(seed))
    bc, h = case["bc"], case["h"]
    n = (case["nx"], case["ny"], case["nz"])
    free = _free_axes(bc)
    charges, spheres = _charges(case, rng)
    prof = []
    for a in range(3):
        c = torch.tensor([p[a] for _, _, p in charges], dtype=torch.float64, device="cuda")[:, None]
        s = torch.tensor([v for _, v, _ in charges], dtype=torch.float64, device="cuda")[:, None]
        x = _axis(n[a], h)[None, :]
        images = (0.0,) if free[a] else (-n[a] * h, 0.0, n[a] * h)
        prof.append(sum(torch.exp(-0.5 * ((x - c + m) / s) ** 2) for m in images) / (math.sqrt(2 * math.pi) * s))
    q = torch.tensor([v for v, _, _ in charges], dtype=torch.float64, device="cuda")
    rho = torch.zeros(n[2], n[1] * n[0], dtype=torch.float64, device="cuda")
    for k in range(0, len(charges), 32):                       # 32 charges at a time bound the scratch
        plane = (prof[1][k:k + 32, :, None] * prof[0][k:k + 32, None, :]).reshape(-1, n[1] * n[0])
        rho += (q[k:k + 32, None] * prof[2][k:k + 32]).T @ plane
    rho = rho.reshape(n[2], n[1], n[0]).contiguous()
    if bc == "surface":
        z = _axis(n[2], h)
        cut = 0.5 * (1.0 + torch.erf((z - 0.29 * n[2] * h) / DELTA))
        eps = (1.0 + (EPS0 - 1.0) * cut)[:, None, None].expand(n[2], n[1], n[0]).contiguous()
        return rho, eps
    prod = torch.ones(n[2], n[1], n[0], dtype=torch.float64, device="cuda")
    for radius, p in spheres:
        reach = radius + 6.0 * DELTA
        ix, d2 = [], []
        for a in range(3):
            lo, hi = math.ceil((p[a] - reach) / h), math.floor((p[a] + reach) / h)
            if free[a]:
                lo, hi = max(lo, 0), min(hi, n[a] - 1)
            elif hi - lo >= n[a]:                              # wider than the cell: every point, nearest image
                lo = round(p[a] / h) - n[a] // 2
                hi = lo + n[a] - 1
            i = torch.arange(lo, hi + 1, device="cuda")
            ix.append(i % n[a])
            d2.append((i.double() * h - p[a]) ** 2)
        r = torch.sqrt(d2[2][:, None, None] + d2[1][None, :, None] + d2[0][None, None, :])
        at = (ix[2][:, None, None], ix[1][None, :, None], ix[0][None, None, :])
        prod[at] = prod[at] * (0.5 * (1.0 + torch.erf((r - radius) / DELTA)))
    return rho, 1.0 + (EPS0 - 1.0) * prod


def _residual(case, seed, rho):
    """A PCG residual: smooth like the charge, with structure on the grid scale."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return -4.0 * math.pi * rho + 1e-3 * torch.randn(rho.shape, generator=g, device="cuda", dtype=torch.float64)


def _density(case, seed, rho):
    """Electron density of a solute: falls off smoothly through the sccs window."""
    return rho.abs() + 1e-6


def _request_case(case, seed, i):
    """Request i of a served mix: cubic grids of edge 48, 64 or 96."""
    rng = random.Random("%d %d" % (int(seed), i))
    edge = (48, 64, 48, 96)[i % 4]
    return dict(op="solve", bc=("free", "periodic", "surface")[i % 3], nx=edge, ny=edge, nz=edge, h=case["h"],
                charges=2 * rng.randrange(1, max(2, case["charges"] // 2 + 1)),
                problem=("gpe", "lpb", "gpe", "lpb", "nlpb")[i % 5], precision=case["precision"], conc=case["conc"])


_handles = {}


def _context():
    """The context that a program creates once and keeps."""
    if "context" not in _handles:
        _handles["context"] = gps.Context(0)
    return _handles["context"]


def _server():
    """The server that a program creates once and keeps."""
    if "server" not in _handles:
        _handles["server"] = gps.Server(0)
    return _handles["server"]


def _grid(case):
    return gps.make_grid(case["nx"], case["ny"], case["nz"], case["h"], case["h"], case["h"], BC[case["bc"]])


def _electrolyte(case):
    return gps.make_electrolyte((1, -1), (case["conc"], case["conc"]), 300.0, EPS0) if case["conc"] else None


def prepare(case, seed):
    op = case["op"]
    if op == "serve":
        requests, phis = [], []
        for i in range(case["requests"]):
            one = _request_case(case, seed, i)
            rho, eps = (t.cpu().numpy() for t in _fields(one, "%d%03d" % (int(seed), i)))
            phi = np.zeros_like(rho)
            el = _electrolyte(one) if one["problem"] != "gpe" else None
            o = gps.default_opts(precision=PRECISION[one["precision"]], mixed_switch=SWITCH, max_iter=3000)
            requests.append((gps.make_request(_grid(one), one["problem"], rho, eps, phi, el, o), (rho, eps, phi)))
            phis.append(phi)
        return dict(op=op, server=_server(), requests=requests, phis=phis)
    rho, eps = _fields(case, seed)
    state = dict(op=op, ctx=_context(), grid=_grid(case), eps=eps)
    if op == "vacuum":
        state.update(rho=rho, w=torch.empty_like(rho))
    elif op == "precondition":
        state.update(s=1.0 / torch.sqrt(eps), r=_residual(case, seed, rho), v=torch.empty_like(rho),
                     precision=PRECISION[case["precision"]])
    elif op == "dft":
        # the potential a solve left behind: that of the charge in the bulk solvent
        phi = _vacuum(case, _kernel(case)[0], rho / EPS0)
        state.update(rho=rho, phi=phi, dens=_density(case, seed, rho), out=[torch.empty_like(rho) for _ in range(4)])
    else:
        phi = torch.empty_like(rho)
        if case["host"]:
            rho, eps, phi = rho.cpu().numpy(), eps.cpu().numpy(), phi.cpu().numpy()
        state.update(rho=rho, eps=eps, phi=phi, el=_electrolyte(case), problem=case["problem"], host=case["host"],
                     opts=gps.default_opts(precision=PRECISION[case["precision"]], mixed_switch=SWITCH,
                                           max_iter=3000))
    return state


def run(state):
    op = state["op"]
    if op == "serve":
        srv = state["server"]
        tickets = [srv.submit(r, keep) for r, keep in state["requests"]]
        for t in tickets:
            status, _ = srv.wait(t)
            if status != gps.GPS_OK:
                raise gps.GpsError(status, "served request")
        return state["phis"]
    ctx, grid = state["ctx"], state["grid"]
    if op == "vacuum":
        ctx.vacuum_solve(grid, state["rho"], state["w"])
        return state["w"]
    if op == "precondition":
        ctx.precondition(grid, state["s"], state["r"], state["v"], precision=state["precision"])
        return state["v"]
    if op == "dft":
        eps, deps, pol, veps = state["out"]
        ctx.sccs_eps(state["dens"], eps, deps)
        ctx.polarization_charge(grid, state["rho"], eps, state["phi"], pol)
        ctx.v_eps(grid, deps, state["phi"], veps)
        a, b = ctx.electrostatic_energy(grid, state["rho"], eps, state["phi"])
        return [eps, deps, pol, veps, a, b]
    if state["problem"] == "gpe":
        solve = ctx.gpe_solve_host if state["host"] else ctx.gpe_solve
        solve(grid, state["rho"], state["eps"], state["phi"], state["opts"])
    else:
        solve = ctx.pb_solve_host if state["host"] else ctx.pb_solve
        solve(grid, state["rho"], state["eps"], state["el"], state["problem"], state["phi"], state["opts"])
    return state["phi"]


# ----------------------------------------------------------------- work --

# Typical PCG iterations of a solve to the default tolerance on these inputs:
# what the algorithm takes, whatever the code does in each.
_ITERATIONS = {"gpe": 50, "lpb": 60, "nlpb": 700}


def _points(case):
    n = case["nx"] * case["ny"] * case["nz"]
    f = _free_axes(case["bc"])
    return n, n << sum(f)


def work(case):
    if case["op"] == "serve":
        parts = [work(_request_case(case, 0, i)) for i in range(case["requests"])]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n, padded = _points(case)
    transform = 2 * 2.5 * padded * math.log2(padded)      # forward and inverse transform of a real array
    if case["op"] == "vacuum":
        return {"bytes": 16 * n, "flops": transform}
    if case["op"] == "precondition":
        return {"bytes": 24 * n, "flops": transform}
    if case["op"] == "dft":
        # reads the density, rho and phi; writes four fields; three gradients (of ln eps and phi)
        return {"bytes": 56 * n, "flops": (2 * 3 * 24 + 40) * n}
    return {"bytes": 24 * n, "flops": _ITERATIONS[case["problem"]] * transform}


# ---------------------------------------------------------------- exact --
# Plain torch in 64 bits: the vacuum kernels by their definitions, the
# order-16 stencils and Algorithm 2 as it is printed.

def _cosines(M, K, scale):
    j = torch.arange(M // 2 + 1, dtype=torch.float64, device="cuda")
    k = torch.arange(K, dtype=torch.float64, device="cuda")
    w = torch.full_like(j, 2.0)
    w[0] = w[-1] = 1.0
    return torch.cos(2.0 * math.pi * torch.remainder(k[:, None] * j[None, :], M) / M) * w * scale


def _kernel(case):
    """Transform of the vacuum kernel on the rfftn layout of the padded grid."""
    bc, h = case["bc"], case["h"]
    nx, ny, nz = case["nx"], case["ny"], case["nz"]

    def waves(n, d, real=False):
        f = (torch.fft.rfftfreq if real else torch.fft.fftfreq)(n, d=d, dtype=torch.float64, device="cuda")
        return 2.0 * math.pi * f

    def mirrored(n):
        i = torch.arange(2 * n, device="cuda")
        return torch.minimum(i, 2 * n - i)

    if bc == "periodic":
        kz, ky, kx = waves(nz, h), waves(ny, h), waves(nx, h, True)
        k2 = kz[:, None, None] ** 2 + ky[None, :, None] ** 2 + kx[None, None, :] ** 2
        t = 4.0 * math.pi / k2
        t[0, 0, 0] = 0.0
        return t, k2
    if bc == "surface":
        kz = waves(2 * nz, h)
        sign = 1.0 - 2.0 * (torch.arange(2 * nz, device="cuda") % 2).double()
        kpar = torch.sqrt(waves(ny, h)[:, None] ** 2 + waves(nx, h, True)[None, :] ** 2)[None]
        length = nz * h
        t = 4.0 * math.pi * (1.0 - sign[:, None, None] * torch.exp(-kpar * length))
        t = t / (kpar ** 2 + kz[:, None, None] ** 2)
        t[0, 0, 0] = 2.0 * math.pi * length * length
        return t, None
    mx, my, mz = 4 * nx, 4 * ny, 4 * nz
    kx = 2.0 * math.pi * torch.arange(mx // 2 + 1, dtype=torch.float64, device="cuda") / (mx * h)
    ky = 2.0 * math.pi * torch.arange(my // 2 + 1, dtype=torch.float64, device="cuda") / (my * h)
    if bc == "free":
        R = h * math.sqrt(nx * nx + ny * ny + nz * nz)
        kz = 2.0 * math.pi * torch.arange(mz // 2 + 1, dtype=torch.float64, device="cuda") / (mz * h)
        g = torch.empty(mz // 2 + 1, ny + 1, nx + 1, dtype=torch.float64, device="cuda")
        cx, cy = _cosines(mx, nx + 1, 1.0 / mx), _cosines(my, ny + 1, 1.0 / my)
        for i in range(mz // 2 + 1):                        # plane by plane: the oversampled table is large
            k2 = kz[i] ** 2 + ky[:, None] ** 2 + kx[None, :] ** 2
            plane = 8.0 * math.pi * torch.sin(0.5 * R * torch.sqrt(k2)) ** 2 / k2
            if i == 0:
                plane[0, 0] = 2.0 * math.pi * R * R
            g[i] = cy @ plane @ cx.T
        g = torch.tensordot(_cosines(mz, nz + 1, 1.0 / mz), g, dims=1)
        t = torch.einsum("cz,zyx->cyx", _cosines(2 * nz, nz + 1, 1.0), g)
        t = _cosines(2 * ny, ny + 1, 1.0) @ (t @ _cosines(2 * nx, nx + 1, 1.0).T)
        return t[mirrored(nz)][:, mirrored(ny)].contiguous(), None
    R = h * math.sqrt(nx * nx + ny * ny)
    kperp = torch.sqrt(ky[:, None] ** 2 + kx[None, :] ** 2)
    x = kperp * R
    j0, j1 = torch.special.bessel_j0(x), torch.special.bessel_j1(x)
    t = torch.empty(nz, 2 * ny, nx + 1, dtype=torch.float64, device="cuda")
    cx, cy = _cosines(mx, nx + 1, 1.0 / mx), _cosines(my, ny + 1, 1.0 / my)
    dx, dy = _cosines(2 * nx, nx + 1, 1.0), _cosines(2 * ny, ny + 1, 1.0)
    for i in range(nz // 2 + 1):
        kz = torch.tensor(2.0 * math.pi * i / (nz * h), dtype=torch.float64, device="cuda")
        if i == 0:
            plane = 4.0 * math.pi * (1.0 - j0) / kperp ** 2
            plane[0, 0] = math.pi * R * R
        else:
            a = kz * R
            plane = 4.0 * math.pi / (kperp ** 2 + kz ** 2) * (
                1.0 + x * j1 * torch.special.modified_bessel_k0(a) - a * j0 * torch.special.modified_bessel_k1(a))
        g = dy @ (cy @ plane @ cx.T) @ dx.T
        t[i] = g[mirrored(ny)]
        if i:
            t[nz - i] = t[i]
    return t, None


def _vacuum(case, kernel, sigma):
    f = _free_axes(case["bc"])
    shape = (case["nz"] << f[2], case["ny"] << f[1], case["nx"] << f[0])
    w = torch.fft.irfftn(torch.fft.rfftn(sigma, s=shape) * kernel, s=shape)
    return w[:case["nz"], :case["ny"], :case["nx"]].contiguous()


def _shifted(u, axis, j, wraps):
    n = u.shape[axis]
    i = torch.arange(n, device=u.device) + j
    return u.index_select(axis, i % n if wraps else i.clamp(0, n - 1))


def _coefficient(j):
    return (-1.0) ** (j + 1) * math.factorial(8) ** 2 / (math.factorial(8 - j) * math.factorial(8 + j))


def _wraps(case):
    f = _free_axes(case["bc"])
    return not f[2], not f[1], not f[0]                     # axes of the (nz, ny, nx) array


def _gradient(case, u):
    return [sum(_coefficient(j) / j * (_shifted(u, a, j, w) - _shifted(u, a, -j, w)) for j in range(1, 9)) / case["h"]
            for a, w in enumerate(_wraps(case))]


def _laplacian(case, u):
    out = torch.zeros_like(u)
    for a, w in enumerate(_wraps(case)):
        for j in range(1, 9):
            c = 2.0 * _coefficient(j) / (j * j)
            out += c * (_shifted(u, a, j, w) + _shifted(u, a, -j, w) - 2.0 * u)
    return out / case["h"] ** 2


def _solution(case, rho, eps):
    """Algorithm 2 to the end of its convergence (linear problems)."""
    kernel, k2 = _kernel(case)
    periodic = case["bc"] == "periodic"
    root, s = torch.sqrt(eps), 1.0 / torch.sqrt(eps)
    if periodic:
        q = root * torch.fft.irfftn(-k2 * torch.fft.rfftn(root), s=root.shape)
    else:
        q = root * _laplacian(case, root)
    if case["problem"] == "lpb":
        density = case["conc"] * 1000.0 * 6.02214076e23 * 5.29177210903e-11 ** 3
        lam = (eps - 1.0) / (EPS0 - 1.0) * (8.0 * math.pi * density / (3.1668115634556e-6 * 300.0))
        q = q + lam
        if periodic:
            kernel = kernel.clone()
            kernel[0, 0, 0] = 4.0 * math.pi * float(eps.mean()) / float(lam.mean())
    elif periodic:
        rho = rho - rho.mean()
    r = -4.0 * math.pi * rho
    phi, p, ap = torch.zeros_like(r), torch.zeros_like(r), torch.zeros_like(r)
    vr_prev = None
    for _ in range(400):
        v = s * _vacuum(case, kernel, s * r)
        if periodic and case["problem"] == "gpe":          # iterates stay on sum sqrt(eps) phi = 0
            v = v - (root * v).mean() * s
        av = -q * v - 4.0 * math.pi * r
        if periodic:
            av = av + 4.0 * math.pi * (s * r).mean() * root
        vr = float((v * r).sum())
        beta = 0.0 if vr_prev is None else vr / vr_prev
        p, ap, vr_prev = v + beta * p, av + beta * ap, vr
        alpha = vr / float((p * ap).sum())
        phi, r = phi + alpha * p, r - alpha * ap
        if float(r.norm()) <= 1e-12:
            break
    if periodic and case["problem"] == "gpe":
        phi = phi - (root * phi).sum() / root.sum()
    return phi


def exact(case, seed):
    op = case["op"]
    if op == "serve":
        out = []
        for i in range(case["requests"]):
            one = _request_case(case, seed, i)
            if one["problem"] == "nlpb":
                out.append(None)
                continue
            out.append(_solution(one, *_fields(one, "%d%03d" % (int(seed), i))).cpu().numpy())
        return out
    rho, eps = _fields(case, seed)
    if op == "vacuum":
        return _vacuum(case, _kernel(case)[0], rho)
    if op == "precondition":
        s = 1.0 / torch.sqrt(eps)
        return s * _vacuum(case, _kernel(case)[0], s * _residual(case, seed, rho))
    if op == "dft":
        dens, phi = _density(case, seed, rho), _vacuum(case, _kernel(case)[0], rho / EPS0)
        top, low = 5e-3, 1e-4
        z = 2.0 * math.pi * torch.log(top / dens) / math.log(top / low)
        inside = (dens < top) & (dens > low)
        e = torch.exp((z - torch.sin(z)) / (2.0 * math.pi) * math.log(EPS0))
        d = -e * math.log(EPS0) * (1.0 - torch.cos(z)) / (math.log(top / low) * dens)
        e = torch.where(inside, e, torch.where(dens >= top, torch.ones_like(e), torch.full_like(e, EPS0)))
        d = torch.where(inside, d, torch.zeros_like(d))
        gl, gp = _gradient(case, torch.log(e)), _gradient(case, phi)
        pol = sum(a * b for a, b in zip(gl, gp)) / (4.0 * math.pi) - (e - 1.0) / e * rho
        g2 = sum(a * a for a in gp)
        cell = case["h"] ** 3
        return [e, d, pol, -d * g2 / (8.0 * math.pi), float(0.5 * (rho * phi).sum() * cell),
                float((e * g2).sum() * cell / (8.0 * math.pi))]
    if case["problem"] == "nlpb":
        return None
    phi = _solution(case, rho, eps)
    return phi.cpu().numpy() if case["host"] else phi
