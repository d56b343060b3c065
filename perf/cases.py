"""The work this library is used for, as cases that can be timed and compared.

Every case is one pass through the package's public entry points
(``solver.Solver``, ``solver.Batch``, ``autograd.rollout``) on seeded synthetic
inputs with the shapes of the paper's runs (arXiv 2105.01865, Sec. 4):

* ``step``      one RK3 step of one box: 2D and 3D, u = 0, imposed shear or a
                turbulent-like flow, FP32 and FP64, periodic, no-flux and
                Dirichlet walls, the split scheme and the standard one;
* ``hotpath``   one coupled step on the fine mesh of a two-mesh run: coarse
                velocity in, transfer, RK3 step, mass and free energy;
* ``coupling``  what a Navier-Stokes solver exchanges with the fine mesh:
                coarse velocity in, fine velocity out, and C, rho, mu and the
                surface tension back on the coarse mesh;
* ``batch``     one step of many independent boxes of uneven sizes;
* ``adjoint``   a rollout and its gradients in the initial field and in the
                mobility.

``exact`` restates each pass in plain float64 torch: whole-array stencils, and
line solves by Fourier transforms of the (mirrored) lines.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2105_01865_gb300 import inputs, stability
from paper_2105_01865_gb300.autograd import rollout
from paper_2105_01865_gb300.solver import Batch, Solver

PERIODIC, NOFLUX, DIRICHLET = 0, 1, 2
DEVICE = "cuda:0"


def listed():
    return [
        # the 2D scheme (a single plane) in a stirred box: the smallest call, launches count
        _step("plane_256_f32", 256, 256, 1, "ppp", "random", "f32", ndrops=6, w=2.0),
        # one drop at rest in a periodic 64^3 box, plain method and precision form: small boxes
        _step("drop_64_f64", 64, 64, 64, "ppp", "none", "f64", ndrops=1),
        _step("drop_64_f32", 64, 64, 64, "ppp", "none", "f32", ndrops=1),
        # the drop in shear between walls, precision form and plain method: the ordinary run
        _step("shear_256_f32", 256, 256, 128, "ppn", "shear", "f32", ndrops=1),
        _step("shear_256_f64", 256, 256, 128, "ppn", "shear", "f64", ndrops=1),
        # an odd box closed on all sides: no size is a multiple of anything
        _step("ragged_211_f32", 211, 157, 93, "nnn", "random", "f32", ndrops=20),
        # the single-resolution convection cell: C held at 0 on its plates, lines of 500 cells
        _step("cell_500_f32", 500, 500, 500, "ppd", "random", "f32", ndrops=200),
        # the explicit comparison scheme on the shear box
        _step("standard_256_f32", 256, 256, 128, "ppn", "shear", "f32", ndrops=1, scheme="standard"),
        # the two-mesh run: 1000 drops, 1024 x 1024 x 512 over 256 x 256 x 128 (the largest box)
        _two_mesh("hotpath_1024", "hotpath", 1024, 1024, 512, 256, 256, 128, "ppn", 1000),
        # the exchange of the two meshes at half that size
        _two_mesh("coupling_512", "coupling", 512, 512, 256, 128, 128, 64, "ppn", 200),
        # 64 uneven periodic boxes advanced together
        {"name": "batch_64", "kind": "batch", "nbox": 64, "sizes": "32,48,64,96,128", "box_seed": 4},
        # gradients of a 50-step rollout, checkpoints every 10 steps
        {"name": "adjoint_128", "kind": "adjoint", "nx": 128, "ny": 128, "nz": 128, "bc": "ppp", "prec": "f32",
         "ndrops": 8, "nsteps": 50, "ckpt": 10},
    ]


def _step(name, nx, ny, nz, bc, flow, prec, ndrops, w=4.0, scheme="split"):
    c = {"kind": "step", "nx": nx, "ny": ny, "nz": nz, "bc": bc, "flow": flow, "prec": prec, "ndrops": ndrops, "w": w,
         "scheme": scheme}
    return dict(c, name=name) if name else c


def _two_mesh(name, kind, nx, ny, nz, ncx, ncy, ncz, bc, ndrops):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "ncx": ncx, "ncy": ncy, "ncz": ncz, "bc": bc, "prec": "f32",
         "ndrops": ndrops}
    return dict(c, name=name) if name else c


def _size(rng, lo, hi):
    """A size in [lo, hi], spread over its logarithm: as often one that meshes are built with (a multiple
    of 16) as any other, odd ones included."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(n / 16)) * 16 if rng.random() < 0.5 else int(round(n))))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["hotpath"] * 2 + ["coupling", "batch", "adjoint"])
    if kind == "step":
        prec = rng.choice(["f32", "f32", "f64"])
        hi = 512 if prec == "f32" else 256
        nx, ny, nz = _size(rng, 24, hi), _size(rng, 24, hi), _size(rng, 24, hi)
        if rng.random() < 0.15:
            return _step("", _size(rng, 64, 1024), _size(rng, 64, 1024), 1, rng.choice(["ppp", "pnp", "nnp"]), "random",
                         prec, ndrops=rng.randint(1, 8), w=2.0)
        if rng.random() < 0.15:
            nx = _size(rng, 513, 1024)  # long lines
            ny, nz = min(ny, 256), min(nz, 128)
        bc = rng.choice(["ppp", "ppn", "ppd", "pnn", "nnn"])
        flow = rng.choice(["none", "random", "random", "shear"] if bc[2] != "p" else ["none", "random"])
        scheme = "standard" if bc[2] != "d" and rng.random() < 0.15 else "split"
        return _step("", nx, ny, nz, bc, flow, prec, ndrops=rng.randint(1, 40), scheme=scheme)
    if kind in ("hotpath", "coupling"):
        r = rng.choice([2, 3, 4])  # fine cells per coarse cell
        hi = (1024, 1024, 512) if kind == "hotpath" else (512, 512, 256)
        n = [_size(rng, 64, h) for h in hi]
        nc = [max(4, int(round(m / r))) for m in n]
        return _two_mesh("", kind, *n, *nc, rng.choice(["ppn", "ppn", "nnn", "ppp"]), rng.randint(10, 300))
    if kind == "batch":
        sizes = rng.choice(["32,48,64,96,128", "24,40,64", "64,96,128,160", "30,50,70,90"])
        return {"kind": "batch", "nbox": rng.randint(8, 64), "sizes": sizes, "box_seed": rng.randint(1, 10 ** 6)}
    n = [_size(rng, 32, 128) for _ in range(3)]
    nsteps = rng.randint(5, 30)
    return {"kind": "adjoint", "nx": n[0], "ny": n[1], "nz": n[2], "bc": rng.choice(["ppp", "ppn", "nnn"]),
            "prec": rng.choice(["f32", "f32", "f64"]), "ndrops": rng.randint(1, 8), "nsteps": nsteps,
            "ckpt": rng.choice([2, 5, 10])}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

_stream = None


def _one_stream():
    """The stream that a program with one solver at a time has it work on."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream(DEVICE)
    return _stream


def _bcs(case):
    return tuple({"p": PERIODIC, "n": NOFLUX, "d": DIRICHLET}[b] for b in case["bc"])


def _dtype(case):
    return torch.float64 if case["prec"] == "f64" else torch.float32


def _drops(shape, h, centres, radii, cn, dtype):
    """C = the largest of the drops' tanh profiles (each touches the cells within 8 Cn of it)."""
    nz, ny, nx = shape
    C = torch.zeros(shape, dtype=dtype, device=DEVICE)
    for c, R in zip(centres, radii):
        lo = [max(int((x - R - 8 * cn) / h), 0) for x in c]
        hi = [min(int((x + R + 8 * cn) / h) + 2, n) for x, n in zip(c, (nx, ny, nz))]
        x, y, z = ((torch.arange(a, b, dtype=torch.float64, device=DEVICE) + 0.5) * h - o for a, b, o in zip(lo, hi, c))
        if nz == 1:
            z = z * 0
        r = torch.sqrt(z[:, None, None] ** 2 + y[None, :, None] ** 2 + x[None, None, :] ** 2)
        p = 0.5 * (1 + torch.tanh((R - r) / (2 * math.sqrt(2) * cn)))
        b = C[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]]
        torch.maximum(b, p.to(dtype), out=b)
    return C


def _edge_basis(n_modes, x, L, periodic, zero):
    """Modes along a line at x: Fourier where it is periodic, else sines (zero at the walls) or cosines."""
    k = torch.arange(0 if not periodic else -n_modes, n_modes + 1, dtype=torch.float64, device=DEVICE)
    if periodic:
        ph = 2 * math.pi * k[:, None] * x[None, :] / L
        return k, torch.where(k[:, None] < 0, torch.sin(ph), torch.cos(ph))
    ph = math.pi * k[:, None] * x[None, :] / L
    return k, (torch.sin(ph) if zero else torch.cos(ph))


def _flow(faces, bc, rng, dtype, kmax=6, umax=1.0):
    """A divergence-free face velocity: the discrete curl of a random vector potential on the cell edges with
    a |k|^(-11/6) spectrum, zero through the walls, scaled to umax."""
    f = [torch.as_tensor(a, dtype=torch.float64, device=DEVICE) for a in faces]
    mid = [0.5 * (a[1:] + a[:-1]) for a in f]
    width = [a[1:] - a[:-1] for a in f]
    L = [float(a[-1]) for a in f]
    A = []
    for c in range(3):  # component c lives at the middle along c and on the faces along the others
        parts = [_edge_basis(kmax, mid[d] if d == c else f[d], L[d], bc[d] == PERIODIC, d != c) for d in range(3)]
        kk = torch.sqrt(sum(p[0].reshape([-1 if e == d else 1 for e in range(3)]) ** 2 for d, p in enumerate(parts)))
        amp = torch.where((kk >= 1) & (kk <= kmax), kk.clamp(min=1) ** (-11 / 6), torch.zeros_like(kk))
        co = amp * torch.as_tensor(rng.standard_normal(tuple(kk.shape)), device=DEVICE)
        t = torch.einsum("xyz,zk->xyk", co, parts[2][1])
        t = torch.einsum("xyk,yj->xkj", t, parts[1][1])
        A.append(torch.einsum("xkj,xi->kji", t, parts[0][1]))
    dx, dy, dz = width[0][None, None, :], width[1][None, :, None], width[2][:, None, None]
    u = A[2].diff(dim=1) / dy - A[1].diff(dim=0) / dz
    v = A[0].diff(dim=0) / dz - A[2].diff(dim=2) / dx
    w = A[1].diff(dim=2) / dx - A[0].diff(dim=1) / dy
    if len(mid[2]) == 1:
        w = torch.zeros_like(w)
    vel = [a[tuple(slice(0, a.shape[e] - 1) if e == 2 - d and bc[d] == PERIODIC else slice(None) for e in range(3))]
           for d, a in enumerate((u, v, w))]
    s = umax / max(float(a.abs().max()) for a in vel)
    return tuple((a * s).to(dtype).contiguous() for a in vel)


def _problem(case, seed):
    """Mesh, constants, initial field and velocity of a case: what the solver is built from."""
    rng = np.random.default_rng(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    shape, bc, dtype = (nz, ny, nx), _bcs(case), _dtype(case)
    two = nz == 1
    h = 1.0 / (min(nx, ny) if two else min(nx, ny, nz))
    cn = 0.75 * h
    box = (nx * h, ny * h) if two else (nx * h, ny * h, nz * h)
    nd, gap = case["ndrops"], 4 * cn
    side = (math.prod(box) / nd) ** (1 / len(box))
    rmax = min(0.3 * side, 0.25 * min(box))
    rmin = min(max(0.3 * rmax, 2 * h), rmax)
    if nd == 1:  # one drop about the middle
        centres, radii = [np.array([0.5 * b + rng.uniform(-1, 1) * h for b in box])], [0.2 * min(box)]
    elif two:
        radii = [float(rng.uniform(rmin, rmax)) for _ in range(nd)]
        centres = [np.array([rng.uniform(R + gap, b - R - gap) for b in box]) for R in radii]
    else:
        centres, radii = inputs.random_drops(rng, nd, box, rmin, rmax, gap, (True,) * len(box), max_tries=4 * nd + 40)
    if not centres:
        centres, radii = [0.5 * np.array(box)], [0.25 * min(box)]
    if two:
        centres = [np.append(c, 0.5 * h) for c in centres]
    C = _drops(shape, h, centres, radii, cn, dtype)
    pe = 0.9 / cn if case.get("flow", "random") != "none" else 1e3
    w = case.get("w", 4.0)
    standard = case.get("scheme") == "standard"
    # a margin from the linear bound; half of it where the trajectory is differentiated
    bound = stability.stable_dt_standard if standard else stability.stable_dt
    dt = (0.5 if case["kind"] == "adjoint" else 0.8) * (bound(shape, h, bc, cn, pe, max_modes=12) if standard else
                bound(shape, h, bc, cn, pe, w=w, max_modes=12))
    p = dict(shape=shape, h=h, bc=bc, cn=cn, pe=pe, dt=dt, w=w, C=C, rng=rng, dtype=dtype, vel=None)
    if case.get("flow", "none") != "none":
        p["dt"] = min(dt, 0.5 * h)
        if case["flow"] == "shear":
            nf = [n + (b != PERIODIC) for n, b in zip((nx, ny, nz), bc)]
            zc = (torch.arange(nz, dtype=torch.float64, device=DEVICE) + 0.5) * h
            u = (zc / (nz * h) - 0.5)[:, None, None].expand(nz, ny, nf[0]).to(dtype).contiguous()
            if bc[0] != PERIODIC:
                u[:, :, 0] = u[:, :, -1] = 0
            p["vel"] = (u, torch.zeros((nz, nf[1], nx), dtype=dtype, device=DEVICE),
                        torch.zeros((nf[2], ny, nx), dtype=dtype, device=DEVICE))
        else:
            p["vel"] = _flow([np.arange(n + 1) * h for n in (nx, ny, nz)], bc, rng, dtype)
    if "ncx" in case:
        p["dt"] = min(dt, 0.5 * h)
        faces = []
        for d, (n, nc) in enumerate(zip((nx, ny, nz), (case["ncx"], case["ncy"], case["ncz"]))):
            f = inputs.stretched_faces(nc, n * h, 2.0) if d == 2 and bc[d] != PERIODIC else inputs.uniform_faces(nc, n * h)
            f[0], f[-1] = 0.0, n * h
            faces.append(f)
        p["faces"] = faces
        p["vel"] = _flow(faces, bc, rng, dtype)
    return p


def _boxes(case, seed):
    """The boxes of a batch: sizes and constants from the case, drops from the seed."""
    srng, rng = np.random.default_rng(case["box_seed"]), np.random.default_rng(seed)
    sizes = [int(s) for s in case["sizes"].split(",")]
    dts, boxes = {}, []
    for _ in range(case["nbox"]):
        n = int(srng.choice(sizes))
        h = 1.0 / n
        cn, pe = float(srng.uniform(0.5, 1.0)) * h, float(10 ** srng.uniform(2, 4))
        shape, bc = (n, n, n), (PERIODIC,) * 3
        centres, radii = inputs.random_drops(rng, int(srng.integers(1, 9)), (1.0, 1.0, 1.0), 0.08, 0.25, 4 * cn,
                                             (True,) * 3, max_tries=60)
        dt = 0.8 * stability.stable_dt(shape, h, bc, cn, pe, max_modes=8)
        boxes.append(dict(shape=shape, h=h, bc=bc, cn=cn, pe=pe, dt=dt,
                          C=_drops(shape, h, centres, radii, cn, torch.float32).cpu()))
    return boxes


def _solver(p, case):
    return Solver(p["shape"], p["h"], p["bc"], p["cn"], p["pe"], p["dt"], p["C"], precision=case["prec"], w=p["w"],
                  advect=p["vel"] is not None, coarse_faces=p.get("faces"), stream=_one_stream(),
                  scheme=case.get("scheme", "split"))


def prepare(case, seed):
    if case["kind"] == "batch":
        return {"kind": "batch", "batch": Batch(_boxes(case, seed), stream=_one_stream())}
    p = _problem(case, seed)
    if case["kind"] == "adjoint":
        target = p["C"].roll(2, dims=2)  # the drops, moved by two cells
        return {"kind": "adjoint", "p": p, "target": target, "M": torch.tensor(1.0 / p["pe"], dtype=p["dtype"]),
                "nsteps": case["nsteps"], "ckpt": case["ckpt"], "prec": case["prec"]}
    s = _solver(p, case)
    if case["kind"] == "step":
        if p["vel"] is not None:
            s.set_velocity_fine(*p["vel"])
        s.sync()
        return {"kind": "step", "solver": s}
    s.sync()
    return {"kind": case["kind"], "solver": s, "vel": p["vel"]}


def run(state):
    kind = state["kind"]
    if kind == "step":
        state["solver"].step(1)
        return [state["solver"].C]
    if kind == "hotpath":
        s = state["solver"]
        s.set_velocity_coarse(*state["vel"])
        s.interp_to_fine()
        s.step(1)
        m, e = s.diagnostics()
        return [s.C, m, e]
    if kind == "coupling":
        s = state["solver"]
        s.set_velocity_coarse(*state["vel"])
        s.interp_to_fine()
        fine = s.velocity_fine()
        back = s.restrict_to_coarse(0.05, 1.5)
        return [*fine, *(back[k] for k in ("C", "rho", "mu", "Fx", "Fy", "Fz"))]
    if kind == "batch":
        state["batch"].step(1)
        return list(state["batch"].C)
    p = state["p"]
    C0 = p["C"].detach().requires_grad_(True)
    M = state["M"].detach().requires_grad_(True)
    CT = rollout(C0, M, p["shape"], p["h"], p["bc"], p["cn"], p["dt"], state["nsteps"], ckpt_every=state["ckpt"],
                 precision=state["prec"])
    (p["h"] ** 3 * (CT - state["target"]) ** 2).sum().backward()
    return [CT.detach(), C0.grad, M.grad]


def work(case):
    """Bytes: every field that goes in, read once, and every one that comes out, written once. Operations:
    the formulas' own, 264 a cell and substep with advection, 60 without, 9 a cell for each line solve."""
    if case["kind"] == "batch":
        cells = sum(math.prod(b) for b in _batch_shapes(case))
        return {"bytes": 8.0 * cells, "flops": 3.0 * (60 + 27) * cells}
    cells = case["nx"] * case["ny"] * case["nz"]
    e = 8 if case["prec"] == "f64" else 4
    if case["kind"] == "adjoint":  # the rollout, and its reverse at twice the work; C0, target in, C_T, gradient out
        return {"bytes": 4.0 * e * cells, "flops": 3.0 * 3 * (60 + 27) * cells * case["nsteps"]}
    if case["kind"] == "step":
        flow = case["flow"] != "none"
        return {"bytes": float(e * cells * (5 if flow else 2)), "flops": 3.0 * ((264 if flow else 60) + 27) * cells}
    coarse = case["ncx"] * case["ncy"] * case["ncz"]
    if case["kind"] == "hotpath":  # C in and out; the fine velocity need not be stored
        return {"bytes": float(e * (2 * cells + 3 * coarse)), "flops": (3.0 * (264 + 27) + 3 * 10 + 25) * cells}
    return {"bytes": float(e * (4 * cells + 9 * coarse)), "flops": 3.0 * 10 * cells + 50.0 * cells}


def _batch_shapes(case):
    rng = np.random.default_rng(case["box_seed"])
    sizes, got = [int(s) for s in case["sizes"].split(",")], []
    for _ in range(case["nbox"]):
        n = int(rng.choice(sizes))
        rng.uniform(0.5, 1.0), rng.uniform(2, 4), rng.integers(1, 9)
        got.append((n, n, n))
    return got


# ---------------------------------------------------------------------------
# The same in float64 torch
# ---------------------------------------------------------------------------

GAMMA, RHO = (8 / 15, 5 / 12, 3 / 4), (0.0, -17 / 60, -5 / 12)


def _ghosts(f, d, g, bc):
    """f with g ghost cells on both ends of direction d: wrapped, mirrored, or mirrored with the other sign."""
    a, n = 2 - d, f.shape[2 - d]
    i = torch.arange(-g, n + g, device=f.device)
    if bc[d] == PERIODIC:
        return f.index_select(a, i % n)
    out = f.index_select(a, torch.where(i < 0, -1 - i, torch.where(i >= n, 2 * n - 1 - i, i)))
    if bc[d] == DIRICHLET:
        sign = torch.where((i < 0) | (i >= n), -1.0, 1.0).to(f.dtype)
        out = out * sign.reshape([-1 if e == a else 1 for e in range(3)])
    return out


def _lap(f, h, bc):
    out = torch.zeros_like(f)
    for d in range(3):
        a, n = 2 - d, f.shape[2 - d]
        p = _ghosts(f, d, 1, bc)
        out = out + (p.narrow(a, 2, n) - 2 * f + p.narrow(a, 0, n)) / h ** 2
    return out


def _fourth(f, d, bc):
    a, n = 2 - d, f.shape[2 - d]
    p = _ghosts(f, d, 2, bc)
    s = [p.narrow(a, k, n) for k in range(5)]
    return s[0] - 4 * s[1] + 6 * s[2] - 4 * s[3] + s[4]


def _weno(v1, v2, v3, v4, v5, eps):
    b = [13 / 12 * (v1 - 2 * v2 + v3) ** 2 + (v1 - 4 * v2 + 3 * v3) ** 2 / 4,
         13 / 12 * (v2 - 2 * v3 + v4) ** 2 + (v2 - v4) ** 2 / 4,
         13 / 12 * (v3 - 2 * v4 + v5) ** 2 + (3 * v3 - 4 * v4 + v5) ** 2 / 4]
    a = [g / (eps + x) ** 2 for g, x in zip((0.1, 0.6, 0.3), b)]
    q = a[0] * (2 * v1 - 7 * v2 + 11 * v3) + a[1] * (-v2 + 5 * v3 + 2 * v4) + a[2] * (2 * v3 + 5 * v4 - v5)
    return q / (6 * (a[0] + a[1] + a[2]))


def _divergence(C, vel, h, bc, eps=1e-6):
    out = torch.zeros_like(C)
    for d in range(3):
        a, n = 2 - d, C.shape[2 - d]
        p = _ghosts(C, d, 3, bc)
        s = [p.narrow(a, k, n) for k in range(6)]  # cells f-3 .. f+2 about the lower face of each cell
        u = vel[d].narrow(a, 0, n).to(torch.float64)
        F = u * torch.where(u >= 0, _weno(*s[:5], eps), _weno(*reversed(s[1:]), eps))
        if bc[d] == PERIODIC:
            F = torch.cat([F, F.narrow(a, 0, 1)], a)
        else:
            F.narrow(a, 0, 1).zero_()
            F = torch.cat([F, torch.zeros_like(F.narrow(a, 0, 1))], a)
        out = out + F.diff(dim=a) / h
    return out


def _line_solve(r, d, c, bc):
    """(1 + c [1,-4,6,-4,1])^-1 r along d; walls by continuing the line with its mirror image."""
    a, n = 2 - d, r.shape[2 - d]
    if n == 1:
        return r
    if bc[d] != PERIODIC:
        m = r.flip(a)
        r = torch.cat([r, -m if bc[d] == DIRICHLET else m], a)
    N = r.shape[a]
    th = 2 * math.pi * torch.arange(N // 2 + 1, dtype=torch.float64, device=r.device) / N
    g = (1 / (1 + c * (2 - 2 * torch.cos(th)) ** 2)).reshape([-1 if e == a else 1 for e in range(3)])
    return torch.fft.irfft(torch.fft.rfft(r, dim=a) * g, n=N, dim=a).narrow(a, 0, n)


def _psi_p(C):
    return C * (C * (C - 1.5) + 0.5)


def _step_exact(C, vel, h, bc, cn, M, dt, w, scheme="split"):
    Hp = torch.zeros_like(C)
    kappa = w * cn ** 2 / h ** 4
    for g, r in zip(GAMMA, RHO):
        if scheme == "standard":
            H = M * _lap(_psi_p(C) - cn ** 2 * _lap(C, h, bc), h, bc)
        else:
            H = M * _lap(_psi_p(C), h, bc)
        if vel is not None:
            H = H - _divergence(C, vel, h, bc)
        q = dt * (g * H + r * Hp)
        if scheme != "standard":
            dirs = [d for d in range(3) if C.shape[2 - d] > 1]
            al = (g + r) * dt * M * kappa
            for d in dirs:
                q = q - al * _fourth(C, d, bc)
            for d in dirs:
                q = _line_solve(q, d, al / 2, bc)
        C, Hp = C + q, H
    return C


def _hermite(nodes, period, queries):
    """Dense matrix of the four-point cubic Hermite interpolation with slopes over the neighbouring nodes."""
    n, out = len(nodes), np.zeros((len(queries), len(nodes)))
    for i, x in enumerate(queries):
        j = int(np.searchsorted(nodes, x, side="right")) - 1
        if period is None:
            a = min(max(j, 0), n - 2)
            k = [max(a - 1, 0), a, a + 1, min(a + 2, n - 1)]
            xs = [nodes[m] for m in k]
        else:
            k = [j - 1, j, j + 1, j + 2]
            xs = [nodes[m % n] + period * (m // n) for m in k]
        dx = xs[2] - xs[1]
        t = (x - xs[1]) / dx
        h10, h11 = (t ** 3 - 2 * t ** 2 + t) * dx, (t ** 3 - t ** 2) * dx
        for m, v in ((1, 2 * t ** 3 - 3 * t ** 2 + 1), (2, 3 * t ** 2 - 2 * t ** 3), (2, h10 / (xs[2] - xs[0])),
                     (0, -h10 / (xs[2] - xs[0])), (3, h11 / (xs[3] - xs[1])), (1, -h11 / (xs[3] - xs[1]))):
            out[i, k[m] % n] += v
    return torch.as_tensor(out, device=DEVICE)


def _apply(W, f, d):
    """W along direction d of f."""
    return torch.movedim(torch.tensordot(W, f, dims=([1], [2 - d])), 0, 2 - d)


def _transfer_exact(p):
    n = [p["shape"][2 - d] for d in range(3)]
    vel = [v.to(torch.float64) for v in p["vel"]]
    W = []
    for d in range(3):
        f = np.asarray(p["faces"][d])
        W.append(_hermite(0.5 * (f[1:] + f[:-1]), n[d] * p["h"] if p["bc"][d] == PERIODIC else None,
                          (np.arange(n[d]) + 0.5) * p["h"]))
    out = []
    for d in range(3):
        a, v = 2 - d, vel[d]
        wrapped = torch.cat([v, v.narrow(a, 0, 1)], a) if p["bc"][d] == PERIODIC else v
        dx = torch.as_tensor(np.diff(p["faces"][d]), device=DEVICE).reshape([-1 if e == a else 1 for e in range(3)])
        g = wrapped.diff(dim=a) / dx
        ref = v.narrow(a, 0, 1) if p["bc"][d] == PERIODIC else torch.zeros_like(v.narrow(a, 0, 1))
        for e in sorted(range(3), key=lambda e: n[e]):
            g = _apply(W[e], g, e)
            if e != d:
                ref = _apply(W[e], ref, e)
        s = p["h"] * g.cumsum(dim=a)
        if p["bc"][d] == PERIODIC:
            s = s.narrow(a, 0, n[d] - 1)
        out.append(ref + torch.cat([torch.zeros_like(ref), s], a))
        del g, s
    return out


def _restrict_exact(p, lam_rho, lam_mu):
    C, h, bc, cn = p["C"].to(torch.float64), p["h"], p["bc"], p["cn"]
    phi = _psi_p(C) - cn ** 2 * _lap(C, h, bc)
    fields = [C]
    for d in range(3):
        a, n = 2 - d, C.shape[2 - d]
        q = _ghosts(C, d, 1, bc)
        fields.append(6 * math.sqrt(2) / cn * phi * (q.narrow(a, 2, n) - q.narrow(a, 0, n)) / (2 * h))
    W = []
    for d in range(3):
        f, n = np.asarray(p["faces"][d]), C.shape[2 - d]
        W.append(_hermite((np.arange(n) + 0.5) * h, n * h if bc[d] == PERIODIC else None, 0.5 * (f[1:] + f[:-1])))
    for k, f in enumerate(fields):
        for d in range(3):
            f = _apply(W[d], f, d)
        fields[k] = f
    Cc = fields[0]
    return [Cc, Cc + lam_rho * (1 - Cc), Cc + lam_mu * (1 - Cc), *fields[1:]]


def exact(case, seed):
    if case["kind"] == "batch":
        return [_step_exact(b["C"].to(DEVICE).to(torch.float64), None, b["h"], b["bc"], b["cn"], 1 / b["pe"], b["dt"], 4.0)
                for b in _boxes(case, seed)]
    p = _problem(case, seed)
    args = (p["h"], p["bc"], p["cn"])
    C = p["C"].to(torch.float64)
    if case["kind"] == "step":
        return [_step_exact(C, p["vel"], *args, 1 / p["pe"], p["dt"], p["w"], case["scheme"])]
    if case["kind"] == "coupling":
        return _transfer_exact(p) + _restrict_exact(p, 0.05, 1.5)
    if case["kind"] == "hotpath":
        vel = _transfer_exact(p)
        C = _step_exact(C, vel, *args, 1 / p["pe"], p["dt"], p["w"])
        del vel
        e = 0.25 * C ** 2 * (C - 1) ** 2
        for d in range(3):
            a, n = 2 - d, C.shape[2 - d]
            e = e + p["cn"] ** 2 / 2 * ((_ghosts(C, d, 1, p["bc"]).narrow(a, 2, n) - C) / p["h"]) ** 2
        return [C, p["h"] ** 3 * float(C.sum()), p["h"] ** 3 * float(e.sum())]
    # gradients of the rollout: each step recomputed in the backward pass
    C0 = C.clone().requires_grad_(True)
    M = torch.tensor(1.0 / p["pe"], dtype=p["dtype"]).to(torch.float64).to(DEVICE).requires_grad_(True)
    one = lambda c, m: _step_exact(c, None, *args, m, p["dt"], 4.0)  # noqa: E731
    CT = C0
    for _ in range(case["nsteps"]):
        CT = torch.utils.checkpoint.checkpoint(one, CT, M, use_reentrant=False)
    target = p["C"].roll(2, dims=2).to(torch.float64)
    (p["h"] ** 3 * (CT - target) ** 2).sum().backward()
    return [CT.detach(), C0.grad, M.grad.cpu()]
