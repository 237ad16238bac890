"""The work that users of this framework have it do, as cases that can be timed and compared.

A case is one chunk of a solve through the public entry points: a number of coarse steps
(``Solver.step``, ``Batch.step``), then what the user reads: the fields of every level and,
where there are walls, the surface loads.  Kinds:

  box      a periodic box without walls (Taylor-Green-like vortices): the level step alone,
           laminar or with SA-neg
  tunnel   a box with the inlet, the outlet and the symmetry planes, any size
  naca     a NACA section on a 2:1 multilevel grid: a polar request (16c x 8c box at c/16),
           the small validation case (c/8) or the bench workload (8c x 4c box at c/128)
  batch    several polar requests stepped in lockstep, as the serving loop does
  request  one polar request from the wall polyline to its loads: grid build, upload, steps

Fields come back in the precision that the solve stores its populations in.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2601_18443_gb300 as pkg
from paper_2601_18443_gb300 import workloads as W

FP32, FP16, BF16 = 0, 1, 2
OUT_TYPE = {FP32: torch.float32, FP16: torch.float16, BF16: torch.bfloat16}
BOX_NU = 0.01          # lattice viscosity of the boxes
CS = math.sqrt(1.0 / 3.0)


# --------------------------------------------------------------------------- the cases

def listed():
    return [
        # a unit-test-sized box, a few steps: launches and the queries' latency
        dict(name="box_64x40_laminar_f32", kind="box", nx=64, ny=40, sa=0, store=FP32, steps=20),
        # an ordinary single level whose state stays in L2
        dict(name="box_512x512_sa_f32", kind="box", nx=512, ny=512, sa=1, store=FP32, steps=200),
        # single levels far larger than L2: the HBM-bound forms, with and without SA-neg
        dict(name="box_2048x2048_sa_f32", kind="box", nx=2048, ny=2048, sa=1, store=FP32, steps=300),
        dict(name="box_3008x2792_laminar_f32", kind="box", nx=3008, ny=2792, sa=0, store=FP32, steps=400),
        dict(name="box_1536x2048_sa_bf16", kind="box", nx=1536, ny=2048, sa=1, store=BF16, steps=400),
        # a wind tunnel of odd size: inlet, outlet, symmetry planes, ragged tiles
        dict(name="tunnel_1003x517_sa_f32", kind="tunnel", nx=1003, ny=517, sa=1, store=FP32, steps=300),
        # the small validation airfoil (6 levels to c/256): tiny levels, many launches
        dict(name="naca_c256_f32", kind="naca", grid="small", code="0012", alpha=0.0, Re=1.0e6, levels=6, layers=8,
             store=FP32, steps=50),
        # one chunk of the serving loop's polar requests, at the ends of their range
        dict(name="polar_4lvl_f16", kind="naca", grid="polar", code="2412", alpha=4.0, Re=3.0e6, levels=4, layers=16,
             store=FP16, steps=100),
        dict(name="polar_6lvl_f16", kind="naca", grid="polar", code="4415", alpha=9.5, Re=6.0e6, levels=6, layers=32,
             store=FP16, steps=100),
        # eight resident requests of one level count in lockstep
        dict(name="batch_8x5lvl_f16", kind="batch", members=8, pick=2026, levels=5, layers=24, store=FP16, steps=100),
        # the bench workload: 1.5M nodes, 6 levels to c/4096
        dict(name="naca_c4096_f32", kind="naca", grid="large", code="0012", alpha=10.0, Re=6.0e6, levels=6, layers=56,
             store=FP32, steps=100),
        # a whole request: polyline, grid build, upload, steps, loads
        dict(name="request_7lvl_f16", kind="request", grid="polar", code="0012", alpha=6.0, Re=4.0e6, levels=7,
             layers=32, store=FP16, steps=100),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _code(rng):
    m = rng.randint(0, 4)
    return "%d%d%02d" % (m, rng.randint(2, 5) if m else 0, rng.randint(9, 18))


def draw(rng):
    kind = rng.choice(["box", "box", "tunnel", "naca", "naca", "batch", "request"])
    store = rng.choice([FP32, FP32, FP16, BF16])
    if kind in ("box", "tunnel"):
        nx, ny = _log(rng, 48, 3000), _log(rng, 24, 2800)
        if kind == "box":
            nx, ny = 32 * max(1, round(nx / 32)), 8 * max(1, round(ny / 8))
        else:
            nx, ny = int(nx), int(ny)
        steps = int(_log(rng, 20, max(21, min(500, 3.0e9 / (nx * ny)))))
        return dict(kind=kind, nx=nx, ny=ny, sa=rng.randint(0, 1), store=store, steps=steps)
    polar = dict(levels=rng.randint(4, 7), store=rng.choice([FP32, FP16]), steps=int(_log(rng, 20, 100)))
    polar["layers"] = {4: 16, 5: 24, 6: 32, 7: 32}[polar["levels"]]
    if kind == "batch":
        polar["levels"] = min(polar["levels"], 6)
        return dict(kind=kind, members=rng.randint(2, 8), pick=rng.randint(1, 99999), **polar)
    case = dict(kind=kind, grid="polar", code=_code(rng), alpha=round(rng.uniform(-4.0, 16.0), 3),
                Re=float("%.4g" % _log(rng, 1e6, 1e7)), **polar)
    if kind == "naca" and rng.random() < 0.5:
        case["store"] = FP32
        if rng.random() < 0.5:
            case.update(grid="small", Re=1.0e6, alpha=round(rng.uniform(0.0, 4.0), 3), levels=rng.randint(3, 6),
                        layers=rng.randint(6, 10))
        else:
            case.update(grid="large", Re=6.0e6, code="0012", alpha=10.0, levels=rng.randint(4, 6),
                        layers=rng.randint(20, 56))
    return case


# --------------------------------------------------------------------------- configurations

def _box_config(case):
    U = 0.1 * CS
    return W.base_config(levels=1, nx0=case["nx"], ny0=case["ny"], h0=1.0, Re=U / BOX_NU, Ma=0.1,
                         periodic=int(case["kind"] == "box"), solid_walls=0, turbulence=case["sa"], wall_model=3,
                         store=case["store"])


def _naca_config(case):
    if case["grid"] == "polar":
        cfg, loops = W.polar_case(dict(code=case["code"], alpha=case["alpha"], Re=case["Re"], levels=case["levels"],
                                       Ma=0.15, store=case["store"]))
    elif case["grid"] == "small":
        cfg, _ = W.naca0012_small(case["levels"])
        loops = [W.naca_loop(case["code"], cfg["h0"] / 2 ** (case["levels"] - 1), alpha_deg=case["alpha"])]
    else:
        cfg, _ = W.naca0012_large(layers=case["layers"])
        loops = [W.naca_loop(case["code"], cfg["h0"] / 2 ** (case["levels"] - 1), alpha_deg=case["alpha"])]
    cfg.update(levels=case["levels"], layers=case["layers"], Re=case["Re"], store=case["store"])
    return cfg, loops


def _batch_configs(case):
    reqs = W.polar_requests(case["members"], seed=case["pick"])
    return [_naca_config(dict(r, grid="polar", levels=case["levels"], layers=case["layers"], store=case["store"]))
            for r in reqs]


# --------------------------------------------------------------------------- inputs

def _generator(seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    return torch.Generator(device=dev).manual_seed(seed), dev


def _box_fields(case, seed):
    """Vortices of a few seeded wavelengths with noise on top: on a slow drift, or on the free
    stream in the tunnel and with 16-bit storage (whose populations are kept relative to it)."""
    free = case["kind"] == "tunnel" or case["store"] != FP32
    amp = 0.015 if case["store"] == FP32 else 0.003
    gen, dev = _generator(seed)
    nx, ny = case["nx"], case["ny"]
    x = 2.0 * math.pi * (torch.arange(nx, dtype=torch.float64, device=dev) + 0.5) / nx
    y = 2.0 * math.pi * (torch.arange(ny, dtype=torch.float64, device=dev) + 0.5)[:, None] / ny
    r = torch.rand(4, 3, generator=gen, dtype=torch.float64, device=dev).tolist()

    def noise(a):
        return a * (2.0 * torch.rand(ny, nx, generator=gen, dtype=torch.float64, device=dev) - 1.0)

    ux, uy = noise(1e-3), noise(1e-3)
    for k, (a, b, c) in enumerate(r, start=1):
        ux += amp * (0.5 + a) * torch.sin(k * x + 6.0 * b) * torch.cos(k * y + 6.0 * c)
        uy -= amp * (0.5 + a) * (ny / nx if ny < nx else 1.0) * torch.cos(k * x + 6.0 * b) * torch.sin(k * y + 6.0 * c)
    ux += 0.1 * CS if free else 0.01
    return 1.0 + noise(1e-3), ux, uy, 4.0 + noise(2.0)


def _noise_on_level0(solver, cfg, seed):
    """A seeded disturbance of the free stream on the coarsest level."""
    rng = np.random.default_rng(seed)
    U = cfg["Ma"] * CS
    _, _, nx, ny = solver.level_box(0)
    solver.set_fields(0, ux=U * (1.0 + rng.uniform(-1e-3, 1e-3, size=(ny, nx))))


def prepare(case, seed):
    pkg.library()
    if case["kind"] == "request":
        cfg, loops = _naca_config(case)
        cfg["Re"] *= 1.0 + 0.1 * float(np.random.default_rng(seed).uniform())
        return dict(case=case, cfg=cfg, loops=loops)
    if case["kind"] in ("box", "tunnel"):
        cfg = _box_config(case)
        s = pkg.Solver(cfg)
        s.set_geometry([])
        rho, ux, uy, chi = (f.cpu().numpy() for f in _box_fields(case, seed))
        s.set_fields(0, rho=rho, ux=ux, uy=uy, chi=chi)
        solvers = [s]
    else:
        solvers = []
        for k, (cfg, loops) in enumerate([_naca_config(case)] if case["kind"] == "naca" else _batch_configs(case)):
            s = pkg.Solver(cfg)
            s.set_geometry(loops)
            _noise_on_level0(s, cfg, [seed, k])
            solvers.append(s)
    state = dict(case=case, solvers=solvers)
    if case["kind"] == "batch":
        state["batch"] = pkg.Batch(solvers)
    return state


# --------------------------------------------------------------------------- one pass

def _read(solver, case):
    """Fields of every level, one after the other, and the loads where there are walls."""
    to = OUT_TYPE[case["store"]]
    boxes = [solver.level_box(l)[2:] for l in range(solver.cfg["levels"])]
    n = sum(nx * ny for nx, ny in boxes)
    out = dict(rho=torch.empty(n, dtype=to), u=torch.empty(2, n, dtype=to), chi=torch.empty(n, dtype=to),
               mask=torch.empty(n, dtype=torch.uint8))
    at = 0
    for l, (nx, ny) in enumerate(boxes):
        f = solver.get_fields(l)
        part = slice(at, at + nx * ny)
        out["rho"][part] = torch.from_numpy(f["rho"].reshape(-1))
        out["u"][0, part] = torch.from_numpy(f["ux"].reshape(-1))
        out["u"][1, part] = torch.from_numpy(f["uy"].reshape(-1))
        out["chi"][part] = torch.from_numpy(f["chi"].reshape(-1))
        out["mask"][part] = torch.from_numpy(f["mask"].reshape(-1))
        at += nx * ny
    if case["kind"] not in ("box", "tunnel"):
        d = solver.get_loads()
        coef = np.array([d["CL"], d["CD"], d["CDp"], d["CDf"]])
        out["loads"] = torch.from_numpy(np.concatenate([coef, d["cp"], d["cf"]])).to(to)
    return out


def run(state):
    case = state["case"]
    if case["kind"] == "request":
        s = pkg.Solver(state["cfg"])
        s.set_geometry(state["loops"])
        s.step(case["steps"])
        out = _read(s, case)
        s.close()
        return out
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
        for s in state["solvers"]:
            s.synchronize()
        return [_read(s, case) for s in state["solvers"]]
    s = state["solvers"][0]
    s.step(case["steps"])
    return _read(s, case)


def work(case):
    """Per node update: nine populations read and nine written, rho - 1 and u written, and with
    SA-neg chi, u and 1/d^2 read and chi written (108 B in FP32; 88 B laminar, where chi is
    read too), and about 170 operations of the stream-collide and 190 of SA-neg."""
    if case["kind"] in ("box", "tunnel"):
        updates, sa = case["nx"] * case["ny"], case["sa"]
    else:
        cfgs = _batch_configs(case) if case["kind"] == "batch" else [_naca_config(case)]
        updates, sa = sum(pkg.plan(c, loops)["node_updates_per_step"] for c, loops in cfgs), 1
    pop = 4 if case["store"] == FP32 else 2
    n = float(updates) * case["steps"]
    return {"bytes": n * (18 * pop + 16 + (20 if sa else 0)), "flops": n * (170 + (190 if sa else 0))}


# --------------------------------------------------------------------------- 64-bit values

_CX = (0, 1, -1, 0, 0, 1, -1, 1, -1)
_CY = (0, 0, 0, 1, -1, 1, -1, -1, 1)
_W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
_OPP_Y = (0, 1, 2, 4, 3, 7, 8, 5, 6)      # same c_x, opposite c_y


def _equilibrium(rho, ux, uy):
    def h(c, u):
        return 2.0 / 3.0 - u * u if c == 0 else 0.5 * (u * u + 1.0 / 3.0 + c * u)
    return torch.stack([rho * h(_CX[q], ux) * h(_CY[q], uy) for q in range(9)])


def _at(a, dx, dy, edges, flip=False):
    """a at the neighbour (x + dx, y + dy): periodic, or with the tunnel's edges (copied in x,
    mirrored in y; the normal velocity changes its sign there)."""
    if not edges:
        return torch.roll(a, (-dy, -dx), (0, 1))
    b = torch.nn.functional.pad(a[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
    if flip:
        b[0], b[-1] = -b[0], -b[-1]
    ny, nx = a.shape
    return b[1 + dy:1 + dy + ny, 1 + dx:1 + dx + nx]


def _sa_step(chi, ux, uy, nu, edges):
    cb1, cb2, sg, kappa, cw2, cw3, cv1, cv2, cv3, ct3, cn1 = 0.1355, 0.622, 2 / 3, 0.41, 0.3, 2.0, 7.1, 0.7, 0.9, 1.2, 16.0
    cw1 = cb1 / kappa**2 + (1 + cb2) / sg
    x = [_at(chi, _CX[q], _CY[q], edges) for q in range(9)]
    u = [_at(ux, _CX[q], _CY[q], edges) for q in range(9)]
    v = [_at(uy, _CX[q], _CY[q], edges, flip=True) for q in range(9)]
    dudy = (u[3] - u[4] + u[5] - u[6] + u[8] - u[7]) / 6
    dvdx = (v[1] - v[2] + v[5] - v[6] + v[7] - v[8]) / 6
    vort = (dvdx - dudy).abs()
    gx, gy = 0.5 * (x[1] - x[2]), 0.5 * (x[3] - x[4])
    gxx, gyy = x[1] - 2 * chi + x[2], x[3] - 2 * chi + x[4]
    gxy = 0.25 * (x[5] - x[8] - x[7] + x[6])
    conv = -(ux * gx + uy * gy) + 0.5 * (ux * ux * gxx + 2 * ux * uy * gxy + uy * uy * gyy)
    coef = [1 + c * torch.where(c < 0, (cn1 + c**3) / (cn1 - c**3), torch.ones_like(c)) for c in x[:5]]
    face = [0.5 * (coef[0] + c) for c in coef[1:]]
    div = face[0] * (x[1] - chi) - face[1] * (chi - x[2]) + face[2] * (x[3] - chi) - face[3] * (chi - x[4])
    diff = nu * (div + cb2 * (gx * gx + gy * gy)) / sg
    id2 = 1e-24                                     # no wall: the distance is capped at 1e12
    c3 = chi**3
    sbar = nu * chi * (1 - chi / (1 + chi * c3 / (c3 + cv1**3))) * id2 / kappa**2
    st = vort + torch.where(sbar >= -cv2 * vort, sbar,
                            vort * (cv2**2 * vort + cv3 * sbar) / ((cv3 - 2 * cv2) * vort - sbar))
    r = torch.where(st > 0, (nu * chi * id2 / kappa**2 / st).clamp(max=10.0), torch.full_like(st, 10.0))
    g = r + cw2 * (r**6 - r)
    fw = g * ((1 + cw3**6) / (g**6 + cw3**6)) ** (1 / 6)
    src = torch.where(chi >= 0, cb1 * st * chi - cw1 * fw * nu * chi * chi * id2,
                      cb1 * (1 - ct3) * vort * chi + cw1 * nu * chi * chi * id2)
    return chi + (conv + src + diff) / (1 + nu * sum(face) / sg)


def _collide(f, rho, ux, uy, omega):
    """Central moments: the second-order deviators relax with omega, all others go to equilibrium."""
    cx = [c - ux for c in _CX]
    cy = [c - uy for c in _CY]
    dev = sum(f[q] * (cx[q]**2 - cy[q]**2) for q in range(9)) * (1 - omega)
    k11 = sum(f[q] * cx[q] * cy[q] for q in range(9)) * (1 - omega)
    k20, k02, k22 = rho / 3 + dev / 2, rho / 3 - dev / 2, rho / 9
    m20, m02, m11 = k20 + rho * ux**2, k02 + rho * uy**2, k11 + rho * ux * uy
    m21 = uy * k20 + 2 * ux * k11 + rho * ux**2 * uy
    m12 = ux * k02 + 2 * uy * k11 + rho * ux * uy**2
    m22 = k22 + uy**2 * k20 + ux**2 * k02 + 4 * ux * uy * k11 + rho * ux**2 * uy**2
    mx, my = rho * ux, rho * uy
    return torch.stack([rho - m20 - m02 + m22,
                        0.5 * (mx + m20 - m12 - m22), 0.5 * (-mx + m20 + m12 - m22),
                        0.5 * (my + m02 - m21 - m22), 0.5 * (-my + m02 + m21 - m22),
                        0.25 * (m11 + m21 + m12 + m22), 0.25 * (m11 - m21 - m12 + m22),
                        0.25 * (-m11 - m21 + m12 + m22), 0.25 * (-m11 + m21 - m12 + m22)])


def _stream(f, edges, U):
    if not edges:
        return torch.stack([torch.roll(f[q], (_CY[q], _CX[q]), (0, 1)) for q in range(9)])
    g = torch.empty_like(f)
    for q in range(9):
        a = torch.roll(f[q], (_CY[q], _CX[q]), (0, 1))
        if _CY[q]:                                   # specular reflection at the symmetry planes
            j = 0 if _CY[q] > 0 else -1
            a[j] = torch.roll(f[_OPP_Y[q], j], _CX[q], 0)
        g[q] = a
    for q in (2, 6, 8):                              # outlet: zero gradient of the streamed values
        a = torch.roll(f[q, :, -1], _CY[q], 0)
        if _CY[q]:
            j = 0 if _CY[q] > 0 else -1
            a[j] = f[_OPP_Y[q], j, -1]
        g[q, :, -1] = a
    i = g[:, :, 0]                                   # Zou-He velocity inlet
    rho = (i[0] + i[3] + i[4] + 2 * (i[2] + i[6] + i[8])) / (1 - U)
    g[1, :, 0] = i[2] + 2 / 3 * rho * U
    g[5, :, 0] = i[6] - 0.5 * (i[3] - i[4]) + rho * U / 6
    g[7, :, 0] = i[8] + 0.5 * (i[3] - i[4]) + rho * U / 6
    return g


def exact(case, seed):
    """The boxes and the tunnel in 64 bits; the airfoils' grids are too large a matter for plain torch."""
    if case["kind"] not in ("box", "tunnel"):
        return None
    edges = case["kind"] == "tunnel"
    rho, ux, uy, chi = _box_fields(case, seed)
    U, nu = 0.1 * CS, BOX_NU
    f = _equilibrium(rho, ux, uy)
    for _ in range(case["steps"]):
        nue = torch.full_like(chi, nu)
        if case["sa"]:
            chin = _sa_step(chi, ux, uy, nu, edges)
            if edges:
                chin[:, -1] = chin[:, -2]
                chin[:, 0] = 3.0
            chi = chin
            nue = nu * (1 + chi.clamp(min=0) * chi**3 / (chi**3 + 7.1**3))
        f = _stream(f, edges, U)
        rho = f.sum(0)
        ux = (f[1] - f[2] + f[5] - f[6] + f[7] - f[8]) / rho
        uy = (f[3] - f[4] + f[5] - f[6] - f[7] + f[8]) / rho
        f = _collide(f, rho, ux, uy, 1.0 / (3.0 * nue + 0.5))
    return dict(rho=rho.reshape(-1).cpu(), u=torch.stack([ux.reshape(-1), uy.reshape(-1)]).cpu(),
                chi=chi.reshape(-1).cpu(), mask=None)
