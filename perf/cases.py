"""Performance cases of the hybrid low-Mach LB/FD library: what its users run, through the public
``Solver`` and ``AdjointProblem`` calls.

A case is one run configuration; a pass advances it by a chunk of time steps and takes the state
out (``Solver.save_state``), as a simulation does between checkpoints or control decisions; the next
pass goes on from there. The adjoint case is one gradient evaluation (forward and backward).

``exact`` is the same numerics in plain 64-bit torch, written from the discrete equations: pull
streaming with bounce-back, moments, source and pre-conditioning, cumulant collision relaxed fully
beyond second order (the post-collision central moments are then those of a Gaussian, i.e. products
of the second moments), WENO3 advection, centred diffusion, Arrhenius sources. Gradients come from
torch autograd through that step.

Grids: cell r = x + nx (y + ny z); torch arrays here are [..., nz, ny, nx].
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2207_11567_gb300 import AdjointProblem, Solver, _lib

R_GAS = 8.314462618
P_ATM = 101325.0


# ------------------------------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest grid in use: planar flame in FP64 (flame property runs); launches and latency
        dict(name="flame_f64", kind="flame", nx=256, ny=8, nz=1, storage="f64", steps=20),
        # the 1-D flame tool's control loop: a chunk of steps, the flame's properties back on the
        # host, a new inlet velocity
        dict(name="flame_tool_f32", kind="flame_tool", nx=256, ny=1, nz=1, storage="f32", steps=20),
        # 2-D baffled chamber, the deflagration study; its state stays in L2
        dict(name="chamber_f32", kind="chamber", nx=1024, ny=256, nz=1, storage="f32", steps=50),
        # gradient of the fuel consumption through K steps (forward with checkpoints, reverse sweep)
        dict(name="adjoint_f32", kind="adjoint", nx=512, ny=128, nz=1, storage="f32", steps=100),
        # 3-D isothermal swirl flow (non-reacting validation runs) in both population storages
        dict(name="cold_f32", kind="cold", nx=256, ny=128, nz=128, storage="f32", steps=20),
        dict(name="cold_f16", kind="cold", nx=256, ny=128, nz=128, storage="f16", steps=20),
        # 3-D reactive swirl burner, the production run, in both population storages
        dict(name="swirl_f32", kind="swirl", nx=384, ny=192, nz=192, storage="f32", steps=10),
        dict(name="swirl_f16", kind="swirl", nx=384, ny=192, nz=192, storage="f16", steps=10),
        # the same burner at half resolution with the curved-wall treatment of injector and exhaust
        dict(name="swirl_curved_f32", kind="swirl", nx=192, ny=96, nz=96, storage="f32", steps=10, walls="curved"),
        # and with temperature-dependent heat capacities
        dict(name="swirl_varcp_f32", kind="swirl", nx=192, ny=96, nz=96, storage="f32", steps=10, cp="variable"),
        # a sealed vessel with a ragged grid: the thermodynamic pressure rises with the combustion
        dict(name="vessel_f32", kind="vessel", nx=135, ny=101, nz=77, storage="f32", steps=10),
        # periodic box (decaying turbulence), odd sizes
        dict(name="box_f32", kind="box", nx=161, ny=129, nz=97, storage="f32", steps=20),
    ]


def _log_int(rng, lo, hi, multiple=1):
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, int(round(n / multiple)) * multiple)


def draw(rng):
    kind = rng.choice(["flame", "flame_tool", "chamber", "adjoint", "cold", "swirl", "swirl", "vessel", "box"])
    c = dict(kind=kind, nz=1, storage="f32")
    if kind == "flame":
        c.update(nx=_log_int(rng, 64, 768), ny=_log_int(rng, 1, 24), storage=rng.choice(["f64", "f64", "f32"]),
                 steps=rng.randrange(8, 25))
    elif kind == "flame_tool":
        c.update(nx=_log_int(rng, 96, 640), ny=rng.choice([1, 1, 2, 5, 8]), storage=rng.choice(["f32", "f64"]),
                 steps=rng.randrange(10, 25))
    elif kind == "chamber":
        c.update(nx=_log_int(rng, 200, 1400), ny=_log_int(rng, 64, 320), steps=rng.randrange(20, 60))
    elif kind == "adjoint":
        c.update(nx=_log_int(rng, 96, 520), ny=_log_int(rng, 40, 128), steps=rng.randrange(30, 101))
    else:
        # 3-D: x is 1.4 to 2.2 times as long as the cross-section; half of the grids are multiples
        # of 4 along x, half are any size
        ny = _log_int(rng, 40, 176)
        nz = max(24, ny + rng.randrange(-12, 13))
        nx = int(ny * rng.uniform(1.4, 2.1))
        nx = nx if rng.random() < 0.5 else nx // 4 * 4
        c.update(nx=nx, ny=ny, nz=nz, steps=rng.randrange(6, 13))
        if kind == "cold":
            c["storage"] = rng.choice(["f32", "f16"])
        elif kind == "swirl":
            c["storage"] = rng.choice(["f32", "f32", "f16"])
            option = rng.choice(["plain", "plain", "plain", "curved", "variable"])
            if option == "curved":
                c["walls"] = "curved"
            elif option == "variable":
                c["cp"] = "variable"
        elif kind == "box":
            c["collision"] = rng.choice(["cumulant", "cumulant", "bgk"])
    return c


def work(case):
    """One pass: per step and fluid cell, populations and velocity in and out, and for thermal runs
    T and Y_k in and out; then the state written out once. Operations: collision and source per
    population, WENO3 faces and diffusion per field and axis, chemistry."""
    dim = 3 if case["nz"] > 1 else 2
    cells = case["nx"] * case["ny"] * case["nz"] * {"swirl": 0.78, "cold": 0.78, "chamber": 0.97,
                                                    "adjoint": 0.97}.get(case["kind"], 1.0)
    S = {"f64": 8, "f32": 4, "f16": 2}[case["storage"]]
    F = 8 if case["storage"] == "f64" else 4
    K = {"flame": 4, "flame_tool": 4, "cold": 0, "box": 0}.get(case["kind"], 6)
    thermal = K > 0
    Q = 3 ** dim
    state = Q * S + dim * F + ((1 + K) * F if thermal else 0)
    step = (2 * state if thermal else 2 * Q * S) + 1
    flops = 30 * Q + (dim * (1 + K) * 28 + 150 if thermal else 0)
    n = case["steps"]
    if case["kind"] == "adjoint":  # forward, recompute, reverse (about twice a forward step)
        return {"bytes": float(n * cells * 4 * step), "flops": float(n * cells * 4 * flops)}
    return {"bytes": float(cells * (n * step + state)), "flops": float(n * cells * flops)}


# ----------------------------------------------------------------------------------------- inputs
_ATOM = {"C": 12.011e-3, "H": 1.008e-3, "O": 15.999e-3, "N": 14.007e-3}
_W = {"CH4": _ATOM["C"] + 4 * _ATOM["H"], "O2": 2 * _ATOM["O"], "CO": _ATOM["C"] + _ATOM["O"],
      "CO2": _ATOM["C"] + 2 * _ATOM["O"], "H2O": 2 * _ATOM["H"] + _ATOM["O"], "N2": 2 * _ATOM["N"]}
_H = {"CH4": -74.87e3, "O2": 0.0, "CO": -110.53e3, "CO2": -393.52e3, "H2O": -241.83e3, "N2": 0.0}
_W["P"] = (_W["CO2"] + 2 * _W["H2O"]) / 3.0  # lumped product of CH4 + 2 O2 -> CO2 + 2 H2O = 3 P
_H["P"] = (_H["CO2"] + 2 * _H["H2O"]) / 3.0
_LE = {"CH4": 1.0, "O2": 1.1, "CO": 1.1, "CO2": 1.4, "H2O": 0.8, "N2": 1.0, "P": 1.0}
_CP = {"CH4": (1590.0, 2.14), "O2": (863.0, 0.19), "CO": (985.0, 0.183), "CO2": (730.0, 0.4),
       "H2O": (1685.0, 0.6), "N2": (990.0, 0.167)}
_SIX = ["CH4", "O2", "CO", "CO2", "H2O", "N2"]
_FOUR = ["CH4", "O2", "P", "N2"]
_PHI = 0.83


def _mix(names, moles):
    m = [moles.get(k, 0.0) * _W[k] for k in names]
    return [v / sum(m) for v in m]


def _fresh(names):
    return _mix(names, {"CH4": _PHI, "O2": 2.0, "N2": 7.52})


def _burnt(names):
    moles = {"O2": 2.0 - 2.0 * _PHI, "N2": 7.52}
    moles.update({"CO2": _PHI, "H2O": 2.0 * _PHI} if "CO2" in names else {"P": 3.0 * _PHI})
    return _mix(names, moles)


def _species(names, unity=False):
    return [{"name": n, "W": _W[n], "Le": 1.0 if unity else _LE[n], "hf": _H[n] / _W[n]} for n in names]


_ONE_STEP = [{"A": 1.0e9, "beta": 0.0, "E": 1.4e5, "nu": {0: -1.0, 1: -2.0, 2: 3.0}, "order": {0: 0.5, 1: 0.65}}]
_TWO_STEP = [{"A": 1.0e9, "beta": 0.0, "E": 1.4e5, "nu": {0: -1.0, 1: -1.5, 2: 1.0, 4: 2.0},
              "order": {0: 0.5, 1: 0.65}},
             {"A": 5.0e6, "beta": 0.0, "E": 5.0e4, "nu": {2: -1.0, 1: -0.5, 3: 1.0}, "order": {2: 1.0, 1: 0.5}}]


def _config(case):
    dim = 3 if case["nz"] > 1 else 2
    kind = case["kind"]
    cfg = {"dim": dim, "nx": case["nx"], "ny": case["ny"], "nz": case["nz"], "storage": case["storage"],
           "collision": case.get("collision", "cumulant"), "T_ref": 300.0, "mu_exp": 0.7, "Pr": 0.7, "cp": 1400.0,
           "rho_ref": 1.17, "P_th0": P_ATM, "P_ref": 0.0, "omega_bulk": 1.0, "omega_hi": [1.0] * 4, "smag_cs": 0.0,
           "thicken_F": 1.0, "flame_sensor": False, "sensor_beta": 10.0, "sensor_wref": 1e-5, "sensor_species": 0,
           "sensor_oxidizer": 1, "sensor_Ta": 8400.0, "closed_domain": False, "thermal": False, "species": [],
           "reactions": [], "T_in": 300.0, "Y_in": [], "nu_ref": 1.8e-5 / 1.17}
    io, walls, per = ("inlet", "outlet"), ("wall", "wall"), ("periodic", "periodic")
    if kind in ("flame", "flame_tool"):
        cfg.update(bc={"x": io, "y": per}, dx=5e-5, dt=5e-7, thermal=True, species=_species(_FOUR, True),
                   reactions=_ONE_STEP, Y_in=_fresh(_FOUR))
    elif kind in ("chamber", "adjoint"):
        cfg.update(bc={"x": io if kind == "adjoint" else ("wall", "outlet"), "y": walls}, dx=1e-4, dt=5e-8,
                   thermal=True, smag_cs=0.17, thicken_F=5.0, species=_species(_SIX), reactions=_TWO_STEP,
                   Y_in=_fresh(_SIX))
    elif kind == "cold":
        cfg.update(bc={"x": io, "y": walls, "z": walls}, dx=1e-3, dt=3e-6, smag_cs=0.17)
    elif kind in ("swirl", "vessel"):
        cfg.update(bc={"x": io if kind == "swirl" else walls, "y": walls, "z": walls}, dx=5e-4, dt=1e-6, smag_cs=0.17,
                   thermal=True, thicken_F=8.0, flame_sensor=True, closed_domain=True, species=_species(_SIX),
                   reactions=_TWO_STEP, T_in=320.0, Y_in=_fresh(_SIX))
    else:
        cfg.update(bc={"x": per, "y": per, "z": per}, dx=1.0, dt=1.0, nu_ref=0.004, smag_cs=0.1)
    if case.get("cp") == "variable":
        cfg.update(variable_cp=True, T0_thermo=298.15)
        for s in cfg["species"]:
            s["cp_poly"] = [*_CP[s["name"]], 0.0, 0.0, 0.0]
    return cfg


def _waves(rng, xyz, n, amp):
    """A smooth random field: a few sine waves of wavelengths between 12 cells and the grid."""
    shape = torch.broadcast_shapes(*[a.shape for a in xyz])
    out = torch.zeros(shape, dtype=torch.float64, device=xyz[0].device)
    for _ in range(n):
        arg = rng.uniform(0, 2 * math.pi)
        for a in xyz:
            size = max(a.numel(), 2)
            if size >= 12:
                arg = arg + 2 * math.pi / math.exp(rng.uniform(math.log(12.0), math.log(size))) * rng.choice([-1, 1]) * a
        out += torch.sin(arg) if torch.is_tensor(arg) else math.sin(arg)
    return out * (amp / math.sqrt(n / 2.0))


def _inputs(case, seed):
    """Configuration, solid mask, inlet velocities and initial fields (64-bit arrays on the GPU whose
    values the storage type holds exactly)."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator("cuda").manual_seed(int(seed))
    f64 = dict(dtype=torch.float64, device="cuda")
    cfg, kind = _config(case), case["kind"]
    nx, ny, nz, dim = cfg["nx"], cfg["ny"], cfg["nz"], cfg["dim"]
    x = torch.arange(nx, **f64).view(1, 1, nx) + 0.5
    y = torch.arange(ny, **f64).view(1, ny, 1) + 0.5
    z = torch.arange(nz, **f64).view(nz, 1, 1) + 0.5
    axes = (x, y, z)[:dim]
    shape = (nz, ny, nx)
    solid = torch.zeros(shape, dtype=torch.bool, device="cuda")
    inlet = torch.zeros((dim, nz, ny), **f64)
    u = torch.zeros((dim, *shape), **f64)
    burnt = hot = None
    solid_at = None
    if kind in ("flame", "flame_tool"):
        # tanh front a quarter down the channel, 20 cells thick, slightly wrinkled across y
        x0 = nx / 4.0 + rng.uniform(-2, 2)
        burnt = 0.5 * (1 + torch.tanh((x - x0 + _waves(rng, (y,), 2, 1.0)) / 5.0))
        hot = 1950.0
        inlet[0] = 0.0034
        u[0] = 0.0034 * (1 + (hot / 300.0 - 1) * burnt)
        u += 0.0003 * torch.stack([_waves(rng, axes, 3, 1.0) for _ in range(dim)])
    elif kind in ("chamber", "adjoint"):
        # three rows of three baffles at random places, a burnt kernel at the left end
        ow, oh = max(2, round(16 * nx / 1024)), max(2, round(48 * ny / 256))
        for k in range(3):
            xc = int(nx * (0.25 + 0.22 * k) + rng.integers(-nx // 32, nx // 32 + 1))
            for j in range(3):
                lo = int(j * ny / 3 + 1)
                yc = int(rng.integers(lo, max(lo, int((j + 1) * ny / 3 - oh - 1)) + 1))
                solid[0, yc:yc + oh, xc:xc + ow] = True
        rad = max(5.0, 24.0 * ny / 128 if kind == "adjoint" else 24.0 * ny / 256)
        dist = torch.sqrt(x ** 2 + (y - ny / 2.0) ** 2) + _waves(rng, (x, y), 3, 0.5)
        burnt = 0.5 * (1 + torch.tanh((rad - dist) / 1.5))
        hot = 1950.0
        flow = 0.005 if kind == "adjoint" else 0.01
        u[0] = flow * (1 + _waves(rng, axes, 4, 0.2))
        u[1] = _waves(rng, axes, 4, 0.3 * flow)
        if kind == "adjoint":
            inlet[0, 0] = 0.02 * 4 * y.view(-1) * (ny - y.view(-1)) / ny ** 2 * (1 + 0.1 * torch.randn(ny, generator=gen, **f64))
    elif kind in ("cold", "swirl"):
        # annular swirling injector, square chamber, conical exhaust
        s = ny / 128.0
        yc, zc = ny / 2.0, nz / 2.0
        Ri, Ro, Rc = 8.0 * s, 16.0 * s, min(ny, nz) / 2.0 - 1.0
        L1 = max(4, int(round(24 * s * nx / (2 * ny))) + int(rng.integers(-2, 3)))
        L2 = int(round(nx * 0.8)) + int(rng.integers(-4, 5))
        Re = 24.0 * s + rng.uniform(-2.0, 2.0) * s
        span = max(1, nx - 1 - L2)

        def solid_at(X, Y, Z):
            r = torch.sqrt((Y - yc) ** 2 + (Z - zc) ** 2)
            return ((X < L1) & ((r < Ri) | (r > Ro))) | ((X >= L2) & (r > Rc + (Re - Rc) * (X - 0.5 - L2) / span))

        solid = solid_at(x, y, z)
        fy, fz = (y - yc).view(1, ny), (z - zc).view(nz, 1)
        fr = torch.sqrt(fy ** 2 + fz ** 2)
        ann = ((fr >= Ri) & (fr <= Ro)).to(torch.float64)
        ut = 0.05 * 0.6 * 3.0 * Ro * (Ro ** 2 - Ri ** 2) / (2.0 * (Ro ** 3 - Ri ** 3))
        inlet[0] = 0.05 * ann
        inlet[1] = -ut * ann * fz / fr.clamp_min(1e-9)
        inlet[2] = ut * ann * fy / fr.clamp_min(1e-9)
        inlet += 0.0025 * ann * torch.randn(inlet.shape, generator=gen, **f64)
        u[0] = 0.03 + _waves(rng, axes, 4, 0.008)
        for a in (1, 2):
            u[a] = _waves(rng, axes, 4, 0.008)
        if kind == "swirl":
            xf = L1 + 16 * s + _waves(rng, (y, z), 3, 2.0 * s)
            burnt, hot = 0.5 * (1 + torch.tanh((x - xf) / max(1.5, 4.0 * s))), 1970.0
    elif kind == "vessel":
        c = [n * (0.5 + rng.uniform(-0.08, 0.08)) for n in (nx, ny, nz)]
        dist = torch.sqrt(sum((a - b) ** 2 for a, b in zip(axes, c))) + _waves(rng, axes, 3, 0.8)
        burnt, hot = 0.5 * (1 + torch.tanh((0.2 * ny - dist) / 2.0)), 1970.0
        for a in range(3):
            u[a] = _waves(rng, axes, 4, 0.006)
    else:
        for a in range(dim):
            u[a] = _waves(rng, axes, 6, 0.03)
    u = u * ~solid
    T = Y = None
    if cfg["thermal"]:
        burnt = burnt.expand(shape)
        names = [s["name"] for s in cfg["species"]]
        Yu, Yb = _fresh(names), _burnt(names)
        if kind == "adjoint":
            # products in the fresh gas and unburnt fuel in the kernel: no species sits at the switch
            # max(Y, 0) of the rate law, where its derivative is unbounded
            for Ym in (Yu, Yb):
                for n in ("CO", "CO2", "H2O"):
                    Ym[names.index(n)] += 1e-4
                Ym[names.index("CH4")] += 5e-3 if Ym is Yb else 0.0
                Ym[names.index("N2")] = 1.0 - sum(v for n, v in zip(names, Ym) if n != "N2")
            cfg["Y_in"] = list(Yu)
        T = cfg["T_in"] + (hot - cfg["T_in"]) * burnt
        Y = torch.stack([a * (1 - burnt) + b * burnt for a, b in zip(Yu, Yb)])
    if case["storage"] != "f64":
        inlet, u = inlet.float().double(), u.float().double()
        T, Y = (None, None) if T is None else (T.float().double(), Y.float().double())
    links = None
    if case.get("walls") == "curved":
        links = _wall_links(solid, x, y, z, solid_at)
    return dict(cfg=cfg, solid=solid, inlet=inlet, u=u.contiguous(), P=torch.zeros(shape, **f64),
                T=T, Y=Y, links=links)


def _velocity(i, dim):
    return i % 3 - 1, i // 3 % 3 - 1, (i // 9 - 1 if dim == 3 else 0)


def _beyond(solid, cfg, c):
    """Whether the point r - c is a solid cell or lies outside a face that is not periodic."""
    nz, ny, nx = solid.shape
    out = solid
    for axis, (d, n) in enumerate(((2, nx), (1, ny), (0, nz))):
        if c[axis]:
            out = torch.roll(out, c[axis], d)
            if cfg["bc"]["xyz"[axis]][0] != "periodic":
                out = out.clone()
                out.select(d, 0 if c[axis] > 0 else n - 1).fill_(True)
    return out


def _wall_links(solid, x, y, z, solid_at):
    """Links from fluid cells into the shaped solids (cell, pull direction, wall fraction), the
    fraction by bisection on the continuous shape."""
    nz, ny, nx = solid.shape
    per = {"bc": {a: ("wall", "wall") for a in "xyz"}}
    none = torch.zeros_like(solid)
    cells, dirs, q = [], [], []
    for i in range(27):
        c = _velocity(i, 3)
        if not any(c):
            continue
        hit = ~solid & _beyond(solid, per, c) & ~_beyond(none, per, c)
        k, j, l = torch.nonzero(hit, as_tuple=True)
        X, Yc, Z = l + 0.5, j + 0.5, k + 0.5
        lo, hi = torch.zeros(l.numel(), dtype=torch.float64, device="cuda"), torch.ones(l.numel(), dtype=torch.float64, device="cuda")
        for _ in range(30):
            mid = 0.5 * (lo + hi)
            inside = solid_at(X - mid * c[0], Yc - mid * c[1], Z - mid * c[2])
            lo, hi = torch.where(inside, lo, mid), torch.where(inside, mid, hi)
        cells.append(l + nx * (j + ny * k))
        dirs.append(torch.full_like(l, i))
        q.append(hi.clamp(1e-3, 1.0).float().double())
    return torch.cat(cells), torch.cat(dirs), torch.cat(q)


# -------------------------------------------------------------------------------------------- runs
def prepare(case, seed):
    p = _inputs(case, seed)
    cfg = p["cfg"]
    mask = p["solid"].to(torch.uint8).cpu().numpy().reshape(-1)
    inlet = p["inlet"].cpu().numpy().reshape(cfg["dim"], -1)
    if case["kind"] == "adjoint":
        host = {k: p[k].cpu().numpy().reshape((-1, mask.size) if k in ("Y", "u") else -1) for k in ("T", "Y", "u", "P")}
        problem = AdjointProblem(cfg, mask, host["Y"], u0=host["u"], P_h0=host["P"], n_steps=case["steps"],
                                 checkpoint_every=max(1, case["steps"] // 2))
        return dict(case=case, problem=problem, inlet=inlet, T0=host["T"])
    s = Solver(cfg, mask, inlet)
    if p["links"] is not None:
        s.set_wall_links(*[a.cpu().numpy() for a in p["links"]])
    torch.cuda.synchronize()
    ptr = [a.contiguous().data_ptr() if a is not None else None for a in (p["T"], p["Y"], p["u"], p["P"])]
    status = _lib.lib.lbm_set_fields(s.ctx, *ptr, None, 1)
    if status != _lib.LBM_OK:
        raise RuntimeError("set_fields: %d" % status)
    # the saved state's arrays (lbm_save_state: g, u, T, Y, then the pressure state)
    buf = torch.zeros(s.state_bytes(), dtype=torch.uint8, device="cuda")
    F = torch.float64 if case["storage"] == "f64" else torch.float32
    S = torch.float16 if case["storage"] == "f16" else F
    out, at = {}, 0
    parts = [("g", s.Q, S), ("u", s.dim, F)] + ([("T", 1, F), ("Y", s.K, F)] if cfg["thermal"] else [])
    fluid = ~p["solid"]
    for name, n, dtype in parts:
        size = n * s.N * dtype.itemsize
        out[name] = buf[at:at + size].view(dtype).view(n, *fluid.shape)
        at += size
    return dict(case=case, solver=s, buf=buf, out=out, u_in=0.0034 * np.ones(s.N // cfg["nx"]))


def run(state):
    case = state["case"]
    if case["kind"] == "adjoint":
        J = state["problem"].forward(state["inlet"], state["T0"])
        grad_inlet, grad_T0 = state["problem"].backward()
        return {"J": J, "grad_inlet": grad_inlet, "grad_T0": grad_T0}
    s = state["solver"]
    s.step(case["steps"])
    extra = {}
    if case["kind"] == "flame_tool":
        # the tool's control: the inlet follows the consumption speed
        p = s.flame_properties(0, profile=True)
        extra = {"props": np.array([p["S_c"], p["T_min"], p["T_max"], p["T_b"], *p["Y_b"]], dtype=_np_type(case)),
                 "profile": np.concatenate([p["T"][None], p["Y"], p["w_F"][None]]).astype(_np_type(case))}
        s.set_inlet(np.concatenate([state["u_in"], np.zeros_like(state["u_in"])]))
    s.save_state(state["buf"])
    out = state["out"]
    if case["storage"] == "f16":
        # velocities are moments of 16-bit populations: that is the precision they are handed on in
        out = {**out, "u": out["u"].half()}
    return {**out, **extra}


def _np_type(case):
    return np.float64 if case["storage"] == "f64" else np.float32


# ------------------------------------------------------------------------------------ 64-bit steps
class _Exact:
    """The discrete hybrid step in 64-bit torch."""

    def __init__(self, p):
        cfg = self.cfg = p["cfg"]
        self.dim = cfg["dim"]
        self.Q = 3 ** self.dim
        self.c = [_velocity(i, self.dim) for i in range(self.Q)]
        one = {-1: 1 / 6, 0: 2 / 3, 1: 1 / 6}
        self.w = [math.prod(one[v] for v in c[:self.dim]) for c in self.c]
        self.solid, self.fluid, self.inlet = p["solid"], ~p["solid"], p["inlet"]
        self.nu = cfg["nu_ref"] * cfg["dt"] / cfg["dx"] ** 2
        self.link = [_beyond(self.solid, cfg, c) for c in self.c]
        nz, ny, nx = self.solid.shape
        col = torch.arange(nx, device="cuda").view(1, 1, nx)
        none = torch.zeros_like(self.solid)
        self.at_inlet = (col == 0) | none if cfg["bc"]["x"][0] == "inlet" else none
        self.at_outlet = (col == nx - 1) | none if cfg["bc"]["x"][1] == "outlet" else none
        self.q_wall, self.ghost = None, {}
        if p["links"] is not None:
            self._walls(*p["links"])
        if cfg["thermal"]:
            self.K = len(cfg["species"])
            col_of = lambda key: torch.tensor([s[key] for s in cfg["species"]], dtype=torch.float64, device="cuda")  # noqa: E731
            self.Wk, self.Le, self.hf = col_of("W"), col_of("Le"), col_of("hf")
            self._kinds()

    # ---- geometry
    def _walls(self, cell, direction, q):
        """Interpolated bounce-back fractions, and the ghost-point weights of the scalar walls."""
        N = self.solid.numel()
        f = torch.full((self.Q, N), 0.5, dtype=torch.float64, device="cuda")
        f[direction, cell] = q
        f = f.view(self.Q, *self.solid.shape)
        for i, c in enumerate(self.c):
            off = ~self.link[i] | self.solid | (self.at_inlet if c[0] == 1 else self.at_outlet if c[0] == -1 else self.solid)
            f[i] = torch.where(off | ((f[i] < 0.5) & self.link[self.Q - 1 - i]), 0.5, f[i])
        self.q_wall = f

    def _kinds(self):
        """Per axis and side: kind of the distance-1 point (0 fluid, 1 wall or solid, 2 inlet, 3
        outlet) and of the distance-2 point (0 fluid, 1 copy of the distance-1 value, 2 inlet)."""
        self.k1, self.k2 = {}, {}
        for a in range(self.dim):
            for s in (-1, 1):
                c = [0, 0, 0]
                c[a] = -s
                k = torch.where(_beyond(self.solid, self.cfg, c), 1, 0)
                if a == 0:
                    k = torch.where(self.at_inlet, 2, k) if s < 0 else torch.where(self.at_outlet, 3, k)
                self.k1[a, s] = k
            for s in (-1, 1):
                k, kn = self.k1[a, s], self._at(self.k1[a, s], a, s)
                self.k2[a, s] = torch.where(k != 0, torch.where(k == 2, 2, 1), torch.where(kn == 0, 0, torch.where(kn == 2, 2, 1)))
        if self.q_wall is None:
            return
        for a in range(self.dim):
            for s in (-1, 1):
                c = [0, 0, 0]
                c[a] = -s
                i = self.c.index(tuple(c))
                q = self.q_wall[i]
                on = (self.k1[a, s] == 1) & (self.k1[a, -s] == 0) & self.fluid
                w1 = torch.where(on, (1 - 2 * q) / (1 + 2 * q), 0.0)
                w2 = torch.where((self.k1[a, s] == 0) & (self.k2[a, s] == 1), self._at(w1, a, s), 0.0)
                self.ghost[a, s] = w1, w2

    @staticmethod
    def _at(v, axis, s):
        """v at r + s e_axis (periodic)."""
        return torch.roll(v, -s, -1 - axis)

    def _stencil(self, v, v_in, a):
        """v at r - 2e, r - e, r + e, r + 2e with the ghost rules of the boundaries."""
        one, two = {}, {}
        raw = {s: self._at(v, a, s) for s in (-1, 1)}
        for s in (-1, 1):
            k1 = self.k1[a, s]
            one[s] = torch.where(k1 == 0, raw[s], torch.where(k1 == 2, v_in, v))
        for s in (-1, 1):
            n = one[s]
            if self.ghost:
                w1, w2 = self.ghost[a, s]
                g = torch.where(self.k1[a, s] == 1, v + w1 * (one[-s] - v), n)
                copy = torch.where(self.k1[a, s] == 1, g, n + w2 * (v - n))
                n = g
            else:
                copy = n
            k2 = self.k2[a, s]
            two[s] = torch.where(k2 == 0, self._at(raw[s], a, s), torch.where(k2 == 2, v_in, copy))
            raw[s] = n
        return two[-1], raw[-1], raw[1], two[1]

    # ---- scalars
    def rates(self, T, Y, rho):
        """Reaction rates in mol/(m^3 s), rho in kg/m^3."""
        out = []
        for rx in self.cfg["reactions"]:
            q = rx["A"] * torch.exp(-rx["E"] / (R_GAS * T))
            for k, n in rx["order"].items():
                pos = Y[k] > 0
                conc = rho * torch.where(pos, Y[k], 1.0) / self.Wk[k]
                q = q * torch.where(pos, conc ** n, 0.0)
            out.append(q)
        return out

    def density(self, T, Y, P):
        W = 1.0 / (Y / self.Wk.view(-1, 1, 1, 1)).sum(0)
        return P * W / (R_GAS * T * self.cfg["rho_ref"]), W

    def thickening(self, T, Y):
        cfg = self.cfg
        if not cfg["flame_sensor"]:
            return cfg["thicken_F"] * torch.ones_like(T)
        om = Y[cfg["sensor_species"]].clamp_min(0) * Y[cfg["sensor_oxidizer"]].clamp_min(0) * torch.exp(-cfg["sensor_Ta"] / T)
        return 1 + (cfg["thicken_F"] - 1) * torch.tanh(cfg["sensor_beta"] * om / cfg["sensor_wref"])

    def scalars(self, T, Y, u, P, dP):
        cfg, K = self.cfg, self.K
        rho, W = self.density(T, Y, P)
        F = self.thickening(T, Y)
        mu = lambda t: self.nu * (t / cfg["T_ref"]) ** cfg["mu_exp"]  # noqa: E731
        q = self.rates(T, Y, rho * cfg["rho_ref"])
        om = [sum(rx["nu"].get(k, 0.0) * qj for rx, qj in zip(cfg["reactions"], q)) * self.Wk[k] for k in range(K)]
        chem = cfg["dt"] / (rho * cfg["rho_ref"] * F)
        var = "cp_poly" in cfg["species"][0]
        cpk = lambda k, t: cfg["species"][k]["cp_poly"][0] + cfg["species"][k]["cp_poly"][1] * t  # noqa: E731
        cp = sum(Y[k] * cpk(k, T) for k in range(K)) if var else cfg["cp"]
        T_st = [self._stencil(T, cfg["T_in"], a) for a in range(self.dim)]
        adv, dif = [0.0] * (K + 1), [0.0] * (K + 1)
        for a in range(self.dim):
            lo, hi, FM, Tn = {}, {}, {}, {-1: T_st[a][1], 1: T_st[a][2]}
            up = {}
            for s in (-1, 1):
                k1 = self.k1[a, s]
                # at the inlet face the neighbour's velocity is the inlet's
                un = torch.where(k1 == 0, self._at(u[a], a, s), torch.where(k1 == 3, u[a], 0.0))
                if a == 0 and s < 0:
                    un = torch.where(k1 == 2, self.inlet[0].unsqueeze(-1), un)
                up[s] = 0.5 * (u[a] + un) >= 0
                FM[s] = torch.where(k1 == 0, self._at(F, a, s), F) * mu(Tn[s])
            FMr = F * mu(T)
            Ys = [self._stencil(Y[k], cfg["Y_in"][k], a) for k in range(K)]
            for f, (m2, m1, p1, p2) in enumerate([T_st[a]] + Ys):
                v = T if f == 0 else Y[f - 1]
                eps = 1e-6 * cfg["T_ref"] ** 2 if f == 0 else 1e-6
                hi = torch.where(up[1], _weno(m1, v, p1, eps), _weno(p2, p1, v, eps))
                lo = torch.where(up[-1], _weno(m2, m1, v, eps), _weno(p1, v, m1, eps))
                adv[f] = adv[f] + u[a] * (hi - lo)
                if var and f == 0:
                    lam = {s: FM[s] * sum(Ys[k][1 if s < 0 else 2] * cpk(k, Tn[s]) for k in range(K)) for s in (-1, 1)}
                    flux = sum((cpk(k, T) - cp) / self.Le[k] * (Ys[k][2] - Ys[k][1]) for k in range(K)) * (p1 - m1)
                    dif[f] = dif[f] + 0.5 * (FMr * cp + lam[1]) * (p1 - v) - 0.5 * (FMr * cp + lam[-1]) * (v - m1) + 0.25 * FMr * flux
                else:
                    dif[f] = dif[f] + 0.5 * (FMr + FM[1]) * (p1 - v) - 0.5 * (FMr + FM[-1]) * (v - m1)
        if var:
            T0 = cfg["T0_thermo"]
            h = [self.hf[k] + cfg["species"][k]["cp_poly"][0] * (T - T0) + 0.5 * cfg["species"][k]["cp_poly"][1] * (T * T - T0 * T0)
                 for k in range(K)]
        else:
            h = list(self.hf)
        heat = -sum(h[k] * om[k] for k in range(K))
        N_T = dif[0] / (cfg["Pr"] * rho * (cp if var else 1.0)) + chem * heat / cp + dP / (cp * rho * cfg["rho_ref"])
        N_Y = [dif[1 + k] / (cfg["Pr"] * self.Le[k] * rho) + chem * om[k] for k in range(K)]
        lam = N_T / T + sum(W / self.Wk[k] * N_Y[k] for k in range(K))
        keep = lambda new, old: torch.where(self.fluid, new, old)  # noqa: E731
        T1 = keep(T - adv[0] + N_T, T)
        Y1 = torch.stack([keep(Y[k] - adv[1 + k] + N_Y[k], Y[k]) for k in range(K)])
        return T1, Y1, torch.where(self.fluid, rho, 1.0), torch.where(self.fluid, lam, 0.0)

    # ---- flow (populations stored as q_i = g_i / w_i)
    def equilibrium(self, P, u, rho):
        usq = sum(v * v for v in u)
        q = []
        for c in self.c:
            cu = sum(k * v for k, v in zip(c, u))
            q.append(P + rho * (cu + 1.5 * cu * cu - 0.5 * usq))
        return torch.stack(q)

    def flow(self, g, u_old, rho, lam, T):
        cfg, dim = self.cfg, self.dim
        thermal = T is not None
        q, grad = [], [0.0] * dim
        near = {}
        shift = lambda v, c: torch.roll(v, c[::-1], (-3, -2, -1))  # noqa: E731
        for i, c in enumerate(self.c):
            o = self.Q - 1 - i
            v = torch.where(self.link[i], g[o], shift(g[i], c))
            if self.q_wall is not None:
                f = self.q_wall[i]
                far = shift(g[o], [-k for k in c])
                v = torch.where(self.link[i] & (f < 0.5), far + 2 * f * (g[o] - far), v)
                v = torch.where(self.link[i] & (f > 0.5), g[i] + (g[o] - g[i]) / (2 * f), v)
            if c[0] == 1:
                cu = sum(k * w for k, w in zip(c, self.inlet)).unsqueeze(-1)
                v = torch.where(self.at_inlet, v + 2 * rho * cu, v)
            if c[0] == -1:
                cu, vv = sum(k * w for k, w in zip(c, u_old)), sum(w * w for w in u_old)
                v = torch.where(self.at_outlet, -g[o] + rho * (3 * cu * cu - vv), v)
            q.append(v)
            if thermal and sum(map(abs, c)) == 1:
                near[c] = torch.where(self.link[i], rho, shift(rho, c))
        u = [3 * sum(c[a] * w * v for c, w, v in zip(self.c, self.w, q)) / rho for a in range(dim)]
        usq = sum(v * v for v in u)
        if thermal:
            for a in range(dim):
                e = [0, 0, 0]
                e[a] = 1
                grad[a] = 0.5 * (near[tuple(-k for k in e)] - near[tuple(e)])
        udg = sum(a * b for a, b in zip(u, grad))
        half = []
        for c in self.c:
            cu, cg = (sum(k * w for k, w in zip(c, v)) for v in (u, grad))
            half.append(0.5 * ((cu + 1.5 * cu * cu - 0.5 * usq) * (cg - udg) + rho * lam / 3))
        s = [a + b for a, b in zip(q, half)]
        S = sum(w * v for w, v in zip(self.w, s))
        h = [w * (1 + 3 * (v - S) / rho) for w, v in zip(self.w, s)]  # unit density, velocity u
        sig = [[None] * dim for _ in range(dim)]
        for a in range(dim):
            for b in range(a, dim):
                sig[a][b] = sig[b][a] = sum((c[a] - u[a]) * (c[b] - u[b]) * v for c, v in zip(self.c, h))
        tau0 = 3 * self.nu * ((T / cfg["T_ref"]) ** cfg["mu_exp"] / rho if thermal else 1.0) + 0.5
        bgk = cfg["collision"] == "bgk"
        if bgk:  # non-equilibrium stress about the polynomial equilibrium
            feq = [w * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * usq)
                   for w, cu in ((w, sum(k * v for k, v in zip(c, u))) for c, w in zip(self.c, self.w))]
            ne = [[sum(c[a] * c[b] * (x - y) for c, x, y in zip(self.c, h, feq)) for b in range(dim)] for a in range(dim)]
        else:
            ne = [[sig[a][b] - (1 / 3 if a == b else 0.0) for b in range(dim)] for a in range(dim)]
        tr = sum(ne[a][a] for a in range(dim)) / dim
        dev = [[ne[a][b] - (tr if a == b else 0.0) for b in range(dim)] for a in range(dim)]
        tau = tau0
        if cfg["smag_cs"] > 0:
            n2 = sum(dev[a][b] ** 2 for a in range(dim) for b in range(dim))
            pos = n2 > 0
            norm = torch.where(pos, torch.sqrt(torch.where(pos, n2, 1.0)), 0.0)
            tau = 0.5 * (tau0 + torch.sqrt(tau0 * tau0 + 18 * math.sqrt(2.0) * cfg["smag_cs"] ** 2 * norm))
        omega = 1 / tau
        if bgk:
            h = [x - omega * (x - y) for x, y in zip(h, feq)]
        else:
            new = [[(1 - omega) * dev[a][b] + ((1 / 3 + (1 - cfg["omega_bulk"]) * tr) if a == b else 0.0) for b in range(dim)]
                   for a in range(dim)]
            h = self._gaussian(new, u)
        q1 = torch.stack([rho / 3 * (v / w - 1) + S + x for v, w, x in zip(h, self.w, half)])
        u1 = torch.stack([v.expand_as(rho) for v in u])
        return torch.where(self.fluid, q1, g), torch.where(self.fluid, u1, u_old)

    def _gaussian(self, s, u):
        """Populations whose central moments up to order 2 per axis are those of a Gaussian with
        covariance s (odd ones vanish) and whose velocity is u."""
        dim = self.dim
        m = {}
        for i in range(self.Q):
            e = (i % 3, i // 3 % 3, i // 9)[:dim]
            idx = [a for a in range(dim) for _ in range(e[a])]
            m[e] = _wick(idx, s)
        for a in range(dim):  # central to raw moments to populations, one axis at a time
            nxt = {}
            for e in m:
                if e[a]:
                    continue
                at = lambda k: m[e[:a] + (k,) + e[a + 1:]]  # noqa: E731, B023
                m0, m1, m2 = at(0), at(1), at(2)
                r1, r2 = m1 + u[a] * m0, m2 + 2 * u[a] * m1 + u[a] * u[a] * m0
                for k, v in enumerate((0.5 * (r2 - r1), m0 - r2, 0.5 * (r2 + r1))):
                    nxt[e[:a] + (k,) + e[a + 1:]] = v
            m = nxt
        return [m[(i % 3, i // 3 % 3, i // 9)[:dim]] for i in range(self.Q)]

    # ---- whole steps
    def start(self, p):
        rho = torch.ones_like(p["P"])
        st = {"u": p["u"], "T": p["T"], "Y": p["Y"], "P": P_ATM, "dP": 0.0}
        if self.cfg["thermal"]:
            rho, _ = self.density(p["T"], p["Y"], P_ATM)
            if self.cfg["closed_domain"]:
                st["M"] = P_ATM * self._integral(p["T"], p["Y"])
        st["g"] = self.equilibrium(p["P"], p["u"], rho)
        return st

    def _integral(self, T, Y):
        return (self.density(T, Y, 1.0)[0] * self.fluid).sum()

    def step(self, st):
        n = dict(st)
        if not self.cfg["thermal"]:
            n["g"], n["u"] = self.flow(st["g"], st["u"], torch.ones_like(st["u"][0]), torch.zeros_like(st["u"][0]), None)
            return n
        n["T"], n["Y"], rho, lam = self.scalars(st["T"], st["Y"], st["u"], st["P"], st["dP"])
        if self.cfg["closed_domain"] and self.cfg["bc"]["x"][1] != "outlet":
            n["P"] = st["M"] / self._integral(n["T"], n["Y"])
            n["dP"] = n["P"] - st["P"]
            lam = lam - n["dP"] / st["P"]
        n["g"], n["u"] = self.flow(st["g"], st["u"], rho, lam, st["T"])
        return n


def _weno(a, b, c, eps):
    t0, t1 = (eps + (b - a) ** 2) ** 2, (eps + (c - b) ** 2) ** 2
    return b + 0.5 * (t1 * (b - a) + 2 * t0 * (c - b)) / (t1 + 2 * t0)


def _wick(idx, s):
    """Moment of a centred Gaussian with covariance s: the sum over pairings of the indices."""
    if not idx:
        return 1.0
    if len(idx) % 2:
        return 0.0
    return sum(s[idx[0]][idx[k]] * _wick(idx[1:k] + idx[k + 1:], s) for k in range(1, len(idx)))


def exact(case, seed):
    p = _inputs(case, seed)
    e = _Exact(p)
    if case["kind"] == "adjoint":
        return _exact_gradient(case, p, e)
    st = e.start(p)
    with torch.no_grad():
        for _ in range(case["steps"]):
            st = e.step(st)
    out = {"g": st["g"], "u": st["u"]}
    if p["cfg"]["thermal"]:
        out.update(T=st["T"].unsqueeze(0), Y=st["Y"])
    if case["kind"] == "flame_tool":
        out.update(_exact_flame(p["cfg"], e, st))
    return out


def _exact_flame(cfg, e, st):
    T, Y = st["T"], st["Y"]
    rho, _ = e.density(T, Y, st["P"])
    fuel = -e.Wk[0] * sum(rx["nu"][0] * q for rx, q in zip(cfg["reactions"], e.rates(T, Y, rho * cfg["rho_ref"])))
    fuel = fuel / cfg["thicken_F"]
    mean = lambda v: v.mean((-3, -2))  # noqa: E731
    Tm, Ym, w = mean(T), mean(Y), mean(fuel)
    W_in = 1.0 / sum(y / k for y, k in zip(cfg["Y_in"], e.Wk.tolist()))
    S_c = w.sum() * cfg["dx"] / (P_ATM * W_in / (R_GAS * cfg["T_in"]) * cfg["Y_in"][0])
    props = torch.stack([S_c, Tm.min(), Tm.max(), Tm[-1], *Ym[:, -1]])
    return {"props": props, "profile": torch.cat([Tm[None], Ym, w[None]])}


def _exact_gradient(case, p, e):
    inlet = p["inlet"].clone().requires_grad_()
    T0 = p["T"].clone().requires_grad_()
    e.inlet = inlet
    st = e.start({**p, "T": T0})

    def one(g, u, T, Y, inlet_):
        e.inlet = inlet_
        n = e.step({"g": g, "u": u, "T": T, "Y": Y, "P": P_ATM, "dP": 0.0})
        return n["g"], n["u"], n["T"], n["Y"]

    s = (st["g"], st["u"], st["T"], st["Y"])
    for _ in range(case["steps"]):
        s = checkpoint(one, *s, inlet, use_reentrant=False)
    T, Y = s[2], s[3]
    rho, _ = e.density(T, Y, P_ATM)
    q = e.rates(T, Y, rho * p["cfg"]["rho_ref"])
    J = -e.Wk[0] * (sum(rx["nu"].get(0, 0.0) * v for rx, v in zip(p["cfg"]["reactions"], q)) * e.fluid).sum()
    gi, gT = torch.autograd.grad(J, (inlet, T0))
    return {"J": J.detach(), "grad_inlet": gi.view(2, -1), "grad_T0": (gT * e.fluid).view(-1)}
