"""The workloads this library's speed is judged on, through its public calls.

One pass of a single-lattice case is one monitored segment of a run, as a user's program
advances a flow: ``step_residual(steps)`` (the last step also forms residual and mass),
the macroscopic fields with ``macros``, and, for the cases that keep a restart state, the
populations with ``get_populations`` into a device buffer. One pass of a batch case is
one serving round: every resident lattice advanced, its residual and mass read, its
fields taken. The state evolves from pass to pass, as it does in a run.

``exact`` advances the same stored state in float64 with plain tensor operations.
"""
import math
import random

import numpy as np
import torch

import paper_0811_4593_gb300 as lbm

# c_1 .. c_19 as the library stores them, and their weights in 36ths
C = ((1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
     (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (-1, 1, 0), (-1, -1, 0),
     (-1, 0, 1), (-1, 0, -1), (0, 1, 1), (0, 1, -1), (0, -1, 1), (0, -1, -1), (0, 0, 0))
W = tuple([2 / 36] * 6 + [1 / 36] * 12 + [12 / 36])
OPP = tuple(C.index(tuple(-a for a in c)) for c in C)
BYTES = {"f64": 8, "f32": 4, "f16": 2}
DTYPE = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16}
FLOPS = 230  # additions and multiplications of one node update (moments, relaxation)
NOISE = 0.01  # spread of the starting populations about their equilibrium, in units of w_i


def _solo(name, kind, nx, ny, nz, precision, steps, tau, scheme="ab", keep=False):
    case = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "precision": precision, "steps": steps, "tau": tau,
            "scheme": scheme, "keep": keep}
    return dict(case, name=name) if name else case


def listed():
    return [
        # validation runs: the Couette flow of the test suite in double (1,088 nodes) and
        # the narrow plane Poiseuille channel in float, thousands of steps of tiny sweeps
        _solo("couette_f64", "couette", 8, 8, 17, "f64", 500, 1.0, keep=True),
        _solo("poiseuille_f32", "poiseuille", 4, 4, 256, "f32", 500, 1.0),
        # the paper's body-force Poiseuille box
        _solo("force_f32", "force", 32, 32, 32, "f32", 200, 2.0),
        # the square duct between pressure planes, width 33 (odd), length three widths
        _solo("pressure_f64", "pressure", 99, 33, 33, "f64", 100, 1.0),
        # the tilted channel (solid nodes, mid-grid bounce-back) at twice the paper's size
        _solo("tilted_f32", "tilted", 128, 16, 256, "f32", 100, 1.0),
        # the 256 x 64 x 64 duct: the float run, and the double run it is checked against
        _solo("duct_f32", "duct", 256, 64, 64, "f32", 100, 0.6),
        _solo("duct_f64", "duct", 256, 64, 64, "f64", 20, 0.6, keep=True),
        # a binary16 run of ragged size that keeps its restart state
        _solo("channel_f16_ragged", "channel", 251, 127, 190, "f16", 100, 0.8, keep=True),
        # one-array streaming, for lattices that would not fit twice; odd sizes
        _solo("channel_f32_aa", "channel", 301, 199, 255, "f32", 50, 0.8, scheme="aa"),
        # the benchmark channel in binary16 and in float
        _solo("channel512_f16", "channel", 512, 512, 512, "f16", 50, 0.8),
        _solo("channel512_f32", "channel", 512, 512, 512, "f32", 50, 0.8),
        # a serving round: duct and channel solves of mixed sizes, 100 steps each
        {"name": "serving_f32", "kind": "batch", "lattices": 14, "low": 32, "high": 192, "mix": 1,
         "precision": "f32", "steps": 100, "scheme": "ab"},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    precision = rng.choice(("f64", "f64", "f32", "f32", "f32", "f16", "f16"))
    kind = rng.choice(("couette", "poiseuille", "force", "pressure", "tilted", "duct", "duct", "channel", "channel",
                       "channel", "batch"))
    scheme = "aa" if kind in ("couette", "duct", "channel", "batch") and rng.random() < 0.3 else "ab"
    if kind == "batch":
        high = int(_log(rng, 64, 192))
        return {"kind": kind, "lattices": rng.randint(3, 14), "low": rng.randint(16, 40), "high": high,
                "mix": rng.randint(2, 10 ** 6), "precision": precision, "steps": 2 * rng.randint(10, 40),
                "scheme": scheme}
    if kind == "poiseuille":
        nx, ny, nz = rng.randint(4, 9), rng.randint(3, 8), rng.randint(16, 400)
    elif kind == "force":
        n = rng.randint(16, 120)
        nx, ny, nz = n, rng.randint(3, n), rng.randint(3, n)
    elif kind == "pressure":
        n = rng.randint(8, 80)
        nx, ny, nz = 3 * n, n, n
    elif kind == "tilted":
        s = rng.randint(1, 3)
        nx, ny, nz = 64 * s, rng.randint(4, 8 * s + 1), 128 * s
    else:
        nodes = _log(rng, 1e3, 3e7 if precision == "f64" else 1.3e8)
        a, b = _log(rng, 0.5, 2.0), _log(rng, 0.5, 2.0)
        side = (nodes / (a * b)) ** (1 / 3)
        nx, ny, nz = (max(8, round(v)) for v in (a * side, b * side, side))
        if rng.random() < 0.4:  # rows of whole 32-node pieces are the common choice of users
            nx = max(32, nx // 32 * 32)
    # about as many node updates as the benchmark channel's fastest case allows, 500 at most
    updates = 4e8 if precision == "f64" else 4e9
    steps = 2 * max(5, min(250, int(updates / (nx * ny * nz) / 2)))
    tau = round(rng.uniform(1.0, 2.0) if kind == "force" else rng.uniform(0.7, 1.4), 3)
    return _solo(None, kind, nx, ny, nz, precision, steps, tau, scheme, keep=rng.random() < 0.4)


# -- the flows -----------------------------------------------------------------------


def _parabola(n):
    s = np.arange(n, dtype=np.float64)
    return 4.0 * s * (n - 1 - s) / float((n - 1) ** 2)


def _flow(kind, nx, ny, nz, speed=0.04, angle=30.0):
    """The faces (None, a velocity, a velocity table or ("rho", density)), the solid mask,
    the body force and a typical velocity of a flow."""
    rest = (0.0, 0.0, 0.0)
    solid = force = None
    if kind == "couette":
        faces, u = [None, None, None, None, rest, (0.05, 0.0, 0.0)], (0.025, 0.0, 0.0)
    elif kind == "poiseuille":
        tab = np.zeros((nz, ny, 3))
        tab[..., 0] = 0.02 * _parabola(nz)[:, None]
        faces, u = [tab, tab, None, None, rest, rest], (0.01, 0.0, 0.0)
    elif kind == "force":
        faces, force, u = [rest, rest, None, None, None, None], (0.0, 0.0, 1e-5), (0.0, 0.0, 0.005)
    elif kind == "pressure":
        faces, u = [("rho", 1.002), ("rho", 0.998), rest, rest, rest, rest], (0.01, 0.0, 0.0)
    elif kind == "duct":
        tab = np.zeros((nz, ny, 3))
        prof = 1.25 * speed * np.outer(_parabola(nz), _parabola(ny))
        tab[..., 0], tab[..., 1] = prof * math.cos(math.radians(angle)), prof * math.sin(math.radians(angle))
        faces, u = [tab, tab, rest, rest, rest, rest], (0.25 * speed, 0.0, 0.0)
    elif kind == "channel":
        v = (speed * math.cos(math.radians(angle / 2)), speed * math.sin(math.radians(angle / 2)), 0.0)
        faces, u = [v, v, None, None, rest, rest], v
    else:  # tilted: a channel along z, its centre line moving in x; solid outside it
        half, g = 10.0 * nx / 64, 40.0 * (nx / 64) / (nz - 1)
        x, z = np.arange(nx)[None, None, :], np.arange(nz)[:, None, None]
        d = (x - (nx - 1) / 2 - g * (z - (nz - 1) / 2)) / half + np.zeros((1, ny, 1))
        solid = (np.abs(d) >= 1.0).astype(np.uint8)
        prof = np.where(solid == 0, 0.01 * (1.0 - d * d), 0.0)
        vel = prof[..., None] * (np.array([g, 0.0, 1.0]) / math.hypot(g, 1.0))
        faces = [None, None, None, None, np.ascontiguousarray(vel[0]), np.ascontiguousarray(vel[-1])]
        u = (0.0, 0.0, 0.005)
    return faces, solid, force, u


def _members(case):
    """The lattices of a batch: (kind, nx, ny, nz, tau, speed, angle)."""
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["lattices"]):
        dims = [int(_log(rng, case["low"], case["high"])) for _ in range(3)]
        out.append((rng.choice(("duct", "channel")), *dims, rng.uniform(0.7, 1.5), rng.uniform(0.01, 0.06),
                    rng.uniform(0.0, 45.0)))
    return out


def _start(nx, ny, nz, u, precision, seed):
    """Stored populations about the equilibrium at density 1 and velocity u (double holds
    f, float and binary16 hold f - w)."""
    gen = torch.Generator("cuda").manual_seed(seed)
    f = torch.empty((19, nz, ny, nx), dtype=DTYPE[precision], device="cuda")
    uu = sum(a * a for a in u)
    for k in range(19):
        cu = sum(a * b for a, b in zip(C[k], u))
        dev = 3 * cu + 4.5 * cu * cu - 1.5 * uu
        r = torch.rand((nz, ny, nx), generator=gen, device="cuda")
        r.mul_(2 * NOISE).add_(dev - NOISE)
        f[k] = W[k] * (1.0 + r.double()) if precision == "f64" else W[k] * r
    return f


def _lattice(flow, nx, ny, nz, tau, precision, scheme, seed):
    faces, solid, force, u = flow
    lat = lbm.Lattice(nx, ny, nz, tau, [lbm.Pressure(f[1]) if isinstance(f, tuple) and f[0] == "rho" else f
                                        for f in faces], precision, scheme=scheme)
    lat.set_populations(_start(nx, ny, nz, u, precision, seed))
    if solid is not None:
        lat.set_solid(solid)
    if force is not None:
        lat.set_body_force(force)
    lat.residual()  # the monitor's first reading: the snapshot the next one is compared with
    dt = torch.float64 if precision == "f64" else torch.float32
    fields = (torch.empty((nz, ny, nx), dtype=dt, device="cuda"), torch.empty((3, nz, ny, nx), dtype=dt, device="cuda"))
    return lat, fields


def prepare(case, seed):
    p, scheme = case["precision"], case["scheme"]
    if case["kind"] == "batch":
        batch = lbm.Batch(case["lattices"], p)
        held = []
        for i, (kind, nx, ny, nz, tau, speed, angle) in enumerate(_members(case)):
            held.append(_lattice(_flow(kind, nx, ny, nz, speed, angle), nx, ny, nz, tau, p, scheme, seed * 64 + i))
            batch.attach(i, held[-1][0])
        return {"batch": batch, "held": held, "steps": case["steps"]}
    dims = case["nx"], case["ny"], case["nz"]
    lat, fields = _lattice(_flow(case["kind"], *dims), *dims, case["tau"], p, scheme, seed * 64)
    state = {"lattice": lat, "fields": fields, "steps": case["steps"]}
    if case["keep"]:
        state["kept"] = torch.empty(lat.shape, dtype=DTYPE[p], device="cuda")
    return state


def run(state):
    if "batch" in state:
        state["batch"].step(state["steps"], residual=True)
        results = state["batch"].results()
        return [(r, m, *lat.macros(*fields)) for (r, m, _), (lat, fields) in zip(results, state["held"])]
    lat = state["lattice"]
    r, m = lat.step_residual(state["steps"])
    rho, u = lat.macros(*state["fields"])
    out = {"residual": r, "mass": m, "rho": rho, "u": u}
    if "kept" in state:
        out["populations"] = lat.get_populations(out=state["kept"])
    return out


def work(case):
    """The state read once and written once, the fields and the kept state written; the
    arithmetic of every node update."""
    if case["kind"] == "batch":
        nodes = sum(m[1] * m[2] * m[3] for m in _members(case))
    else:
        nodes = case["nx"] * case["ny"] * case["nz"]
    b = BYTES[case["precision"]]
    field = 4 * (8 if b == 8 else 4)
    return {"bytes": nodes * (2 * 19 * b + field + (19 * b if case.get("keep") else 0)),
            "flops": nodes * case["steps"] * FLOPS}


# -- the same in 64 bits, with tensor operations ----------------------------------------


def _close_face(g, at, axis, sign, u, rho):
    """Plane with inward normal sign e_axis on the nodes ``at``: velocity u prescribed, or
    (rho given) density and tangential velocity."""
    f = [g[k][at] for k in range(19)]
    total = sum(f[k] * (1 if C[k][axis] == 0 else 2) for k in range(19) if sign * C[k][axis] <= 0)
    u = list(u)
    if rho is None:
        rho = total / (1 - sign * u[axis])
    else:
        u[axis] = sign * (1 - total / rho)
    shift = [None] * 3
    for t in range(3):
        if t != axis:
            shift[t] = 0.5 * sum(f[k] * C[k][t] for k in range(19) if C[k][axis] == 0 and C[k][t]) - rho * u[t] / 3
    for k in range(19):
        if sign * C[k][axis] > 0:
            cu = sum(C[k][a] * u[a] for a in range(3) if C[k][a])
            g[k][at] = f[OPP[k]] + 6 * W[k] * rho * cu - sum(C[k][t] * shift[t] for t in range(3) if t != axis and C[k][t])


def _close_corner(g, at, normals, rho):
    """Concave edge (two normals, each (axis, sign)) or corner (three), at rest, on ``at``."""
    n = [0, 0, 0]
    for a, s in normals:
        n[a] = s
    unknown = [k for k in range(19) if any(s * C[k][a] > 0 for a, s in normals)]
    if len(normals) == 2:
        (a1, s1), (a2, s2) = normals
        link = [0, 0, 0]
        link[a1], link[a2] = s1, -s2
        buried = [C.index(tuple(link)), C.index(tuple(-v for v in link))]
        parts = (22, 14)
    else:
        buried = [k for k in range(18) if sum(C[k][a] * n[a] for a in range(3)) == 0]
        parts = (18, 18)
    f = [g[k][at].clone() for k in range(19)]
    for k in unknown:
        if k not in buried:
            f[k] = f[OPP[k]].clone()
    if len(normals) == 2:
        e = next(a for a in range(3) if n[a] == 0)
        plus = [0, 0, 0]
        plus[e] = 1
        k0 = C.index(tuple(plus))
        slip = 0.25 * (f[k0] - f[OPP[k0]])
        for k in unknown:
            if k not in buried and C[k][e]:
                f[k] = f[k] - C[k][e] * slip
    total = sum(f[k] for k in range(18) if k not in buried)
    fb = total / parts[0] if rho is None else (rho - total) / parts[1]
    for k in buried:
        f[k] = fb
    f[18] = 12 * fb
    for k in range(19):
        g[k][at] = f[k]


def _closures(dims, faces):
    """What has to be closed: functions of the streamed populations."""
    walled = [faces[2 * a] is not None for a in range(3)]
    ends = [(0, 1), (1, -1)]  # (which end, inward sign)
    out = []

    def region(fixed):
        # index of [z, y, x] with the fixed axes at an end and the others inside their walls
        idx = []
        for a in (2, 1, 0):
            if a in fixed:
                i = 0 if fixed[a] == 0 else dims[a] - 1
                idx.append(slice(i, i + 1))
            else:
                idx.append(slice(1, dims[a] - 1) if walled[a] else slice(None))
        return tuple(idx)

    def value(table, a, at):
        # a face's table is [second axis][first axis]; as an array over [z, y, x] nodes
        t = torch.as_tensor(table, dtype=torch.float64, device="cuda")
        return t.unsqueeze(2 - a)[at]

    open_axes = [a for a in range(3) if walled[a]]
    for a in open_axes:
        for e, s in ends:
            face, at = faces[2 * a + e], region({a: e})
            flat = tuple(slice(None) if i == 2 - a else v for i, v in enumerate(at))
            if isinstance(face, tuple) and face[0] == "rho":
                out.append(lambda g, at=at, a=a, s=s, r=face[1]: _close_face(g, at, a, s, (0.0, 0.0, 0.0), r))
            elif isinstance(face, np.ndarray):
                u = [value(face[..., j], a, flat) for j in range(3)]
                out.append(lambda g, at=at, a=a, s=s, u=u: _close_face(g, at, a, s, u, None))
            else:
                out.append(lambda g, at=at, a=a, s=s, u=face: _close_face(g, at, a, s, u, None))

    def density(fixed):
        for a, e in fixed.items():
            face = faces[2 * a + e]
            if isinstance(face, tuple) and face[0] == "rho":
                return face[1]
        return None

    groups = [(a, b) for i, a in enumerate(open_axes) for b in open_axes[i + 1:]]
    if len(open_axes) == 3:
        groups.append((0, 1, 2))
    for group in groups:
        for code in range(2 ** len(group)):
            fixed = {a: (code >> i) & 1 for i, a in enumerate(group)}
            normals = [(a, ends[fixed[a]][1]) for a in group]
            out.append(lambda g, at=region(fixed), n=normals, r=density(fixed): _close_corner(g, at, n, r))
    return out


def _velocity(f):
    rho = f.sum(0)
    c = torch.tensor(C, dtype=torch.float64, device=f.device)
    return rho, (c.T @ f.reshape(19, -1)).reshape(3, *f.shape[1:]) / rho


def _fields(f):
    rho = torch.empty(f.shape[1:], dtype=torch.float64, device=f.device)
    u = torch.empty((3, *f.shape[1:]), dtype=torch.float64, device=f.device)
    n = max(1, 4_000_000 // (f.shape[2] * f.shape[3]))
    for z in range(0, f.shape[1], n):
        rho[z:z + n], u[:, z:z + n] = _velocity(f[:, z:z + n])
    return rho, u


def _exact_one(flow, nx, ny, nz, tau, precision, steps, seed, keep):
    faces, solid, force, u_start = flow
    f = _start(nx, ny, nz, u_start, precision, seed).double()
    w = torch.tensor(W, dtype=torch.float64, device="cuda")
    shift = 0.0 if precision == "f64" else 1.0
    for k in range(19):
        f[k] += shift * W[k]
    before = _fields(f)[1]
    g = torch.empty_like(f)
    closures = _closures((nx, ny, nz), faces)
    c = torch.tensor(C, dtype=torch.float64, device="cuda")
    blocked = None
    if solid is not None:
        solid = torch.as_tensor(solid, device="cuda").bool()
        blocked = []
        for k in range(19):
            from_solid = torch.roll(solid, (C[k][2], C[k][1], C[k][0]), (0, 1, 2))
            for a in range(3):  # nothing streams in through a walled face
                if faces[2 * a] is not None and C[k][a]:
                    from_solid.select(2 - a, 0 if C[k][a] > 0 else -1).fill_(False)
            blocked.append(from_solid)
    planes = max(1, 4_000_000 // (nx * ny))
    for _ in range(steps):
        for k in range(19):
            g[k] = torch.roll(f[k], (C[k][2], C[k][1], C[k][0]), (0, 1, 2))
            if blocked is not None:
                g[k] = torch.where(blocked[k], f[OPP[k]], g[k])
        for close in closures:
            close(g)
        for z in range(0, nz, planes):
            at = slice(z, z + planes)
            rho, u = _velocity(g[:, at])
            if force is not None:
                for a in range(3):
                    u[a] += tau * force[a] / rho
            cu = (c @ u.reshape(3, -1)).reshape(19, *rho.shape)
            eq = cu.mul_(4.5 * cu + 3.0).add_(1.0 - 1.5 * (u * u).sum(0)).mul_(rho).mul_(w.reshape(19, 1, 1, 1))
            eq.sub_(g[:, at]).div_(tau).add_(g[:, at])
            f[:, at] = eq if solid is None else torch.where(solid[at], f[:, at], eq)
    del g
    rho, u = _fields(f)
    diff = (u - before).square_().sum().sqrt()
    out = {"residual": float(diff / u.square().sum().sqrt()), "mass": float(rho.sum()), "rho": rho, "u": u}
    if keep:
        for k in range(19):
            f[k] -= shift * W[k]
        out["populations"] = f
    return out


def exact(case, seed):
    if case["kind"] == "batch":
        out = []
        for i, (kind, nx, ny, nz, tau, speed, angle) in enumerate(_members(case)):
            e = _exact_one(_flow(kind, nx, ny, nz, speed, angle), nx, ny, nz, tau, case["precision"], case["steps"],
                           seed * 64 + i, False)
            out.append((e["residual"], e["mass"], e["rho"], e["u"]))
        return out
    dims = case["nx"], case["ny"], case["nz"]
    return _exact_one(_flow(case["kind"], *dims), *dims, case["tau"], case["precision"], case["steps"], seed * 64,
                      case["keep"])
