"""What the solvers are timed on: time steps of 2D cavities and
Rayleigh-Benard layers, uneven batches, 3D cavities and the heated cylinder,
each followed by the download of the fields.

A case is one window of a running simulation: the handle, its mesh and its
state exist, `run` takes `steps` time steps and reads the state back, as a
program does that monitors or stores a run.  Fields come back in the handle's
own precision: float32 tensors from FP32 handles, float64 from FP64 ones.

Values: the fluid starts near the conduction profile (or the free stream) with
smooth convection rolls and weak noise, velocities up to a few hundredths
(Ma = 0.1), as after a restart; wave numbers, phases and noise come from the
seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2202_13449_gb300 import capi, inputs

MA = 0.1
# floating point operations of one cell-update (each face and gradient once,
# a fused multiply-add as one), by solver and face stage (RTLBFS, TLBFS)
OPS = {"plane": (439, 755), "batch": (439, 755), "cube": (1463, 2291), "ring": (685,)}


def listed():
    return [
        # The smallest calls: a few steps of the stability map's mesh between
        # two looks at the wall Nusselt number; launches and latency count.
        dict(name="cavity50_short", kind="plane", nx=50, ny=50, phi=0.0, Ra=1e5, periodic=False,
             precision="fp32", scheme=0, steps=16, tune=False),
        # The validation case of Table 1 in double precision.
        dict(name="cavity64_fp64", kind="plane", nx=64, ny=64, phi=0.0, Ra=1e3, periodic=False,
             precision="fp64", scheme=0, steps=200, tune=True),
        # The headline workload: the stretched 512 x 512 cavity in FP32.
        dict(name="cavity512", kind="plane", nx=512, ny=512, phi=2.0, Ra=1e8, periodic=False,
             precision="fp32", scheme=0, steps=1000, tune=True),
        # An ordinary odd-sized stretched cavity, schedule left to the library.
        dict(name="cavity301x203", kind="plane", nx=301, ny=203, phi=1.5, Ra=1e6, periodic=False,
             precision="fp32", scheme=0, steps=1000, tune=False),
        # Rayleigh-Benard convection, periodic in x.
        dict(name="rb1024x512", kind="plane", nx=1024, ny=512, phi=0.0, Ra=1e6, periodic=True,
             precision="fp32", scheme=0, steps=500, tune=True),
        # A large mesh: the state does not fit in L2.
        dict(name="cavity4096", kind="plane", nx=4096, ny=4096, phi=2.0, Ra=1e8, periodic=False,
             precision="fp32", scheme=0, steps=100, tune=False),
        # The original face stage of Section 2.2, for comparisons of the two.
        dict(name="cavity512_tlbfs", kind="plane", nx=512, ny=512, phi=2.0, Ra=1e8, periodic=False,
             precision="fp32", scheme=1, steps=500, tune=True),
        # Many uneven cavities in one handle: parameter studies, the request loop.
        dict(name="batch256", kind="batch", count=256, spec_seed=1234, precision="fp32", steps=100,
             tune=True),
        # The cubic cavity of Table 5 on the paper's mesh, FP32 and FP64.
        dict(name="cubic80", kind="cube", nx=80, ny=80, nz=80, phi=1.8, Ra=1e6, precision="fp32",
             scheme=0, steps=300, tune=True),
        dict(name="cubic80_fp64", kind="cube", nx=80, ny=80, nz=80, phi=1.8, Ra=1e6,
             precision="fp64", scheme=0, steps=20, tune=True),
        # The heated cylinder of Table 4 on its body-fitted mesh.
        dict(name="cylinder450x300", kind="ring", nx=450, ny=300, Gr=100.0, precision="fp32",
             steps=500),
        # A double-precision continuation of a stretched 2D run.
        dict(name="cavity400_fp64", kind="plane", nx=400, ny=400, phi=2.4, Ra=1e8, periodic=False,
             precision="fp64", scheme=0, steps=40, tune=True),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _ra(rng, top, *n):
    """A Rayleigh number up to 10^top that the mesh resolves."""
    return round(10 ** rng.uniform(3, min(top, 2 + 2 * math.log10(min(n)))), 1)


def draw(rng):
    kind = rng.choice(["plane", "plane", "plane", "batch", "cube", "ring"])
    fp64 = rng.random() < 0.25
    prec = "fp64" if fp64 else "fp32"
    if kind == "plane":
        hi = 512 if fp64 else 4096
        nx, ny = _size(rng, 32, hi), _size(rng, 32, hi)
        budget = 4e6 if fp64 else 1.5e8  # cell-updates of a pass
        scheme = 1 if rng.random() < 0.15 else 0
        return dict(kind=kind, nx=nx, ny=ny, phi=round(rng.choice([0.0, rng.uniform(1.0, 2.4)]), 3),
                    Ra=_ra(rng, 8, nx, ny), periodic=rng.random() < 0.3,
                    precision=prec, scheme=scheme,
                    steps=int(min(1000, max(8, budget / (nx * ny) / (1 + scheme)))),
                    tune=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind=kind, count=_size(rng, 16, 512), spec_seed=rng.randrange(1 << 20),
                    precision="fp32", steps=rng.randrange(20, 100), tune=rng.random() < 0.5)
    if kind == "cube":
        hi = 90 if fp64 else 200
        n = [_size(rng, 24, hi) for _ in range(3)]
        cells = n[0] * n[1] * n[2]
        budget = 4e6 if fp64 else 6e7
        scheme = 1 if rng.random() < 0.15 else 0
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2],
                    phi=round(rng.choice([0.0, rng.uniform(1.0, 2.0)]), 3),
                    Ra=_ra(rng, 6, *n), precision=prec, scheme=scheme,
                    steps=int(min(300, max(6, budget / cells / (1 + scheme)))), tune=rng.random() < 0.5)
    nx, ny = _size(rng, 64, 512 if fp64 else 1800), _size(rng, 48, 384 if fp64 else 1200)
    budget = 3e6 if fp64 else 6e7
    return dict(kind=kind, nx=nx, ny=ny, Gr=round(rng.uniform(0, 1600), 1), precision=prec,
                steps=int(min(500, max(8, budget / (nx * ny)))))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _faces(n, phi):
    """n + 1 face coordinates on [0, n]: uniform, or Eq. 74's tanh stretching."""
    s = np.arange(n + 1) / n
    if phi > 0:
        s = 0.5 * (1.0 + np.tanh(phi * (2.0 * s - 1.0)) / np.tanh(phi))
        s[0], s[-1] = 0.0, 1.0
    return s * n


def _physics(L, Ra, Pr=0.71):
    nu = MA * L * math.sqrt(Pr / Ra)
    return nu, nu / Pr, MA * MA / L


def _time_step(faces, nu, chi):
    """Half the smallest width, capped by the explicit diffusive limit there."""
    w = min(float(np.min(np.diff(f))) for f in faces)
    return min(0.5 * w, (0.2 if len(faces) == 2 else 0.13) * w * w / max(nu, chi))


def _unit(f):
    c = 0.5 * (f[1:] + f[:-1])
    return (c - f[0]) / (f[-1] - f[0])


def _rolls2(xf, yf, periodic, seed):
    """(rho, u, v, T) of a cavity (hot west wall) or a layer heated from below."""
    g = inputs.rng(seed)
    x, y = _unit(np.asarray(xf))[None, :], _unit(np.asarray(yf))[:, None]
    k, m, a = int(g.integers(1, 4)), int(g.integers(1, 3)), g.uniform(0.01, 0.03)
    ph = g.uniform(0, 2 * np.pi) if periodic else 0.0
    kx = 2 * np.pi * k if periodic else np.pi * k
    sx, cx = np.sin(kx * x + ph), np.cos(kx * x + ph)
    sy, cy = np.sin(np.pi * m * y), np.cos(np.pi * m * y)
    sh = (len(yf) - 1, len(xf) - 1)
    nz = [g.uniform(-1.0, 1.0, size=sh) for _ in range(4)]
    T = (1.0 - y if periodic else 1.0 - x) + 0.1 * sx * sy
    return (1.0 + 1e-4 * nz[0], a * sx * cy + 1e-4 * nz[1], -a * cx * sy + 1e-4 * nz[2],
            T + 1e-3 * nz[3])


def _rolls3(f, seed):
    g = inputs.rng(seed)
    x, y, z = _unit(f[0])[None, None, :], _unit(f[1])[None, :, None], _unit(f[2])[:, None, None]
    a, k = g.uniform(0.01, 0.03), int(g.integers(1, 3))
    p = np.pi
    nz = [g.uniform(-1.0, 1.0, size=(len(f[2]) - 1, len(f[1]) - 1, len(f[0]) - 1)) for _ in range(5)]
    u = a * np.sin(p * k * x) * np.cos(p * z) * np.sin(p * y)
    w = -a * np.cos(p * k * x) * np.sin(p * z) * np.sin(p * y)
    v = 0.3 * a * np.sin(p * x) * np.sin(2 * p * y) * np.sin(p * z)
    T = x + 0.1 * np.sin(p * k * x) * np.sin(p * z)
    return (1.0 + 1e-4 * nz[0], u + 1e-4 * nz[1], v + 1e-4 * nz[2], w + 1e-4 * nz[3], T + 1e-3 * nz[4])


def _ring(case):
    """Mesh and physics of the heated cylinder (Re = 20, Pr = 0.7, D = 1)."""
    X, Y = inputs.cylinder_o_mesh(case["nx"], case["ny"])
    uinf = MA / math.sqrt(3.0)
    nu = uinf / 20.0
    chi = nu / 0.7
    w = min(float(np.min(np.diff(np.hypot(X, Y), axis=0))),
            float(np.min(np.hypot(np.diff(X, axis=1), np.diff(Y, axis=1)))))
    return X, Y, uinf, nu, chi, case["Gr"] * nu * nu, min(0.5 * w, 0.2 * w * w / max(nu, chi))


def _ring_state(X, Y, uinf, seed):
    g = inputs.rng(seed)
    sh = (X.shape[0] - 1, X.shape[1] - 1)
    xc = 0.25 * (X[1:, 1:] + X[1:, :-1] + X[:-1, 1:] + X[:-1, :-1])
    yc = 0.25 * (Y[1:, 1:] + Y[1:, :-1] + Y[:-1, 1:] + Y[:-1, :-1])
    r = np.hypot(xc, yc)
    near = np.exp(-(r - 0.5) / g.uniform(0.5, 1.5))
    nz = [g.uniform(-1.0, 1.0, size=sh) for _ in range(4)]
    return (1.0 + 1e-5 * nz[0], uinf * (1.0 - near) + 1e-5 * nz[1],
            0.1 * uinf * near * yc / r + 1e-5 * nz[2], near * (1.0 + 1e-3 * nz[3]))


def _batch(case):
    """(faces, Ra) of each cavity of a batch, by the batch workload's recipe."""
    return [(_faces(sp.n, sp.phi), sp.Ra) for sp in inputs.batch_specs(case["count"], case["spec_seed"])]


def _pinned(nbytes):
    return torch.empty(nbytes, dtype=torch.uint8, pin_memory=True)


def prepare(case, seed):
    prec = capi.FP64 if case["precision"] == "fp64" else capi.FP32
    if case["kind"] == "plane":
        xf, yf = _faces(case["nx"], case["phi"]), _faces(case["ny"], case["phi"])
        s = capi.Solver(xf, yf, prec)
        if case["periodic"]:
            s.set_bc(capi.WEST, capi.PERIODIC)
            s.set_bc(capi.EAST, capi.PERIODIC)
            s.set_bc(capi.SOUTH, capi.WALL_DIRICHLET, 1.0)
            s.set_bc(capi.NORTH, capi.WALL_DIRICHLET, 0.0)
        L = float(yf[-1] if case["periodic"] else xf[-1])
        nu, chi, _ = _physics(L, case["Ra"])
        s.set_params_ref(case["Ra"], 0.71, MA, _time_step((xf, yf), nu, chi), L)
        if case["scheme"]:
            s.set_scheme(capi.TLBFS)
        s.set_state(*_rolls2(xf, yf, case["periodic"], seed))
        if case["tune"]:
            s.autotune(16)
        # the records come back through a pinned buffer, as bench.py reads them
        return dict(case=case, solver=s, buf=_pinned(s.raw_bytes()))
    if case["kind"] == "batch":
        mesh = _batch(case)
        b = capi.Batch(prec, len(mesh))
        slots = []
        for k, (f, Ra) in enumerate(mesh):
            n = len(f) - 1
            nu, chi, _ = _physics(float(n), Ra)
            slots.append(b.add(f, f, Ra, 0.71, MA, _time_step((f, f), nu, chi)))
            b.set_state(slots[-1], *_rolls2(f, f, False, 1000 * seed + k))
        if case["tune"]:
            b.arm_many(slots, 0.0, 100)
            b.autotune(8)
        size = [b.raw_bytes(s) for s in slots]
        buf = _pinned(sum(size))
        at = np.concatenate([[0], np.cumsum(size)])
        host = buf.numpy()
        return dict(case=case, solver=b, slots=slots, buf=buf,
                    parts=[host[at[k]:at[k + 1]] for k in range(len(slots))])
    if case["kind"] == "cube":
        f = [_faces(case[a], case["phi"]) for a in ("nx", "ny", "nz")]
        s = capi.Solver3(*f, precision=prec)
        nu, chi, _ = _physics(float(f[0][-1]), case["Ra"])
        s.set_params(case["Ra"], 0.71, MA, _time_step(f, nu, chi))
        s.set_lattice(0.5)
        if case["scheme"]:
            s.set_scheme(capi.TLBFS)
        s.set_state(*_rolls3(f, seed))
        if case["tune"]:
            s.autotune(8)
        return dict(case=case, solver=s)
    X, Y, uinf, nu, chi, bg, dt = _ring(case)
    s = capi.SolverC(X, Y, True, prec)
    s.set_physics(nu, chi, bg, dt)
    s.set_gravity(1.0, 0.0, 0.0)
    s.set_bc(2, capi.WALL_DIRICHLET, 1.0)
    s.set_bc(3, capi.FARFIELD)
    s.set_farfield(1.0, uinf, 0.0, 0.0)
    s.set_state(*_ring_state(X, Y, uinf, seed))
    return dict(case=case, solver=s)


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _fields(buf, fp64, T_unit=1.0):
    """Cell records (rho - 1, u, v, T) as the four fields on the GPU."""
    if fp64:
        q = buf.view(torch.float64).view(-1, 4).cuda()
    else:
        unit = torch.tensor([2.0 ** -32, 2.0 ** -31, 2.0 ** -31, 2.0 ** -30 * T_unit], device="cuda")
        q = buf.view(torch.int32).view(-1, 4).cuda() * unit
    q[:, 0] += 1.0
    return dict(zip(("rho", "u", "v", "T"), q.unbind(1)))


def run(state):
    case, s = state["case"], state["solver"]
    fp64 = case["precision"] == "fp64"
    if case["kind"] == "plane":
        s.step(case["steps"])
        nu = None
        if case["steps"] < 50:  # a short window between two readings of the heat transfer
            nu = torch.tensor(s.nusselt(capi.NU_SOUTH if case["periodic"] else capi.NU_WEST),
                              dtype=torch.float64 if fp64 else torch.float32)
        T_unit = s.get_state_raw(state["buf"].numpy())[1]
        return dict(_fields(state["buf"], fp64, T_unit), nu=nu)
    if case["kind"] == "batch":
        s.arm_many(state["slots"], -1.0, case["steps"])
        s.step(case["steps"])
        s.get_states_raw(state["slots"], state["parts"])  # the walls' unit, 1, holds for all
        return _fields(state["buf"], fp64)
    s.step(case["steps"])
    out = s.get_state()
    return [torch.from_numpy(a if fp64 else a.astype(np.float32)) for a in out]


def work(case):
    steps, scheme = case["steps"], case.get("scheme", 0)
    if case["kind"] == "batch":
        cells = sum((len(f) - 1) ** 2 for f, _ in _batch(case))
    else:
        cells = case["nx"] * case["ny"] * case.get("nz", 1)
    # the state read once and written once; steps in between need no memory traffic
    record = (5 if case["kind"] == "cube" else 4) * (8 if case["precision"] == "fp64" else 4)
    return {"bytes": 2.0 * record * cells, "flops": float(OPS[case["kind"]][scheme]) * cells * steps}


# ---------------------------------------------------------------------------
# The same in 64 bits, from the paper's equations
# ---------------------------------------------------------------------------
CS2 = 1.0 / 3.0


def _lattice(D):
    axis = [tuple(s if i == a else 0 for i in range(D)) for a in range(D) for s in (-1, 1)]
    edge = [tuple(s if i == a else (t if i == b else 0) for i in range(D))
            for a in range(D) for b in range(a + 1, D) for s in (-1, 1) for t in (-1, 1)]
    return [(0,) * D] + axis + edge


def _face(pL, pR, gL, gR, h, nu, chi, wall, scheme):
    """Fluxes (mass, momenta, energy) along the normal of a set of faces.
    pL, pR: the two cells' planes at the face (rho, u_n, u_t.., T); gL, gR:
    [quantity][direction] gradients in the face frame; wall: 1 on wall faces
    (at rest), else 0.  The constant c_s^2 is left out of the pressure."""
    D = len(pL) - 2
    r = range(D)

    def node(o):
        out = []
        for k in range(D + 2):
            L = pL[k] + h * sum(o[a] * gL[k][a] for a in r if o[a]) if any(o) else pL[k]
            R = pR[k] + h * sum(o[a] * gR[k][a] for a in r if o[a]) if any(o) else pR[k]
            out.append(L if o[0] < 0 else (R if o[0] > 0 else 0.5 * (L + R)))
        return out

    N = {o: node(o) for o in _lattice(D)}
    O = (0,) * D
    open_ = 1.0 - wall

    def e(*s):
        o = [0] * D
        for a, v in s:
            o[a] = v
        return tuple(o)

    if scheme == 1:  # Section 2.2: equilibria at the nodes x_S - e_i h and their moments
        wt = {0: 4 / 9 if D == 2 else 1 / 3, 1: 1 / 9 if D == 2 else 1 / 18, 2: 1 / 36}

        def equil(q, c):
            w = wt[sum(abs(v) for v in c)]
            eu = sum(c[a] * q[1 + a] for a in r if c[a]) + 0.0 * q[0]
            u2 = sum(q[1 + a] * q[1 + a] for a in r)
            return w * (q[0] * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * u2) - 1), w * q[0] * q[-1] * (1 + 3 * eu)

        f = {c: equil(N[tuple(-v for v in c)], c) for c in N}
        rs = 1 + sum(f[c][0] for c in f)
        m = [sum(c[a] * f[c][0] for c in f if c[a]) * open_ for a in r]
        qs = [rs] + [m[a] / rs for a in r] + [sum(f[c][1] for c in f) / rs]
        F = [m[0]] + [0.0] * (D + 1)
        for c in f:
            if c[0]:
                fs, gs = equil(qs, c)
                pf = fs - 3 * nu / h * (fs - f[c][0])
                for a in r:
                    F[1 + a] = F[1 + a] + c[0] * c[a] * pf
                F[-1] = F[-1] + c[0] * (gs - 3 * chi / h * (gs - f[c][1]))
        return F

    mom = {o: [N[o][0] * N[o][1 + a] for a in r] for o in N}

    def X(o, a, b):
        x = mom[o][a] * N[o][1 + b]
        return x + CS2 * (N[o][0] - 1.0) if a == b else x

    def d(fn, a):
        return fn(e((a, 1))) - fn(e((a, -1)))

    def dd(fn, a, b):
        if a == b:
            return fn(e((a, 1))) - 2 * fn(O) + fn(e((a, -1)))
        return fn(e((a, 1), (b, 1))) - fn(e((a, 1), (b, -1))) - fn(e((a, -1), (b, 1))) + fn(e((a, -1), (b, -1)))

    M = lambda a: (lambda o: mom[o][a])  # noqa: E731
    E = lambda o: N[o][0] * N[o][-1]  # noqa: E731
    # Eqs. 46-48
    rs = N[O][0] - 0.5 * sum(d(M(a), a) for a in r)
    rs = rs + 0.5 * sum(dd(lambda o: X(o, a, a), a, a) for a in r)
    rs = rs + 0.25 * sum(dd(lambda o: X(o, a, b), a, b) for a in r for b in r if a < b)
    ms = []
    for a in r:
        br = sum(dd(M(a), b, b) for b in r) + 2 * dd(M(a), a, a)
        br = br + 0.5 * sum(dd(M(b), a, b) for b in r if b != a)
        ms.append(mom[O][a] - 0.5 * sum(d(lambda o: X(o, a, b), b) for b in r) + 0.5 * CS2 * br)
    es = E(O) - 0.5 * sum(d(lambda o: mom[o][a] * N[o][-1], a) for a in r)
    es = es + 0.5 * CS2 * sum(dd(E, a, a) for a in r)
    ms = [x * open_ for x in ms]
    us, Ts = [x / rs for x in ms], es / rs
    # Eqs. 57-59
    F = [ms[0]]
    tf, tg = 1 - 3 * nu / h, 1 - 3 * chi / h
    div = sum(d(M(a), a) for a in r)
    for a in r:
        X0 = X(O, a, 0)
        Xs = ms[a] * us[0] + (CS2 * (rs - 1.0) if a == 0 else 0.0)
        visc = d(M(a), 0) + d(M(0), a) + (div if a == 0 else 0.0)
        F.append(X0 + tf * (Xs - X0) - nu / (2 * h) * visc)
    Q0 = mom[O][0] * N[O][-1]
    F.append(Q0 + tg * (ms[0] * Ts - Q0) - chi / (2 * h) * d(E, 0))
    return F


def _update(q, div, src, dt):
    r1 = q[0] - div[0]
    out = [r1]
    for k in range(1, len(q)):
        s = dt * q[0] * src[k - 1] if k < len(q) - 1 and src[k - 1] is not None else 0.0
        out.append(q[k] + (q[k] * div[0] - div[k] + s) / r1)
    return out


def _march(q, w, nu, chi, bg, dt, kappa, bc, g_axis, scheme, steps):
    """`steps` steps on rectilinear meshes.  q: fields [batch, (z,) y, x]; w:
    widths per axis; bc per axis: "periodic" or the two wall temperatures
    (None: adiabatic); gravity along g_axis, T_ref = 1/2."""
    D = len(w)
    dim = [-(a + 1) for a in range(D)]
    cut = lambda t, a, i, n: t.narrow(dim[a], i, n)  # noqa: E731
    n = [q[0].shape[dim[a]] for a in range(D)]

    def extend(t, a, lo, hi):
        return torch.cat([lo(cut(t, a, 0 if bc[a] != "periodic" else n[a] - 1, 1)), t,
                          hi(cut(t, a, n[a] - 1 if bc[a] != "periodic" else 0, 1))], dim[a])

    same = lambda t: t  # noqa: E731
    we = [extend(w[a], a, same, same) for a in range(D)]
    wl = [cut(we[a], a, 0, n[a] + 1) for a in range(D)]
    wr = [cut(we[a], a, 1, n[a] + 1) for a in range(D)]
    h = [kappa * torch.minimum(wl[a], wr[a]) for a in range(D)]
    wall = []
    for a in range(D):
        z = torch.zeros(n[a] + 1, dtype=torch.float64, device=q[0].device)
        if bc[a] != "periodic":
            z[0] = z[-1] = 1.0
        wall.append(z.reshape([-1] + [1] * a))

    def odd(k, a, side):
        return 1 <= k <= D or (k == D + 1 and bc[a][side] is not None)

    def ghost_value(k, a, side):
        if bc[a] == "periodic" or not odd(k, a, side):
            return same
        return lambda t: (2.0 * bc[a][side] if k == D + 1 else 0.0) - t

    def ghost_slope(k, a, b, side):
        if bc[a] == "periodic" or odd(k, a, side) == (a == b):
            return same
        return lambda t: -t

    for _ in range(steps):
        ext = [[extend(q[k], a, ghost_value(k, a, 0), ghost_value(k, a, 1)) for a in range(D)]
               for k in range(D + 2)]
        grad = []
        for k in range(D + 2):
            grad.append([])
            for a in range(D):
                s = (cut(ext[k][a], a, 1, n[a] + 1) - cut(ext[k][a], a, 0, n[a] + 1)) / (wl[a] + wr[a])
                grad[k].append(cut(s, a, 1, n[a]) + cut(s, a, 0, n[a]))
        div = [0.0] * (D + 2)
        for a in range(D):
            fr = [(a + i) % D for i in range(D)]  # normal, tangents
            comp = [0] + [1 + b for b in fr] + [D + 1]
            pL, pR, gL, gR = [], [], [], []
            for k in comp:
                ge = [extend(grad[k][b], a, ghost_slope(k, a, b, 0), ghost_slope(k, a, b, 1)) for b in fr]
                gL.append([cut(x, a, 0, n[a] + 1) for x in ge])
                gR.append([cut(x, a, 1, n[a] + 1) for x in ge])
                pL.append(cut(ext[k][a], a, 0, n[a] + 1) + 0.5 * wl[a] * gL[-1][0])
                pR.append(cut(ext[k][a], a, 1, n[a] + 1) - 0.5 * wr[a] * gR[-1][0])
            F = _face(pL, pR, gL, gR, h[a], nu, chi, wall[a], scheme)
            for i, k in enumerate(comp):
                div[k] = div[k] + dt / w[a] * (cut(F[i], a, 1, n[a]) - cut(F[i], a, 0, n[a]))
        src = [None] * D
        src[g_axis] = bg * (q[D + 1] - 0.5)
        q = _update(q, div, src, dt)
    return q


def _march_ring(q, X, Y, nu, chi, bg, dt, uinf, steps):
    """`steps` steps on the O-mesh: periodic around, hot wall inside, far
    field outside, buoyancy along +x with T_ref = 0."""
    dev = q[0].device
    X, Y = (torch.as_tensor(a, dtype=torch.float64, device=dev) for a in (X, Y))
    quad = lambda A: (A[:-1, :-1], A[:-1, 1:], A[1:, 1:], A[1:, :-1])  # noqa: E731
    xs, ys = quad(X), quad(Y)
    cx, cy = sum(xs) / 4, sum(ys) / 4
    area = 0.5 * sum(xs[i] * ys[(i + 1) % 4] - xs[(i + 1) % 4] * ys[i] for i in range(4))
    # faces around (i) and outward (j): face vector S towards increasing index, midpoint
    Si = (Y[1:] - Y[:-1], -(X[1:] - X[:-1]))
    mi = (0.5 * (X[1:] + X[:-1]), 0.5 * (Y[1:] + Y[:-1]))
    Sj = (-(Y[:, 1:] - Y[:, :-1]), X[:, 1:] - X[:, :-1])
    mj = (0.5 * (X[:, 1:] + X[:, :-1]), 0.5 * (Y[:, 1:] + Y[:, :-1]))
    geo = []
    for axis, (S, m) in enumerate(((Si, mi), (Sj, mj))):
        ln = torch.hypot(*S)
        nn = (S[0] / ln, S[1] / ln)
        if axis == 0:
            c = [torch.cat([t[:, -1:], t, t[:, :1]], 1) for t in (cx, cy)]
            L, R = [t[:, :-1] for t in c], [t[:, 1:] for t in c]
        else:  # ghost centres: mirror images across the boundary edges
            c = [torch.zeros(cx.shape[0] + 2, cx.shape[1], dtype=torch.float64, device=dev) for _ in range(2)]
            for t, v in zip(c, (cx, cy)):
                t[1:-1] = v
            for g, p, fj in ((0, 1, 0), (-1, -2, -1)):
                dist = (m[0][fj] - c[0][p]) * nn[0][fj] + (m[1][fj] - c[1][p]) * nn[1][fj]
                for i in range(2):
                    c[i][g] = c[i][p] + 2 * dist * nn[i][fj]
            L, R = [t[:-1] for t in c], [t[1:] for t in c]
        dL, dR = [m[i] - L[i] for i in range(2)], [m[i] - R[i] for i in range(2)]
        aL, aR = torch.hypot(*dL), torch.hypot(*dR)
        wl = 2 * (dL[0] * nn[0] + dL[1] * nn[1]).abs()
        wr = 2 * (dR[0] * nn[0] + dR[1] * nn[1]).abs()
        wall = torch.zeros_like(ln)
        if axis == 1:
            wall[0] = 1.0
        geo.append((S, ln, nn, dL, dR, aR / (aL + aR), aL / (aL + aR), torch.minimum(wl, wr), wall))
    far = (1.0, uinf, 0.0, 0.0)
    nb = [g[0] for g in (geo[1][2][0], geo[1][2][1])]  # the wall's unit normal

    def ext_i(t):
        return torch.cat([t[:, -1:], t, t[:, :1]], 1)

    def pair(t, axis):
        return (t[:, :-1], t[:, 1:]) if axis == 0 else (t[:-1], t[1:])

    for _ in range(steps):
        ev = []
        for k in range(4):
            p = q[k][:1]
            lo = p if k == 0 else (-p if k < 3 else 2.0 - p)
            ev.append((ext_i(q[k]), torch.cat([lo, q[k], torch.full_like(p, far[k])], 0)))
        grad = []
        for k in range(4):
            g = []
            for c in range(2):
                tot = 0.0
                for axis in range(2):
                    S, aL, aR = geo[axis][0], geo[axis][5], geo[axis][6]
                    L, R = pair(ev[k][axis], axis)
                    f = (L * aL + R * aR) * S[c]
                    tot = tot + ((f[:, 1:] - f[:, :-1]) if axis == 0 else (f[1:] - f[:-1]))
                g.append(tot / area)
            grad.append(g)
        div = [0.0] * 4
        for axis in range(2):
            S, ln, nn, dL, dR, _, _, h, wall = geo[axis]
            pg, gg = [], []  # per quantity: planes at the face; gradients along n and t
            for k in range(4):
                if axis == 0:
                    ge = [ext_i(x) for x in grad[k]]
                else:
                    gn = grad[k][0][0] * nb[0] + grad[k][1][0] * nb[1]
                    sg = 1.0 if k == 0 else -1.0
                    ge = [torch.cat([(sg * (grad[k][c][0] - 2 * gn * nb[c]))[None], grad[k][c],
                                     torch.zeros_like(gn)[None]], 0) for c in range(2)]
                v, g0, g1 = pair(ev[k][axis], axis), pair(ge[0], axis), pair(ge[1], axis)
                pg.append([v[s] + g0[s] * d[0] + g1[s] * d[1] for s, d in ((0, dL), (1, dR))])
                gg.append([(g0[s] * nn[0] + g1[s] * nn[1], -g0[s] * nn[1] + g1[s] * nn[0]) for s in range(2)])

            def turn(a, b):  # (x, y) components to (n, t)
                return a * nn[0] + b * nn[1], -a * nn[1] + b * nn[0]

            sides = []
            for s in range(2):
                un, ut = turn(pg[1][s], pg[2][s])
                gr = [turn(gg[1][s][b], gg[2][s][b]) for b in range(2)]
                sides.append(([pg[0][s], un, ut, pg[3][s]],
                              [gg[0][s], (gr[0][0], gr[1][0]), (gr[0][1], gr[1][1]), gg[3][s]]))
            F = _face(sides[0][0], sides[1][0], sides[0][1], sides[1][1], h, nu, chi, wall, 0)
            F = [F[0], F[1] * nn[0] - F[2] * nn[1], F[1] * nn[1] + F[2] * nn[0], F[3]]
            for k in range(4):
                f = F[k] * ln
                div[k] = div[k] + dt / area * ((f[:, 1:] - f[:, :-1]) if axis == 0 else (f[1:] - f[:-1]))
        q = _update(q, div, [bg * q[3], None], dt)
    return q


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    up = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)  # noqa: E731
    if case["kind"] == "ring":
        X, Y, uinf, nu, chi, bg, dt = _ring(case)
        q = [up(a) for a in _ring_state(X, Y, uinf, seed)]
        return list(_march_ring(q, X, Y, nu, chi, bg, dt, uinf, case["steps"]))
    if case["kind"] == "batch":
        mesh = _batch(case)
        out = [None] * len(mesh)
        for n in sorted({len(f) for f, _ in mesh}):
            ids = [k for k, (f, _) in enumerate(mesh) if len(f) == n]
            st = [_rolls2(mesh[k][0], mesh[k][0], False, 1000 * seed + k) for k in ids]
            w = up([np.diff(mesh[k][0]) for k in ids])
            ph = [_physics(float(n - 1), mesh[k][1]) for k in ids]
            col = lambda v: up(v)[:, None, None]  # noqa: E731
            q = _march([up(np.stack([s[i] for s in st])) for i in range(4)], [w[:, None, :], w[:, :, None]],
                       col([p[0] for p in ph]), col([p[1] for p in ph]), col([p[2] for p in ph]),
                       col([_time_step((mesh[k][0],) * 2, p[0], p[1]) for k, p in zip(ids, ph)]),
                       1.0, [(1.0, 0.0), (None, None)], 1, 0, case["steps"])
            for j, k in enumerate(ids):
                out[k] = torch.stack([x[j].reshape(-1) for x in q], 1)
        return dict(zip(("rho", "u", "v", "T"), torch.cat(out).unbind(1)))
    names = ("nx", "ny", "nz") if case["kind"] == "cube" else ("nx", "ny")
    f = [_faces(case[a], case["phi"]) for a in names]
    w = [up(np.diff(f[a])).reshape([1, -1] + [1] * a) for a in range(len(f))]
    if case["kind"] == "cube":
        nu, chi, bg = _physics(float(f[0][-1]), case["Ra"])
        q = _march([up(a)[None] for a in _rolls3(f, seed)], w, nu, chi, bg, _time_step(f, nu, chi), 0.5,
                   [(0.0, 1.0), (None, None), (None, None)], 2, case["scheme"], case["steps"])
        return [x[0] for x in q]
    L = float(f[1][-1] if case["periodic"] else f[0][-1])
    nu, chi, bg = _physics(L, case["Ra"])
    bc = ["periodic", (1.0, 0.0)] if case["periodic"] else [(1.0, 0.0), (None, None)]
    q = _march([up(a)[None] for a in _rolls2(f[0], f[1], case["periodic"], seed)], w, nu, chi, bg,
               _time_step(f, nu, chi), 1.0, bc, 1, case["scheme"], case["steps"])
    return dict(zip(("rho", "u", "v", "T"), (x.reshape(-1) for x in q)))
