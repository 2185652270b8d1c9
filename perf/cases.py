"""Performance cases: what a user of the library has it do, through its public
entry points.

Every case is a dict of plain values.  `kind` says which call it makes:

  solve    one Helmholtz inverse (I - lam Delta) u = f or, with `lam` 0, the
           inverse Laplacian -Delta u = f, on a stretched box
  step     what one velocity-pressure time step asks for: three Dirichlet
           Helmholtz inverses at three time steps in one batched call and one
           zero-flux pressure Laplacian
  batch    independent Helmholtz inverses on uneven grids in one batched call
           (the right-hand sides of an Arnoldi-style iteration)
  stokes   one inverse of the staggered Stokes operator
  host     a sequence of Helmholtz inverses from and to host memory
  cyl      one Helmholtz inverse on a cylindrical grid

Sizes go from 8 to 256 cells per direction.  Grids are tanh-stretched boxes (the
workloads of the benchmark and the tests), right-hand sides uniform in [-1, 1],
forcings normal.  `precision` "fp64" or "mixed" is the plan's; `axis` 2, 1, 0 is
the Thomas direction, -2 the longest one, -1 the eigen decomposition in all
three directions; `walls` is one letter per direction: d (Dirichlet), n (zero
flux), m (Dirichlet below, zero flux above).  `own_stream`: the call is made on
a stream of the program's own, as the benchmark, the server and a pipelined
program do; otherwise on the current (default) stream, as in a first script.

`exact` solves the same problems in plain torch and numpy, in 64 bits.
"""
import math

import numpy as np
import torch

import paper_1107_2461_gb300 as fdi

_DEVICE = torch.device("cuda")
_STREAM = []


def _own_stream():
    # one stream for the whole program, made when first asked for
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


# --------------------------------------------------------------------------- the cases


def listed():
    return [
        # the smallest call: the plain FP64 eigen solve on a 16^3 box that the
        # first tests of the library use; all latency
        dict(name="fp64_16", kind="solve", precision="fp64", nx=16, ny=16, nz=16, beta=1.5, lam=1.0, axis=-1,
             walls="ddd", own_stream=True),
        # a small ragged box from a first script, on the default stream
        dict(name="mixed_ragged_75", kind="solve", precision="mixed", nx=75, ny=50, nz=67, beta=1.5, lam=1e-3, axis=2,
             walls="dnm", own_stream=False),
        # the four inverses of a time step at 128^3, refined mixed precision
        dict(name="mixed_step_128", kind="step", precision="mixed", nx=128, ny=128, nz=128, beta=2.0, Re=1000.0,
             own_stream=True),
        # the same in FP64: what a code without refinement asks for
        dict(name="fp64_step_128", kind="step", precision="fp64", nx=128, ny=128, nz=128, beta=2.0, Re=1000.0,
             own_stream=True),
        # the benchmark's workload, both precisions: the largest single solves
        dict(name="mixed_256", kind="solve", precision="mixed", nx=256, ny=256, nz=256, beta=1.5, lam=1.0, axis=2,
             walls="ddd", own_stream=True),
        dict(name="fp64_256", kind="solve", precision="fp64", nx=256, ny=256, nz=256, beta=1.5, lam=1.0, axis=2,
             walls="ddd", own_stream=True),
        # the eigen decomposition in all three directions on a ragged box
        dict(name="mixed_tpf_200", kind="solve", precision="mixed", nx=200, ny=100, nz=150, beta=1.5, lam=1e-2,
             axis=-1, walls="ddd", own_stream=True),
        # one large-time-step Stokes inverse as the server runs it (mixed, CG)
        dict(name="mixed_stokes_64", kind="stokes", precision="mixed", nx=64, ny=64, nz=64, beta=1.5, dt=1e3,
             Re=1000.0, krylov=2, own_stream=True),
        # a small-time-step Stokes inverse in FP64 with the default Krylov method
        dict(name="fp64_stokes_48", kind="stokes", precision="fp64", nx=48, ny=64, nz=40, beta=1.5, dt=1e-2,
             Re=1000.0, krylov=0, own_stream=True),
        # 64 uneven grids of an Arnoldi-style iteration in one call
        dict(name="mixed_batch_64", kind="batch", precision="mixed", count=64, grids=0, own_stream=True),
        # right-hand sides that live in host memory, copies pipelined
        dict(name="mixed_host_160", kind="host", precision="mixed", nx=160, ny=128, nz=192, beta=1.5, lam=0.1,
             count=6, own_stream=True),
        # an annulus: theta and z transforms, radial Thomas sweep
        dict(name="fp64_cyl_96", kind="cyl", precision="fp64", nr=96, ntheta=128, nz=80, r0=0.5, lam=1e-2, tpf=False,
             walls="ddd", own_stream=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["step", "batch", "stokes", "host", "cyl", "cyl"])
    precision = rng.choice(["fp64", "mixed"])
    beta = round(rng.uniform(1.0, 2.0), 3)
    own = rng.random() < 0.75
    if kind == "solve":
        n = [_log_int(rng, 8, 256) for _ in range(3)]
        lam = 0.0 if rng.random() < 0.2 else float("%.4g" % 10.0 ** rng.uniform(-4.0, 0.0))
        # at least one Dirichlet wall, or (the pressure problem) zero flux all round
        walls = "nnn" if lam == 0.0 and rng.random() < 0.5 else "d" + "".join(rng.choice("dnm") for _ in range(2))
        axis = rng.choice([2, 2, 2, -1, -2, 0, 1])
        if axis == -1 and precision == "fp64" and n[0] * n[1] * n[2] > 2**23:
            n[2] = max(8, n[2] // 2)  # no more work than the largest listed case
        return dict(kind=kind, precision=precision, nx=n[0], ny=n[1], nz=n[2], beta=beta, lam=lam, axis=axis,
                    walls=walls, own_stream=own)
    if kind == "step":
        n = [_log_int(rng, 24, 140) for _ in range(3)]
        return dict(kind=kind, precision=precision, nx=n[0], ny=n[1], nz=n[2], beta=beta,
                    Re=float(rng.choice([100, 1000, 5000])), own_stream=own)
    if kind == "batch":
        return dict(kind=kind, precision=precision, count=_log_int(rng, 2, 20), grids=rng.randrange(1, 1 << 20),
                    own_stream=own)
    if kind == "stokes":
        n = [_log_int(rng, 16, 72) for _ in range(3)]
        return dict(kind=kind, precision=precision, nx=n[0], ny=n[1], nz=n[2], beta=min(beta, 1.5),
                    dt=float("%.4g" % 10.0 ** rng.uniform(-2.0, 3.0)), Re=float(rng.choice([100, 1000, 5000])),
                    krylov=rng.choice([0, 2]), own_stream=True)
    if kind == "host":
        n = [_log_int(rng, 32, 200) for _ in range(3)]
        return dict(kind=kind, precision="mixed", nx=n[0], ny=n[1], nz=n[2], beta=beta,
                    lam=float("%.4g" % 10.0 ** rng.uniform(-4.0, 0.0)), count=rng.randint(2, 6), own_stream=True)
    return dict(kind=kind, precision=precision, nr=_log_int(rng, 16, 128), ntheta=_log_int(rng, 16, 144),
                nz=_log_int(rng, 16, 144), r0=rng.choice([0.0, 0.5, 1.0]),
                lam=float("%.4g" % 10.0 ** rng.uniform(-4.0, 0.0)),
                tpf=precision == "fp64" and rng.random() < 0.5, walls="d" + rng.choice("dnm") + rng.choice("dnm"),
                own_stream=own)


# --------------------------------------------------------------------------- inputs


def _tanh_faces(n, beta):
    s = np.arange(n + 1) / n
    x = 0.5 * (1.0 + np.tanh(beta * (2.0 * s - 1.0)) / np.tanh(beta))
    x[0], x[-1] = 0.0, 1.0
    return x


def _faces(c):
    return [_tanh_faces(c[k], c["beta"]) for k in ("nx", "ny", "nz")]


_WALLS = {"d": (0, 0), "n": (1, 1), "m": (0, 1)}


def _bcs(walls):
    return [_WALLS[w][0] for w in walls], [_WALLS[w][1] for w in walls]


def _prec(c):
    return fdi.PREC_FP64 if c["precision"] == "fp64" else fdi.PREC_MIXED_F16


def _generator(seed):
    return torch.Generator(device=_DEVICE).manual_seed(int(seed))


def _uniform(shape, g):
    return torch.rand(shape, generator=g, dtype=torch.float64, device=_DEVICE) * 2.0 - 1.0


def _batch_problems(c):
    """The uneven grids of a batch: cells from a few sizes with aspect at most
    1:4, stretching in [1, 2], lam log-uniform in [1e-4, 1]."""
    rng = np.random.default_rng(c["grids"])
    got = []
    while len(got) < c["count"]:
        n = [int(v) for v in rng.choice((32, 48, 64, 96, 128, 160), size=3)]
        if max(n) > 4 * min(n):
            continue
        got.append(dict(nx=n[0], ny=n[1], nz=n[2], beta=float(rng.uniform(1.0, 2.0)),
                        lam=float(10.0 ** rng.uniform(-4.0, 0.0)), walls="ddd"))
    return got


_STEP_DT = (1e-2, 1.0, 1e3)


def _mac_shapes(c):
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    return [(nz, ny, nx - 1), (nz, ny - 1, nx), (nz - 1, ny, nx)], (nz, ny, nx)


def _radial_faces(c):
    return c["r0"] + _tanh_faces(c["nr"], 1.0)


def _inputs(c, seed):
    """The right-hand sides of a case, on the GPU."""
    g = _generator(seed)
    kind = c["kind"]
    if kind in ("solve", "cyl"):
        shape = (c["nz"], c["ny"], c["nx"]) if kind == "solve" else (c["nz"], c["ntheta"], c["nr"])
        return [_uniform(shape, g)]
    if kind == "step":
        return [_uniform((c["nz"], c["ny"], c["nx"]), g) for _ in range(4)]
    if kind == "batch":
        return [_uniform((q["nz"], q["ny"], q["nx"]), g) for q in _batch_problems(c)]
    if kind == "host":
        return [_uniform((c["nz"], c["ny"], c["nx"]), g) for _ in range(c["count"])]
    return [torch.randn(s, generator=g, dtype=torch.float64, device=_DEVICE) for s in _mac_shapes(c)[0]]


def prepare(case, seed):
    c = case
    kind = c["kind"]
    s = {"kind": kind, "stream": _own_stream() if c["own_stream"] else None}
    f = _inputs(c, seed)
    if kind == "solve":
        lo, hi = _bcs(c["walls"])
        s["plan"] = fdi.plan_create(_faces(c), None, lo, hi, prec=_prec(c), thomas_axis=c["axis"])
        s["lam"] = c["lam"]
    elif kind == "step":
        s["plans"] = [fdi.plan_create(_faces(c), prec=_prec(c)) for _ in range(3)]
        s["pressure"] = fdi.plan_create(_faces(c), None, (1, 1, 1), (1, 1, 1), prec=_prec(c))
        s["lam"] = [dt / c["Re"] for dt in _STEP_DT]
    elif kind == "batch":
        q = _batch_problems(c)
        s["plans"] = [fdi.plan_create(_faces(x), prec=_prec(c)) for x in q]
        s["lam"] = [x["lam"] for x in q]
    elif kind == "host":
        s["plan"] = fdi.plan_create(_faces(c), prec=_prec(c))
        s["lam"] = c["lam"]
        f = [x.cpu().pin_memory() for x in f]
        s["out"] = [torch.empty(x.shape, dtype=torch.float64, pin_memory=True) for x in f]
    elif kind == "stokes":
        s["plan"] = fdi.plan_create(_faces(c), grid=fdi.GRID_MAC, prec=_prec(c))
        fdi.set_krylov(s["plan"], c["krylov"])
        s["dt"], s["Re"] = c["dt"], c["Re"]
        s["p"] = torch.empty(_mac_shapes(c)[1], dtype=torch.float64, device=_DEVICE)
    else:
        s["plan"] = fdi.plan_create_cyl(_radial_faces(c), c["ntheta"], _tanh_faces(c["nz"], 1.0),
                                        _WALLS[c["walls"][0]], _WALLS[c["walls"][2]], prec=_prec(c), tpf=c["tpf"])
        s["lam"] = c["lam"]
    s["f"] = f
    if "out" not in s:
        s["out"] = [torch.empty_like(x) for x in f]
    torch.cuda.synchronize()  # the inputs are made on another stream than the calls'
    return s


def run(state):
    s = state
    kind, f, out, stream = s["kind"], s["f"], s["out"], s["stream"]
    if kind == "solve":
        if s["lam"] == 0.0:
            fdi.laplace_solve(s["plan"], f[0], out[0], stream)
        else:
            fdi.helmholtz_solve(s["plan"], s["lam"], f[0], out[0], stream)
    elif kind == "step":
        fdi.helmholtz_solve_batched(s["plans"], s["lam"], f[:3], out[:3], stream)
        fdi.laplace_solve(s["pressure"], f[3], out[3], stream)
    elif kind == "batch":
        fdi.helmholtz_solve_batched(s["plans"], s["lam"], f, out, stream)
    elif kind == "host":
        fdi.field_solve_host(s["plan"], fdi.FIELD_CELL, 1.0, s["lam"], f, out, stream)
    elif kind == "stokes":
        fdi.stokes_solve(s["plan"], s["dt"], s["Re"], f, out, s["p"], stream)
        return {"u": out, "p": s["p"]}
    else:
        fdi.helmholtz_solve(s["plan"], s["lam"], f[0], out[0], stream)
    return out


def work(case):
    """One read of every right-hand side and one write of every solution; the
    two directions transformed forward and back (all three for axis -1) and
    the sweep of one direct solve."""
    c = case
    kind = c["kind"]

    def direct(n, tpf):
        return float(n[0] * n[1] * n[2]) * (4.0 * (n[0] + n[1] + (n[2] if tpf else 0)) + 8.0)

    if kind == "batch":
        probs = [(q["nx"], q["ny"], q["nz"]) for q in _batch_problems(c)]
        return {"bytes": 16.0 * sum(n[0] * n[1] * n[2] for n in probs), "flops": sum(direct(n, False) for n in probs)}
    if kind == "cyl":
        n = (c["nz"], c["ntheta"], c["nr"])
    else:
        n = (c["nx"], c["ny"], c["nz"])
        if kind == "solve" and c["axis"] in (0, 1, -2):
            # the Thomas direction last
            d = c["axis"] if c["axis"] >= 0 else max(range(3), key=lambda q: (n[q], q))
            n = tuple(n[q] for q in range(3) if q != d) + (n[d],)
    points = float(n[0] * n[1] * n[2])
    if kind == "stokes":
        # forcing in, velocity and pressure out; three predictor and three
        # corrector solves, at least one pressure-matrix product (three) and one
        # preconditioner solve
        return {"bytes": 8.0 * 7.0 * points, "flops": 10.0 * direct(n, False)}
    count = {"step": 4, "host": c.get("count", 1)}.get(kind, 1)
    tpf = c.get("axis") == -1 or bool(c.get("tpf"))
    return {"bytes": 16.0 * points * count, "flops": direct(n, tpf) * count}


# --------------------------------------------------------------------------- the same in plain torch, 64 bits


def _cell_operator(faces, lo, hi):
    """Widths m and the tridiagonal K (diagonal, off-diagonal) of the
    cell-centred second difference; walls 0 Dirichlet, 1 zero flux."""
    h = np.diff(faces)
    cen = 0.5 * (faces[1:] + faces[:-1])
    off = 1.0 / np.diff(cen)
    dia = np.zeros(h.size)
    dia[:-1] -= off
    dia[1:] -= off
    if lo == 0:
        dia[0] -= 2.0 / h[0]
    if hi == 0:
        dia[-1] -= 2.0 / h[-1]
    return h, dia, off


def _face_operator(faces):
    """The same for unknowns on the interior faces, zero at both walls."""
    h = np.diff(faces)
    cen = 0.5 * (faces[1:] + faces[:-1])
    return np.diff(cen), -(1.0 / h[:-1] + 1.0 / h[1:]), 1.0 / h[1:-1]


class _Direction:
    """One 1D operator: eigenvalues and basis of M^-1 K, and its fluxes."""

    def __init__(self, m, dia, off):
        sq = np.sqrt(m)
        S = np.diag(dia / m)
        o = off / (sq[1:] * sq[:-1])
        S += np.diag(o, 1) + np.diag(o, -1)
        lam, Q = np.linalg.eigh(S)
        to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(_DEVICE)  # noqa: E731
        wall = dia.copy()
        wall[:-1] += off
        wall[1:] += off
        wall[np.abs(wall) <= 1e-12 * np.abs(dia)] = 0.0
        self.singular = not wall.any()
        if self.singular:
            k = int(np.argmax(lam))
            lam[k] = 0.0
            Q[:, k] = sq / np.linalg.norm(sq)
        self.lam, self.m = to(lam), to(m)
        self.E, self.Einv = to(Q / sq[:, None]), to(Q.T * sq[None, :])
        self.off, self.wall = to(off), to(wall)


class _Box:
    """sigma I - lam Delta on a box: its action by fluxes and its inverse by
    eigen decomposition, refined until the residual stops falling."""

    def __init__(self, ops):
        self.d = [_Direction(*o) for o in ops]  # x, y, z
        self.singular = all(q.singular for q in self.d)
        self.V = self.d[2].m[:, None, None] * self.d[1].m[None, :, None] * self.d[0].m[None, None, :]

    def laplacian(self, u):
        out = torch.zeros_like(u)
        for q, axis in zip(self.d, (2, 1, 0)):
            shape = [1, 1, 1]
            shape[axis] = -1
            n = u.shape[axis]
            t = q.wall.view(shape) * u
            if n > 1:
                flux = q.off.view(shape) * (u.narrow(axis, 1, n - 1) - u.narrow(axis, 0, n - 1))
                t.narrow(axis, 0, n - 1).add_(flux)
                t.narrow(axis, 1, n - 1).sub_(flux)
            out += t / q.m.view(shape)
        return out

    def mean(self, u):
        return (u * self.V).sum() / self.V.sum()

    def direct(self, f, sigma, lam):
        x, y, z = self.d
        t = torch.matmul(f, x.Einv.T)
        t = torch.matmul(y.Einv, t)
        t = torch.tensordot(z.Einv, t, dims=([1], [0]))
        den = sigma - lam * (z.lam[:, None, None] + y.lam[None, :, None] + x.lam[None, None, :])
        if sigma == 0.0 and self.singular:
            den = torch.where(den == 0.0, torch.full_like(den, math.inf), den)
        t = t / den
        t = torch.tensordot(z.E, t, dims=([1], [0]))
        t = torch.matmul(y.E, t)
        return torch.matmul(t, x.E.T)

    def solve(self, f, sigma, lam, steps=2):
        null = sigma == 0.0 and self.singular
        if null:
            f = f - self.mean(f)
        u = self.direct(f, sigma, lam)
        for _ in range(steps):
            u = u + self.direct(f - (sigma * u - lam * self.laplacian(u)), sigma, lam)
        return u - self.mean(u) if null else u


def _exact_box(c, walls):
    lo, hi = _bcs(walls)
    return _Box([_cell_operator(f, lo[k], hi[k]) for k, f in enumerate(_faces(c))])


def _exact_stokes(c, f):
    faces = _faces(c)
    lam = c["dt"] / c["Re"]
    vel = [_Box([_face_operator(faces[d]) if d == k else _cell_operator(faces[d], 0, 0) for d in range(3)])
           for k in range(3)]
    prs = _Box([_cell_operator(faces[d], 1, 1) for d in range(3)])
    h = [torch.from_numpy(np.diff(x)).to(_DEVICE) for x in faces]
    dc = [torch.from_numpy(np.diff(0.5 * (x[1:] + x[:-1]))).to(_DEVICE) for x in faces]

    def shaped(v, axis):
        shape = [1, 1, 1]
        shape[axis] = -1
        return v.view(shape)

    def grad(p, k):
        axis = 2 - k
        n = p.shape[axis]
        return (p.narrow(axis, 1, n - 1) - p.narrow(axis, 0, n - 1)) / shaped(dc[k], axis)

    def div(u):
        out = torch.zeros(_mac_shapes(c)[1], dtype=torch.float64, device=_DEVICE)
        for k in range(3):
            axis = 2 - k
            n = out.shape[axis]
            t = torch.zeros_like(out)
            t.narrow(axis, 0, n - 1).add_(u[k])
            t.narrow(axis, 1, n - 1).sub_(u[k])
            out += t / shaped(h[k], axis)
        return out

    def apply(q):  # -C q, self-adjoint and positive in the volume-weighted product
        return -div([vel[k].solve(grad(q, k), 1.0, lam, 1) for k in range(3)])

    def precondition(r):  # -(L_p^-1 - lam) r, with L_p the zero-flux Laplacian
        return prs.solve(r, 0.0, 1.0, 1) + lam * r

    V = prs.V
    dot = lambda a, b: (V * a * b).sum()  # noqa: E731
    hat = [vel[k].solve(f[k], 1.0, lam) for k in range(3)]
    b = -div(hat)
    b -= prs.mean(b)
    q = torch.zeros_like(b)
    r, best, at_best = b.clone(), math.inf, q
    z = precondition(r)
    p, rz = z, dot(r, z)
    for it in range(200):
        Ap = apply(p)
        a = rz / dot(p, Ap)
        q = q + a * p
        r = r - a * Ap
        if it % 5 == 4:
            r = b - apply(q)
            r -= prs.mean(r)
            rel = float((dot(r, r) / dot(b, b)).sqrt())
            if rel < best:
                best, at_best = rel, q
            if rel < 1e-15 or rel > 0.5 * best and best < 1e-12 and rel != best:
                break
        z = precondition(r)
        rz_new = dot(r, z)
        p = z + (rz_new / rz) * p
        rz = rz_new
    q = at_best - prs.mean(at_best)
    u = [hat[k] - vel[k].solve(grad(q, k), 1.0, lam) for k in range(3)]
    return {"u": u, "p": q / c["dt"]}


def _exact_cyl(c, f):
    """Discrete Fourier transform along theta, eigenbasis along z, one
    symmetric radial eigenproblem per theta mode."""
    rho, M = _radial_faces(c), c["ntheta"]
    h = np.diff(rho)
    cen = 0.5 * (rho[1:] + rho[:-1])
    A = 0.5 * (rho[1:] ** 2 - rho[:-1] ** 2)
    off = rho[1:-1] / np.diff(cen)
    dia = np.zeros(h.size)
    dia[:-1] -= off
    dia[1:] -= off
    lo, hi = _WALLS[c["walls"][0]]
    if rho[0] > 0 and lo == 0:
        dia[0] -= rho[0] / (0.5 * h[0])
    if hi == 0:
        dia[-1] -= rho[-1] / (0.5 * h[-1])
    zl, zh = _WALLS[c["walls"][2]]
    z = _Direction(*_cell_operator(_tanh_faces(c["nz"], 1.0), zl, zh))
    ht = 2.0 * np.pi / M
    sq = np.sqrt(A)
    t = torch.fft.rfft(f, dim=1)
    out = torch.empty_like(t)
    K = np.diag(dia) + np.diag(off, 1) + np.diag(off, -1)
    for m in range(t.shape[1]):
        mu = -(2.0 * np.sin(np.pi * m / M) / ht) ** 2
        lr, Q = np.linalg.eigh((K + mu * np.diag(h / cen)) / (sq[:, None] * sq[None, :]))
        E = torch.from_numpy(Q / sq[:, None]).to(_DEVICE).to(t.dtype)
        Ei = torch.from_numpy(Q.T * sq[None, :]).to(_DEVICE).to(t.dtype)
        v = z.Einv.to(t.dtype) @ t[:, m, :] @ Ei.T
        v = v / (1.0 - c["lam"] * (z.lam[:, None] + torch.from_numpy(lr).to(_DEVICE)[None, :]))
        out[:, m, :] = z.E.to(t.dtype) @ v @ E.T
    return torch.fft.irfft(out, n=M, dim=1)


def exact(case, seed):
    c = case
    kind = c["kind"]
    f = _inputs(c, seed)
    if kind == "solve":
        box = _exact_box(c, c["walls"])
        return [box.solve(f[0], 0.0, 1.0) if c["lam"] == 0.0 else box.solve(f[0], 1.0, c["lam"])]
    if kind == "step":
        box = _exact_box(c, "ddd")
        got = [box.solve(f[k], 1.0, dt / c["Re"]) for k, dt in enumerate(_STEP_DT)]
        return got + [_exact_box(c, "nnn").solve(f[3], 0.0, 1.0)]
    if kind == "batch":
        return [_exact_box(q, "ddd").solve(x, 1.0, q["lam"]) for q, x in zip(_batch_problems(c), f)]
    if kind == "host":
        box = _exact_box(c, "ddd")
        return [box.solve(x, 1.0, c["lam"]).cpu() for x in f]
    if kind == "stokes":
        return _exact_stokes(c, f)
    return [_exact_cyl(c, f[0])]
