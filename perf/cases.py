"""What a user of this solver has it do, as calls that can be timed and checked.

A case is one call (or the short sequence of calls that belongs together) of the
public Python API: Runge-Kutta stepping of a device or a host state, one
right-hand side, a limited step, an adjoint step, a differentiated time
integration.  Meshes are the jittered split-square meshes of
``paper_1601_07944_gb300.inputs``; the initial states are projected here, with
this file's own rule and basis, so that a case's inputs do not depend on the
library.  ``exact`` is the same method written densely in torch float64 (basis
tables, Euler flux, local Lax-Friedrichs flux, limiter, Runge-Kutta schemes; the
adjoint by torch's reverse mode).
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1601_07944_gb300 import autograd, dg, inputs

GAMMA = 1.4
STAGES = {"ssp_rk3": 3, "rk2": 2, "rk4": 4}
DEV = "cuda" if torch.cuda.is_available() else "cpu"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _case(name=None, **kw):
    c = dict(call="step", n=64, p=3, ne=0, rule="collapsed", precision="fp64", method="ssp_rk3", steps=1, box="",
             limiter=False, data="perturbed")
    unknown = set(kw) - set(c)
    if unknown:
        raise ValueError("unknown case fields %s" % sorted(unknown))
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one step of the 512-element mesh in a loop that looks at every state
        _case("step_16_p1", n=16, p=1),
        # a whole small run in one call: the low end of the mesh-size sweep (800 elements, p = 4, classical RK4)
        _case("rk4_20_p4", n=20, p=4, method="rk4", steps=20),
        # shock-capturing: p = 1, classical RK2, every stage limited, about the paper's 68,622-element mesh
        _case("limited_185_p1", n=185, p=1, method="rk2", steps=5, limiter=True, data="bands"),
        # one right-hand side for a caller's own integrator, with walls and prescribed states; a ragged mesh
        _case("rhs_box_181_p2", call="rhs", n=181, p=2, box="wall_state", data="still"),
        # the float64 throughput workload: one step and the conserved totals that a run monitors
        _case("monitored_256_p3", call="monitored", n=256, p=3),
        # the same state kept in page-locked host memory by the caller
        _case("host_256_p3", call="host", n=256, p=3),
        # many steps per call on the tensor cores at single TF32
        _case("run_256_p3_tf32x1", n=256, p=3, precision="tf32x1", steps=20),
        # the mixed-precision workload: 524,288 elements, p = 4, split TF32
        _case("run_512_p4_tf32x3", n=512, p=4, precision="tf32x3", steps=5),
        # the largest: the highest degree in float64 (half a million elements, 44 million unknowns)
        _case("run_512_p5", n=512, p=5, steps=2),
        # the paper's own point counts: symmetric volume rule, classical RK4, an odd mesh
        _case("symmetric_151_p2", n=151, p=2, rule="symmetric", method="rk4", steps=2),
        # one transposed step of a caller's own reverse sweep
        _case("adjoint_256_p2", call="adjoint", n=256, p=2),
        # gradient of a run: forward, checkpoints, backward through torch.autograd
        _case("gradient_128_p2", call="gradient", n=128, p=2, steps=10),
    ]


def draw(rng):
    """One more case of the same ranges: any call, degree, rule, precision and
    method, meshes from 4 x 4 to 512 x 512 squares (log-uniform, odd sizes too)."""
    call = rng.choice(["step", "step", "step", "step", "limited", "rhs", "monitored", "host", "adjoint", "gradient"])
    c = {"call": "step" if call == "limited" else call}
    p = 1 if call == "limited" else rng.randint(1, 3) if call in ("adjoint", "gradient") else rng.randint(1, 5)
    c["p"] = p
    top = {"gradient": 128, "adjoint": 256}.get(call, 512)
    c["n"] = int(round(math.exp(rng.uniform(math.log(4), math.log(top)))))
    if call in ("step", "rhs", "monitored", "host") and rng.random() < 0.4:
        c["precision"] = rng.choice(["tf32x1", "tf32x3"])
    if call in ("step", "rhs", "monitored") and p == 2 and rng.random() < 0.4:
        c["rule"] = "symmetric"
    if p == 3 and call in ("step", "rhs", "monitored") and rng.random() < 0.3:
        c["ne"] = 3
    if call == "step" and rng.random() < 0.4:
        c["method"] = rng.choice(["rk2", "rk4"])
    if call == "limited":
        c.update(limiter=True, data="bands", method=rng.choice(["ssp_rk3", "rk2", "rk4"]))
    if call in ("step", "rhs", "adjoint") and rng.random() < 0.3:
        c["box"] = rng.choice(["wall_state", "wall_wall", "state_state"])
        c["data"] = "still"
    if call == "gradient":
        c["steps"] = rng.randint(2, 12)
    elif call in ("step", "limited", "host"):
        # at most the largest listed case's unknowns times stages
        dof = 2 * c["n"] ** 2 * 2 * (p + 1) * (p + 2) * STAGES[c.get("method", "ssp_rk3")]
        c["steps"] = rng.randint(1, max(1, min(24, int(2e8 // dof))))
        if call == "host":
            c["steps"] = min(2, c["steps"])
    return _case(**c)


# ---------------------------------------------------------------------------
# reference element: rules and basis (numpy, float64)
# ---------------------------------------------------------------------------

def _jacobi(n, a, b, x):
    """P_0..P_n^{(a,b)} and their derivatives at x."""
    x = np.asarray(x, dtype=np.longdouble)
    P = [np.ones_like(x)]
    D = [np.zeros_like(x)]
    if n >= 1:
        P.append(((a - b) + (a + b + 2) * x) / 2)
        D.append(np.full_like(x, (a + b + 2) / 2))
    for k in range(2, n + 1):
        c = 2 * k + a + b
        a1 = 2 * k * (k + a + b) * (c - 2)
        a2 = (c - 1) * (a * a - b * b)
        a3 = (c - 1) * c * (c - 2)
        a4 = 2 * (k + a - 1) * (k + b - 1) * c
        P.append(((a2 + a3 * x) * P[k - 1] - a4 * P[k - 2]) / a1)
        D.append((a3 * P[k - 1] + (a2 + a3 * x) * D[k - 1] - a4 * D[k - 2]) / a1)
    return P, D


def _gauss(n, a):
    """Gauss-Jacobi rule of n points for the weight (1-x)^a, a in (0, 1):
    Golub-Welsch start values, polished by Newton's method on P_n^{(a,0)}."""
    k = np.arange(n, dtype=np.float64)
    if a == 0:
        diag = np.zeros(n)
    else:
        diag = -1.0 / ((2 * k + 1) * (2 * k + 3))
    k = k[1:]
    off = 2.0 / (2 * k + a) * np.sqrt(k * (k + a) * k * (k + a) / ((2 * k + a + 1) * (2 * k + a - 1)))
    x = np.linalg.eigvalsh(np.diag(diag) + np.diag(off, 1) + np.diag(off, -1)).astype(np.longdouble)
    for _ in range(4):
        P, D = _jacobi(n, a, 0, x)
        x = x - P[n] / D[n]
    P, D = _jacobi(n, a, 0, x)
    w = np.longdouble(2) ** (a + 1) / ((1 - x * x) * D[n] ** 2)
    return x.astype(np.float64), w.astype(np.float64)


def _basis(p, r, s):
    """Orthonormal Dubiner basis (ordered by degree, then second index) and its
    gradients at (r, s): three arrays [points, N_p]."""
    r = np.asarray(r, dtype=np.longdouble)
    s = np.asarray(s, dtype=np.longdouble)
    t = 1 - s
    z = 2 * r - t
    # Q_a = t^a P_a(z / t), polynomial in (r, s): (a+1) Q_{a+1} = (2a+1) z Q_a - a t^2 Q_{a-1}
    Q, Qr, Qs = [np.ones_like(r)], [np.zeros_like(r)], [np.zeros_like(r)]
    for a in range(p):
        q0 = Q[a - 1] if a else 0 * r
        qr0 = Qr[a - 1] if a else 0 * r
        qs0 = Qs[a - 1] if a else 0 * r
        Q.append(((2 * a + 1) * z * Q[a] - a * t * t * q0) / (a + 1))
        Qr.append(((2 * a + 1) * (2 * Q[a] + z * Qr[a]) - a * t * t * qr0) / (a + 1))
        Qs.append(((2 * a + 1) * (Q[a] + z * Qs[a]) - a * (-2 * t * q0 + t * t * qs0)) / (a + 1))
    f, fr, fs = [], [], []
    for d in range(p + 1):
        for b in range(d + 1):
            a = d - b
            P, D = _jacobi(b, 2 * a + 1, 0, 2 * s - 1)
            norm = np.sqrt(np.longdouble(2 * (2 * a + 1) * (a + b + 1)))
            f.append(norm * Q[a] * P[b])
            fr.append(norm * Qr[a] * P[b])
            fs.append(norm * (Qs[a] * P[b] + 2 * Q[a] * D[b]))
    return tuple(np.stack(v, -1).astype(np.float64) for v in (f, fr, fs))


def _symmetric_p2():
    """The 6-point fully symmetric rule of degree 4: two orbits (a, a, 1-2a), from
    its moment conditions by Newton's method."""
    def moment(i, j):
        return math.factorial(i) * math.factorial(j) / math.factorial(i + j + 2)

    def points(a):
        return np.array([[a, a], [a, 1 - 2 * a], [1 - 2 * a, a]], dtype=np.longdouble)

    mons = [(0, 0), (2, 0), (2, 1), (2, 2)]
    v = np.array([0.4459, 0.1117, 0.0916, 0.0550], dtype=np.longdouble)   # a1, w1, a2, w2

    def res(v):
        out = []
        for i, j in mons:
            t = -np.longdouble(moment(i, j))
            for a, w in ((v[0], v[1]), (v[2], v[3])):
                P = points(a)
                t = t + w * (P[:, 0] ** i * P[:, 1] ** j).sum()
            out.append(t)
        return np.array(out, dtype=np.longdouble)

    for _ in range(30):
        f = res(v)
        J = np.stack([(res(v + h) - res(v - h)) / 2e-6
                      for h in (np.eye(4, dtype=np.longdouble)[k] * np.longdouble(1e-6) for k in range(4))], 1)
        v = v - np.linalg.solve(J.astype(np.float64), f.astype(np.float64)).astype(np.longdouble)
    pts = np.concatenate([points(v[0]), points(v[2])])
    w = np.concatenate([np.full(3, v[1]), np.full(3, v[3])])
    return pts[:, 0].astype(np.float64), pts[:, 1].astype(np.float64), w.astype(np.float64)


@functools.lru_cache(maxsize=None)
def _collapsed(p):
    xa, wa = _gauss(p + 1, 0)
    xb, wb = _gauss(p + 1, 1)
    B, A = np.meshgrid(xb, xa, indexing="ij")
    s = (1 + B) / 2
    r = (1 + A) / 2 * (1 - s)
    w = (wb[:, None] * wa[None, :]) / 8
    return r.reshape(-1), s.reshape(-1), w.reshape(-1)


@functools.lru_cache(maxsize=None)
def _tables(p, ne, rule):
    """Volume rule and basis tables, edge rule and traces, as float64 tensors."""
    if rule == "collapsed":
        r, s, w = _collapsed(p)
    elif p == 2:
        r, s, w = _symmetric_p2()
    else:
        return None
    f, fr, fs = _basis(p, r, s)
    xi, om = _gauss(ne or p + 1, 0)
    faces = [((1 + xi) / 2, 0 * xi), ((1 - xi) / 2, (1 + xi) / 2), (0 * xi, (1 - xi) / 2)]
    T = np.stack([_basis(p, a, b)[0] for a, b in faces])                   # [3, ne, N_p]
    to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)       # noqa: E731
    return dict(phi=to(f), dr=to(w[:, None] * fr), ds=to(w[:, None] * fs), tr=to(T), om=to(om),
                lift=to(T * om[None, :, None]), face_r=np.stack([a for a, _ in faces]),
                face_s=np.stack([b for _, b in faces]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _mesh(case, seed):
    code = {"wall": inputs.BC_WALL, "state": inputs.BC_STATE}
    if case["box"]:
        x, y = case["box"].split("_")
        return inputs.box_mesh(case["n"], code[x], code[y], seed=seed)
    return inputs.periodic_mesh(case["n"], seed=seed)


def _wrap(d):
    return d - 10.0 * torch.floor((d + 5.0) / 10.0)


def _state(case, seed, x, y):
    """Conserved initial state [..., 4] at the points (x, y) (tensors)."""
    if case["data"] == "bands":
        # two gases at rest, separated by discontinuities
        shift = 0.5 * (2.0 * float(inputs.uniform01(seed + 7, 1)[0]) - 1.0)
        inside = (x - shift).abs() < 2.5
        rho = torch.where(inside, 1.0, 0.125).to(x.dtype)
        pr = torch.where(inside, 1.0, 0.1).to(x.dtype)
        u = v = torch.zeros_like(x)
    elif case["data"] == "still":
        rho, u, v, pr = torch.ones_like(x), torch.zeros_like(x), torch.zeros_like(x), torch.ones_like(x)
    else:
        # isentropic vortex on a uniform stream
        xr, yr = _wrap(x), _wrap(y)
        g = torch.exp(0.5 * (1.0 - xr * xr - yr * yr))
        u = 1.0 - 5.0 / (2.0 * math.pi) * g * yr
        v = 1.0 + 5.0 / (2.0 * math.pi) * g * xr
        rho = (1.0 - (GAMMA - 1.0) * 25.0 / (8.0 * GAMMA * math.pi ** 2) * g * g) ** (1.0 / (GAMMA - 1.0))
        pr = rho ** GAMMA
    if case["data"] != "bands":
        # smooth seeded perturbations of density and pressure
        a, th = inputs.fourier_coefficients(seed + 2)
        rho, pr = rho.clone(), pr.clone()
        for q, f in enumerate((rho, pr)):
            for kx in range(1, 5):
                for ky in range(1, 5):
                    ph = 2.0 * math.pi * (kx * x + ky * y) / 10.0 + float(th[q, kx - 1, ky - 1])
                    f += 1e-2 * float(a[q, kx - 1, ky - 1]) * torch.sin(ph)
    E = pr / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)
    return torch.stack([rho, rho * u, rho * v, E], -1)


def _points(xy, r, s):
    """Physical points [N, len(r)] of reference points, xy [N, 3, 2] a tensor."""
    r = torch.from_numpy(np.ascontiguousarray(r)).to(xy)
    s = torch.from_numpy(np.ascontiguousarray(s)).to(xy)
    P = xy[:, 0, None] + r[None, :, None] * (xy[:, 1] - xy[:, 0])[:, None] + s[None, :, None] * (xy[:, 2] - xy[:, 0])[:, None]
    return P[..., 0], P[..., 1]


def _coefficients(case, seed, xy):
    """L2 projection [N, 4, N_p] of the initial state on the collapsed rule."""
    r, s, w = _collapsed(case["p"])
    B = torch.from_numpy(w[:, None] * _basis(case["p"], r, s)[0]).to(xy)
    out = []
    for part in xy.split(131072):
        U = _state(case, seed, *_points(part, r, s))
        out.append(torch.einsum("ekm,kj->emj", U, B))
    return torch.cat(out).contiguous()


def _dt(case, mesh, seed):
    ic = lambda x, y: _state(case, seed, torch.from_numpy(np.ascontiguousarray(x)).to(DEV),  # noqa: E731
                             torch.from_numpy(np.ascontiguousarray(y)).to(DEV)).cpu().numpy()
    return inputs.fixed_dt(mesh, ic, case["p"])


def _boundary(case, seed, mesh, xy, ne):
    """(element, face) of the boundary faces in element order, and the state
    prescribed at their points [Nb, n_e, 4]."""
    e, q = np.nonzero(mesh.nbr < 0)
    T = _tables(case["p"], ne, "collapsed")
    out = torch.empty((len(e), T["face_r"].shape[1], 4), dtype=torch.float64, device=xy.device)
    for f in range(3):
        x, y = _points(xy, T["face_r"][f], T["face_s"][f])
        sel = torch.from_numpy(np.nonzero(q == f)[0]).to(xy.device)
        el = torch.from_numpy(e[q == f]).to(xy.device)
        out[sel] = _state(case, seed, x[el], y[el])
    return e, q, out


def _inputs(case, seed):
    mesh = _mesh(case, 1 + seed)
    xy = torch.from_numpy(mesh.elem_xy).to(DEV)
    c = _coefficients(case, seed, xy)
    dt = _dt(case, mesh, seed)
    bst = _boundary(case, seed, mesh, xy, case["ne"])[2] if case["box"] else None
    lam = None
    if case["call"] in ("adjoint", "gradient"):
        g = torch.Generator().manual_seed(seed + 11)
        lam = torch.randn(c.shape, generator=g, dtype=torch.float64).to(DEV)
    return mesh, xy, c, dt, bst, lam


def prepare(case, seed):
    mesh, _, c, dt, bst, lam = _inputs(case, seed)
    m = dg.Mesh.from_mesh(mesh, case["p"], n_edge_pts=case["ne"], vol_rule=case["rule"])
    if bst is not None:
        m.set_boundary_state(bst)
    if case["limiter"]:
        m.set_limiter(True)
        m.limit(c)
    st = dict(case=case, mesh=m, c=c, dt=dt, lam=lam)
    if case["call"] == "host":
        st["c"] = c.cpu().pin_memory()
    if case["call"] in ("rhs", "adjoint"):
        st["out"] = torch.empty_like(c)
    if case["call"] == "gradient":
        st["c"] = c.requires_grad_(True)
    return st


def run(st):
    case, m, c = st["case"], st["mesh"], st["c"]
    call = case["call"]
    if call == "rhs":
        return m.rhs(c, out=st["out"], precision=case["precision"])
    if call == "host":
        return m.rk_step_host(c, st["dt"], case["steps"], precision=case["precision"])
    if call == "adjoint":
        return m.adjoint_step(c, st["dt"], st["lam"], out=st["out"])
    if call == "gradient":
        cT = autograd.solve(m, c, st["dt"], case["steps"], every=5)
        g, = torch.autograd.grad(cT, c, st["lam"])
        return [cT.detach(), g]
    m.rk_step(c, st["dt"], case["steps"], precision=case["precision"], method=case["method"])
    if call == "monitored":
        return [c, m.conserved_totals(c)]
    return c


def work(case):
    """State (and cotangent) read and written once, the mesh's vertices read once;
    the arithmetic of the sum-factorised contractions, the point fluxes, the lift,
    the stage update and the edge fluxes."""
    p, N = case["p"], 2 * case["n"] ** 2
    nd, npm, ne = p + 1, (p + 1) * (p + 2) // 2, case["ne"] or p + 1
    nq = 6 if case["rule"] == "symmetric" else nd * nd
    state = N * 4 * npm * 8
    volume = 4 * 2 * (npm * nd + nd ** 3) * 3 if case["rule"] == "collapsed" else 4 * 2 * nq * npm * 3
    edges = 4 * 2 * (npm * ne + nd * ne) * 2
    stage = N * (volume + edges + 45 * nq + 4 * npm * 6 + 1.5 * ne * 90)
    call = case["call"]
    steps = case["steps"]
    evals = 1 if call == "rhs" else STAGES[case["method"]] * steps
    reads = {"adjoint": 3, "gradient": 4}.get(call, 2)
    # a transposed step needs the two inner stages again and about twice a stage's arithmetic for each of its three
    times = {"adjoint": 2 + 2 * 3, "gradient": evals * (1 + 1 + 2)}.get(call, evals)
    return {"bytes": float(reads * state + N * 6 * 8), "flops": float(stage * times)}


# ---------------------------------------------------------------------------
# the method in torch float64
# ---------------------------------------------------------------------------

class _Reference:
    def __init__(self, case, seed):
        self.mesh, xy, self.c0, self.dt, bst, self.lam = _inputs(case, seed)
        self.T = _tables(case["p"], case["ne"], case["rule"])
        self.limiter = case["limiter"]
        d1, d2 = xy[:, 1] - xy[:, 0], xy[:, 2] - xy[:, 0]
        self.det = d1[:, 0] * d2[:, 1] - d1[:, 1] * d2[:, 0]
        self.jr = torch.stack([d2[:, 1], -d2[:, 0]], -1)                   # G_r = jr . (F1, F2)
        self.js = torch.stack([-d1[:, 1], d1[:, 0]], -1)
        e = xy[:, [1, 2, 0]] - xy
        ln = e.norm(dim=-1)
        self.half = 0.5 * ln
        self.nx, self.ny = e[..., 1] / ln, -e[..., 0] / ln
        nbr = torch.from_numpy(self.mesh.nbr).to(xy.device)
        nf = torch.from_numpy(self.mesh.nbr_face.astype(np.int64)).to(xy.device)
        self.nbr = nbr
        self.across = (3 * nbr + nf).clamp(min=0)
        self.inner = nbr >= 0
        self.bnd = None
        if case["box"]:
            be, bq, _ = _boundary(case, seed, self.mesh, xy, case["ne"])
            self.bnd = (torch.from_numpy(be).to(xy.device), torch.from_numpy(bq).to(xy.device), bst)

    def flux(self, U, ax, ay):
        """Euler flux of U[..., 4] along the direction (ax, ay)."""
        rho, mx, my, E = U.unbind(-1)
        u, v = mx / rho, my / rho
        pr = (GAMMA - 1.0) * (E - 0.5 * (mx * u + my * v))
        vn = u * ax + v * ay
        return torch.stack([rho * vn, mx * vn + pr * ax, my * vn + pr * ay, (E + pr) * vn], -1), vn, pr

    def rhs(self, c):
        T = self.T
        U = torch.einsum("emj,kj->ekm", c, T["phi"])
        Gr = self.flux(U, self.jr[:, None, 0], self.jr[:, None, 1])[0]
        Gs = self.flux(U, self.js[:, None, 0], self.js[:, None, 1])[0]
        V = torch.einsum("ekm,kj->emj", Gr, T["dr"]) + torch.einsum("ekm,kj->emj", Gs, T["ds"])
        Ul = torch.einsum("emj,qkj->eqkm", c, T["tr"])
        N, _, ne, _ = Ul.shape
        Ur = Ul.reshape(N * 3, ne, 4)[self.across.reshape(-1)].flip(1).reshape(N, 3, ne, 4)
        if self.bnd is not None:
            be, bq, bst = self.bnd
            code = self.nbr[be, bq]
            Ub = Ul[be, bq]
            nx, ny = self.nx[be, bq][:, None], self.ny[be, bq][:, None]
            mn = Ub[..., 1] * nx + Ub[..., 2] * ny
            wall = torch.stack([Ub[..., 0], Ub[..., 1] - 2 * mn * nx, Ub[..., 2] - 2 * mn * ny, Ub[..., 3]], -1)
            ghost = torch.where((code == inputs.BC_WALL)[:, None, None], wall, bst)
            Ur = Ur.index_put((be, bq), ghost)
        nx, ny = self.nx[..., None], self.ny[..., None]
        Fl, vl, pl = self.flux(Ul, nx, ny)
        Fr, vr, pr = self.flux(Ur, nx, ny)
        a = torch.maximum(vl.abs() + torch.sqrt(GAMMA * pl / Ul[..., 0]), vr.abs() + torch.sqrt(GAMMA * pr / Ur[..., 0]))
        F = 0.5 * (Fl + Fr) - 0.5 * a[..., None] * (Ur - Ul)
        S = torch.einsum("eqkm,qkj->emj", F * self.half[:, :, None, None], T["lift"])
        return (V - S) / self.det[:, None, None]

    def limit(self, c):
        """Barth-Jespersen limiting of a p = 1 state."""
        if not self.limiter:
            return c
        mean = math.sqrt(2.0) * c[..., 0]
        near = torch.where(self.inner[..., None], mean[self.nbr.clamp(min=0)], mean[:, None])
        hi = torch.maximum(mean, near.amax(1))
        lo = torch.minimum(mean, near.amin(1))
        d = torch.einsum("emj,qkj->emqk", c, self.T["tr"]).flatten(2) - mean[..., None]
        one = torch.ones_like(d)
        safe = torch.where(d == 0, one, d)
        a = torch.where(d > 0, (hi - mean)[..., None] / safe, torch.where(d < 0, (lo - mean)[..., None] / safe, one))
        a = torch.minimum(a, one).amin(-1, keepdim=True)
        return torch.cat([c[..., :1], a * c[..., 1:]], -1)

    def step(self, c, method):
        h, L, B = self.dt, self.rhs, self.limit
        if method == "ssp_rk3":
            u = B(c + h * L(c))
            u = B(0.75 * c + 0.25 * (u + h * L(u)))
            return B(c / 3 + 2.0 / 3.0 * (u + h * L(u)))
        if method == "rk2":
            u = B(c + h * L(c))
            return B(0.5 * c + 0.5 * (u + h * L(u)))
        k1 = L(c)
        k2 = L(B(c + 0.5 * h * k1))
        k3 = L(B(c + 0.5 * h * k2))
        k4 = L(B(c + h * k3))
        return B(c + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4))


def exact(case, seed):
    if _tables(case["p"], case["ne"], case["rule"]) is None:
        return None
    R = _Reference(case, seed)
    call = case["call"]
    if call == "adjoint":
        c = R.c0.clone().requires_grad_(True)
        return torch.autograd.grad(R.step(c, "ssp_rk3"), c, R.lam)[0]
    if call == "gradient":
        states = [R.c0]
        with torch.no_grad():
            for _ in range(case["steps"]):
                states.append(R.step(states[-1], "ssp_rk3"))
        lam = R.lam
        for c in reversed(states[:-1]):
            c = c.clone().requires_grad_(True)
            lam, = torch.autograd.grad(R.step(c, "ssp_rk3"), c, lam)
        return [states[-1], lam]
    with torch.no_grad():
        if call == "rhs":
            return R.rhs(R.c0)
        c = R.limit(R.c0)
        for _ in range(case["steps"]):
            c = R.step(c, case["method"])
        if call == "monitored":
            return [c, (c[..., 0] * R.det[:, None]).sum(0).div(math.sqrt(2.0)).cpu().numpy()]
        return c.cpu() if call == "host" else c
