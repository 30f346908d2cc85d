"""The split-product float64 element kernel (meshes too large for the fused
small-mesh stepper) against the oracle, at the sizes where its tiling can
go wrong: 7,442 elements leave 18 of 32 in the last tile, 8,192 none; every degree
covers its batches of points and of contraction columns, both volume rules, each
Runge-Kutta form of the update (one and two outputs), boundary faces, host-memory
traces and element ranges (the host-buffer step), and rows whose entries span
hundreds of orders of magnitude or are not finite.

Tolerances: a right-hand side is a difference of a volume and a surface term, so
||dR|| <= 1e-12 ||R|| + 16 eps ||V / det J|| with V the oracle's volume term; one
step adds dt R to a state of order one: 1e-14 relative, 45 eps.
"""
import numpy as np
import pytest

from paper_1601_07944_gb300 import inputs as I

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53
CASES = [(1, 0, "collapsed"), (1, 0, "symmetric"), (2, 0, "collapsed"), (3, 0, "collapsed"), (3, 3, "collapsed"), (4, 0, "collapsed"), (5, 0, "collapsed"),
         (2, 0, "symmetric"), (3, 0, "symmetric"), (3, 3, "symmetric"), (4, 0, "symmetric"), (5, 0, "symmetric")]


@pytest.fixture(scope="module")
def dgmod():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1601_07944_gb300 import _build, dg
    _build.build()
    dg.load()
    return dg


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _host(t):
    import torch
    torch.cuda.synchronize()
    return t.cpu().numpy()


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def check_rhs(m, o, c):
    ref, vol = o.rhs_and_volume(c)
    got = _host(m.rhs(_dev(c)))
    scale = np.linalg.norm(vol / o.det_j()[:, None, None])
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref) + 16 * EPS * scale
    return got


@pytest.mark.parametrize("n", [61, 64])
@pytest.mark.parametrize("p,ne,rule", CASES)
def test_rhs_and_steps(dgmod, oracle_mod, p, ne, rule, n):
    mesh = I.periodic_mesh(n)
    m = dgmod.Mesh.from_mesh(mesh, p, n_edge_pts=ne, vol_rule=rule)
    o = oracle_mod.OracleDG.from_mesh(mesh, p, n_edge_pts=ne, vol_rule=rule)
    c = o.project_ic(I.perturbed_vortex)
    check_rhs(m, o, c)
    dt = I.fixed_dt(mesh, I.perturbed_vortex, p)
    m.set_timing(True)
    for method, ref in (("ssp_rk3", o.ssp_rk3), ("rk4", o.rk4)):
        got = _host(m.rk_step(_dev(c), dt, 1, method=method))
        assert rel_l2(got, ref(c, dt, 1)) < 1e-14
    assert "stepper" not in m.kernel_times()       # the separate launches ran
    m.device_status()


@pytest.mark.parametrize("p", [2, 4])
def test_boundary_faces(dgmod, oracle_mod, p):
    mesh = I.box_mesh(61, I.BC_WALL, I.BC_STATE)
    m = dgmod.Mesh.from_mesh(mesh, p)
    o = oracle_mod.OracleDG.from_mesh(mesh, p)
    xy = o.boundary_points()
    ub = np.ascontiguousarray(I.steady_vortex(xy[..., 0], xy[..., 1]))
    o.set_boundary_state(ub)
    m.set_boundary_state(_dev(ub))
    check_rhs(m, o, o.project_ic(I.steady_vortex))


@pytest.mark.parametrize("p,rule", [(1, "collapsed"), (2, "collapsed"), (3, "collapsed"), (5, "collapsed"), (4, "symmetric")])
def test_host_state_and_repeats_same_bits(dgmod, p, rule):
    """The traces read from host memory, the ranges of the last stage and a second
    call after the state's own traces give the bits of plain one-step calls."""
    import torch
    mesh = I.periodic_mesh(107)          # 22,898 elements: several ranges of resident tiles
    m = dgmod.Mesh.from_mesh(mesh, p, vol_rule=rule)
    c = m.project_function(I.perturbed_vortex)
    dt = I.fixed_dt(mesh, I.perturbed_vortex, p)
    pinned = c.cpu().pin_memory()
    m.rk_step_host(pinned, dt, 2)
    a, b = c.clone(), c.clone()
    m.rk_step(a, dt, 2)
    for _ in range(2):
        m.rk_step(b, dt, 1)
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    assert torch.equal(a.cpu(), pinned)


@pytest.mark.parametrize("rule", ["collapsed", "symmetric"])
def test_limited_steps_same_bits(dgmod, oracle_mod, rule):
    """p = 1 with every stage limited: the traces that the limiter rewrites are those
    the next call forms, so two steps in one call and in two give the same bits."""
    import torch
    mesh = I.periodic_mesh(107)
    m = dgmod.Mesh.from_mesh(mesh, 1, vol_rule=rule)
    c = m.project_function(I.density_steps)
    dt = I.fixed_dt(mesh, I.density_steps, 1)
    m.set_limiter(True)
    m.limit(c)
    a, b = c.clone(), c.clone()
    m.rk_step(a, dt, 2, method="rk2")
    for _ in range(2):
        m.rk_step(b, dt, 1, method="rk2")
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    o = oracle_mod.OracleDG.from_mesh(mesh, 1, vol_rule=rule)
    o.set_limiter(True)
    assert rel_l2(_host(a), o.rk2(c.cpu().numpy(), dt, 2)) < 1e-14


def test_wide_range_rows(dgmod, oracle_mod):
    """Rows whose modes differ by up to 10^200, rows of zeros and rows below the
    smallest exponent the kernel keeps (2^-959): the error bound holds for the
    whole right-hand side."""
    mesh = I.periodic_mesh(61)
    p = 3
    m = dgmod.Mesh.from_mesh(mesh, p)
    o = oracle_mod.OracleDG.from_mesh(mesh, p)
    c = o.project_ic(I.perturbed_vortex)
    e = np.arange(mesh.n_elem)
    c[e % 7 == 1, :, 4:] *= 1e-200
    c[e % 7 == 2, 1] = 0.0
    c[e % 7 == 3, 2] *= 1e-300
    c[e % 7 == 4, :, 1:] *= 1e-12
    check_rhs(m, o, c)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf"), 1e300])
def test_non_finite_rows(dgmod, bad):
    """A coefficient that is not finite (or too large to square) is reported, and
    reaches its element and the neighbours only."""
    mesh = I.periodic_mesh(61)
    m = dgmod.Mesh.from_mesh(mesh, 2)
    c = m.project_function(I.perturbed_vortex)
    clean = _host(m.rhs(c))
    m.device_status()
    hit = 4321
    c[hit, 1, 2] = bad
    got = _host(m.rhs(c))
    with pytest.raises(dgmod.DGError) as err:
        m.device_status()
    assert dgmod.STATUS[err.value.status] == "DG_ENONPHYS"
    assert not np.isfinite(got[hit, 1:]).any()
    near = np.zeros(mesh.n_elem, bool)
    near[hit] = True
    near[mesh.nbr[hit]] = True
    assert np.array_equal(got[~near], clean[~near])


# The fixed-point edge flux against the oracle's float64 one: still fluid (momenta
# exactly zero), momenta far below the energies, supersonic flow, jumps inside and
# beyond the range it takes (a factor of 2^4 between the sides; the float64 form
# serves the rest), and units in which density and energy are far from one.
def _gas(rho_pm, p_pm, u, v, scale=1.0):
    def ic(x, y):
        s = np.sin(0.7 * x + 0.4 * y)
        b = np.sign(np.sin(2.1 * x) * np.cos(1.3 * y))
        return I.primitive_to_conserved(scale * np.exp(rho_pm * b + 0.1 * s), u * (1 + 0.1 * s) + 0.0 * x,
                                        v * (1 - 0.1 * s) + 0.0 * x, scale * np.exp(p_pm * b - 0.1 * s))
    return ic


@pytest.mark.parametrize("p", [1, 3])
@pytest.mark.parametrize("ic", [_gas(0, 0, 0, 0), _gas(0, 0, 1e-9, 2e-9), _gas(0.2, 0.1, 9.0, -4.0),
                                _gas(0.9, 0.9, 0.5, 0.2), _gas(3.0, 4.0, 0.1, 0.3), _gas(0.1, 0.1, 0.7, 0.3, 1e-60),
                                _gas(0.1, 0.1, 0.7, 0.3, 1e120), _gas(1.0, 0.1, 1e-180, 0.0)],
                         ids=["rest", "slow", "supersonic", "jumps", "strong_jumps", "tiny_units", "huge_units", "floor"])
def test_edge_flux_range(dgmod, oracle_mod, p, ic):
    mesh = I.periodic_mesh(61)
    m = dgmod.Mesh.from_mesh(mesh, p)
    o = oracle_mod.OracleDG.from_mesh(mesh, p)
    cen = mesh.elem_xy.mean(axis=1)
    c = np.zeros((mesh.n_elem, 4, m.np))
    c[:, :, 0] = ic(cen[:, 0], cen[:, 1]) / np.sqrt(2.0)          # constant in each element: jumps at every face
    c[:, :, 1] = 1e-3 * c[:, :, 0]
    ref, vol = o.rhs_and_volume(c)
    got = _host(m.rhs(_dev(c)))
    det = o.det_j()[:, None, None]
    # the scale of each variable by itself: the edge terms of a piecewise constant
    # state are as large as h alpha U / det J, which the residual itself shows
    for k in range(4):
        scale = np.linalg.norm((vol / det)[:, k]) + np.linalg.norm(ref[:, k])
        wave = np.linalg.norm(c[:, k] / np.sqrt(det[:, 0])) * 10.0 * max(1.0, np.sqrt(np.max(np.abs(c[:, 3] / c[:, :1, 0][:, 0:1]))))
        assert np.linalg.norm(got[:, k] - ref[:, k]) <= 1e-12 * scale + 16 * EPS * (scale + wave)
    m.device_status()


# The adjoint's kernels of the same meshes (p <= 3) against the oracle's reverse
# sweep: 1e-12 relative, as for the float64 kernels they replace, on states with the
# small noise of the other adjoint tests: on the unperturbed stream (1, 1) the normal
# velocity vanishes on the mesh's diagonals, and the derivative of its magnitude there
# is the sign of a rounding error.
@pytest.mark.parametrize("n", [61, 64])
@pytest.mark.parametrize("p,ne,rule", [c for c in CASES if c[0] <= 3])
def test_adjoint(dgmod, oracle_mod, p, ne, rule, n):
    mesh = I.periodic_mesh(n)
    m = dgmod.Mesh.from_mesh(mesh, p, n_edge_pts=ne, vol_rule=rule)
    o = oracle_mod.OracleDG.from_mesh(mesh, p, n_edge_pts=ne, vol_rule=rule)
    rng = np.random.default_rng(7)
    c = o.project_ic(I.perturbed_vortex) + 0.002 * rng.standard_normal((o.N, 4, o.np))
    lam = rng.standard_normal(c.shape)
    assert rel_l2(_host(m.rhs_adjoint(_dev(c), _dev(lam))), o.rhs_vjp(c, lam)) < 1e-12
    dt = I.fixed_dt(mesh, I.perturbed_vortex, p)
    assert rel_l2(_host(m.adjoint_step(_dev(c), dt, _dev(lam))), o.ssp_rk3_vjp(c, dt, lam)) < 1e-12
    m.device_status()


def test_adjoint_boundary_and_stages(dgmod, oracle_mod):
    mesh = I.box_mesh(61, I.BC_WALL, I.BC_STATE)
    m = dgmod.Mesh.from_mesh(mesh, 2)
    o = oracle_mod.OracleDG.from_mesh(mesh, 2)
    xy = o.boundary_points()
    ub = np.ascontiguousarray(I.steady_vortex(xy[..., 0], xy[..., 1]))
    o.set_boundary_state(ub)
    m.set_boundary_state(_dev(ub))
    rng = np.random.default_rng(8)
    c = o.project_ic(I.steady_vortex) + 0.002 * rng.standard_normal((o.N, 4, o.np))
    lam = rng.standard_normal(c.shape)
    dt = I.fixed_dt(mesh, I.steady_vortex, 2)
    got = _host(m.adjoint_step(_dev(c), dt, _dev(lam)))
    assert rel_l2(got, o.ssp_rk3_vjp(c, dt, lam)) < 1e-12
    import torch
    d = _dev(c)
    u1, u2 = torch.empty_like(d), torch.empty_like(d)
    m.rk_step_stages(d, dt, u1, u2)
    assert np.array_equal(got, _host(m.adjoint_step_stages(_dev(c), u1, u2, dt, _dev(lam))))


@pytest.mark.parametrize("n", [8, 61])
@pytest.mark.parametrize("precision", ["fp64", "tf32x3"])
def test_non_physical_boundary_state(dgmod, precision, n):
    """A prescribed state without pressure meets only the edge flux, which reports it
    whatever the ratio of its kinetic energy to its energy."""
    mesh = I.box_mesh(n, I.BC_STATE, I.BC_STATE)
    m = dgmod.Mesh.from_mesh(mesh, 2)
    c = m.project_function(lambda x, y: I.primitive_to_conserved(1 + 0 * x, 0.1 + 0 * x, 0.2 + 0 * x, 1 + 0 * x))
    u = np.zeros((m.n_boundary, m.ne, 4))
    u[..., 0] = u[..., 3] = 1.0
    for mom in (1.3, 1.5, 2.0, 4.5, 5.0, 5.5, 5.8, 7.5, 7.9, 8.5, 20.0):
        u[..., 1], u[..., 2] = 0.6 * mom, 0.8 * mom
        m.set_boundary_state(_dev(u))
        m.rhs(c, precision=precision)
        if mom < 2.0 ** 0.5:
            m.device_status()
            continue
        with pytest.raises(dgmod.DGError) as err:
            m.device_status()
        assert dgmod.STATUS[err.value.status] == "DG_ENONPHYS"


# Rows far from one.  The Euler fluxes are homogeneous, so that gas at rest may have any
# unit of density and energy (moving gas may not: the square of a momentum leaves the
# range), and the adjoint is linear in its cotangent.  In units of 2^-950 the fluxes of
# mass, jumps of 1e-10, lie below the 2^-959 that the kernel takes its smallest rows
# relative to: an error of 2^-1017, 2^-67 of the state, 2^-49 of a residual (sums of up
# to 90, divided by det J of 2^-5 or more).
@pytest.mark.parametrize("k", [-950, -900, 960, 990])
@pytest.mark.parametrize("p,ne,rule", [(1, 0, "collapsed"), (2, 0, "symmetric"), (3, 0, "collapsed"), (4, 0, "collapsed"), (5, 0, "collapsed")])
def test_rows_far_from_one(dgmod, oracle_mod, p, ne, rule, k):
    mesh = I.periodic_mesh(61)
    m = dgmod.Mesh.from_mesh(mesh, p, n_edge_pts=ne, vol_rule=rule)
    o = oracle_mod.OracleDG.from_mesh(mesh, p, n_edge_pts=ne, vol_rule=rule)
    c = o.project_ic(_gas(0.1, 0.1, 0, 0))
    ref, vol = o.rhs_and_volume(c)
    scale = np.linalg.norm(vol / o.det_j()[:, None, None])
    unit = 2.0 ** k
    got = _host(m.rhs(_dev(c * unit))) / unit
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref) + 16 * EPS * scale
    # a step so short that the kinetic energy (which underflows) is below a rounding;
    # in large units any motion's would overflow: a step of length zero
    for method in ("ssp_rk3", "rk4"):
        got = _host(m.rk_step(_dev(c * unit), 1e-9 if k < 0 else 0.0, 1, method=method)) / unit
        if k < 0:
            assert rel_l2(got - c, 1e-9 * ref) < 1e-4
        else:
            assert rel_l2(got, c) < 1e-14
    m.device_status()
    if p <= 3:
        rng = np.random.default_rng(7)
        u = o.project_ic(I.perturbed_vortex) + 0.002 * rng.standard_normal((o.N, 4, o.np))
        lam = rng.standard_normal(u.shape)
        assert rel_l2(_host(m.rhs_adjoint(_dev(u), _dev(lam * unit))) / unit, o.rhs_vjp(u, lam)) < 1e-12


@pytest.mark.parametrize("p,rule", [(3, "collapsed"), (4, "collapsed"), (4, "symmetric"), (5, "collapsed"), (5, "symmetric")])
def test_rows_lined_up_with_a_table(dgmod, oracle_mod, p, rule):
    """Momentum rows that are a column of the interpolation or the trace table (a delta at
    one of its points): their digits are the table's, so that the products of one level
    all have one sign for that point."""
    mesh = I.periodic_mesh(61)
    m = dgmod.Mesh.from_mesh(mesh, p, vol_rule=rule)
    o = oracle_mod.OracleDG.from_mesh(mesh, p, vol_rule=rule)
    c = o.project_ic(_gas(0.1, 0.1, 0, 0))
    phi = dgmod.volume_rule(p, rule)[3]
    face = dgmod.host_tables(p)["phi_face"].reshape(-1, phi.shape[1])
    cols = np.concatenate([phi, face])
    for k in (1, 2):
        c[:, k] = 1e-3 * (-1.0) ** k * cols[(np.arange(mesh.n_elem) * k) % len(cols)]
    check_rhs(m, o, c)
    m.device_status()
