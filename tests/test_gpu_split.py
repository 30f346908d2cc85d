"""The split-product float64 element kernel (meshes too large for the fused
small-mesh stepper, p >= 2) against the oracle, at the sizes where its tiling can
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
CASES = [(2, 0, "collapsed"), (3, 0, "collapsed"), (3, 3, "collapsed"), (4, 0, "collapsed"), (5, 0, "collapsed"),
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


@pytest.mark.parametrize("p,rule", [(2, "collapsed"), (3, "collapsed"), (5, "collapsed"), (4, "symmetric")])
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
