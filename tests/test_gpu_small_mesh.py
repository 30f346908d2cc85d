"""The fused small-mesh stepper (dg_set_small_mesh_stepper): on a mesh whose
element tiles fit in one wave of the GPU, a float64 Runge-Kutta call runs every
stage in one cooperative launch, the edge, element and (with the limiter on)
limiter phases separated by a barrier over the grid.  It runs the same code as
the separate launches, so the states agree bit for bit; every small-mesh parity
test of the suite (against the oracle) goes through it by default."""
import numpy as np
import pytest

from paper_1601_07944_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dgmod():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1601_07944_gb300 import _build, dg
    _build.build()
    dg.load()
    return dg


def _host(t):
    import torch
    torch.cuda.synchronize()
    return t.cpu().numpy()


def _run(m, c0, dt, steps, method, fused):
    """The state after `steps` steps in one call, and the kernel kinds one more
    call launches (per-kernel timing is on for that call only: it turns the CUDA
    graphs of the separate-launch path off)."""
    m.set_small_mesh_stepper(fused)
    c = c0.clone()
    m.rk_step(c, dt, steps, method=method)
    out = _host(c)
    m.set_timing(True)
    m.rk_step(c, dt, 2, method=method)
    kt = m.kernel_times()
    m.set_timing(False)
    m.device_status()
    return out, kt


@pytest.mark.parametrize("method", ["ssp_rk3", "rk2", "rk4"])
@pytest.mark.parametrize("p,ne,n", [(1, 0, 10), (2, 0, 8), (3, 0, 8), (3, 3, 7), (4, 0, 6), (5, 0, 5)])
def test_fused_equals_separate_launches(dgmod, p, ne, n, method):
    """Ragged last tiles (50 to 200 elements); 20 steps (a 16-step graph replay
    and plain steps on the separate-launch side)."""
    mesh = I.periodic_mesh(n)
    m = dgmod.Mesh.from_mesh(mesh, p, n_edge_pts=ne)
    c0 = m.project_function(I.perturbed_vortex)
    dt = I.fixed_dt(mesh, I.perturbed_vortex, p)
    a, kta = _run(m, c0, dt, 20, method, True)
    b, ktb = _run(m, c0, dt, 20, method, False)
    assert "stepper" in kta and kta["stepper"][0] == 1 and "element" not in kta
    assert "stepper" not in ktb and "element" in ktb
    assert np.array_equal(a, b)


@pytest.mark.parametrize("rule", ["collapsed", "symmetric"])
def test_fused_with_boundary_faces(dgmod, rule):
    """A closed box of walls and a channel with prescribed states on its sides."""
    import torch
    for mesh in (I.box_mesh(10), I.box_mesh(10, x_code=I.BC_STATE, y_code=I.BC_STATE)):
        m = dgmod.Mesh.from_mesh(mesh, 2, vol_rule=rule)
        if m.n_boundary:
            xy = m.boundary_points().cpu().numpy()
            m.set_boundary_state(torch.from_numpy(np.ascontiguousarray(I.steady_vortex(xy[..., 0], xy[..., 1]))).cuda())
        c0 = m.project_function(I.steady_vortex)
        dt = I.fixed_dt(mesh, I.steady_vortex, 2)
        a, kta = _run(m, c0, dt, 12, "ssp_rk3", True)
        b, _ = _run(m, c0, dt, 12, "ssp_rk3", False)
        assert "stepper" in kta
        assert np.array_equal(a, b)


@pytest.mark.parametrize("method", ["ssp_rk3", "rk2", "rk4"])
@pytest.mark.parametrize("n", [10, 16])
def test_fused_with_limiter(dgmod, n, method):
    """p = 1 with every stage limited (density steps: the limiter acts on most
    elements); 200 and 512 elements, ragged last tiles; no limiter launch on the
    fused side."""
    mesh = I.periodic_mesh(n)
    m = dgmod.Mesh.from_mesh(mesh, 1)
    c0 = m.limit(m.project_function(I.density_steps))
    dt = I.fixed_dt(mesh, I.density_steps, 1)
    m.set_limiter(True)
    a, kta = _run(m, c0, dt, 20, method, True)
    b, ktb = _run(m, c0, dt, 20, method, False)
    m.set_limiter(False)
    assert "stepper" in kta and "other" not in kta and "element" not in kta
    assert "stepper" not in ktb and "other" in ktb
    assert np.array_equal(a, b)
    try:
        free, _ = _run(m, c0, dt, 20, method, True)
        assert not np.array_equal(free, a)        # limiting changed the run
    except dgmod.DGError as e:
        assert dgmod.STATUS[e.status] == "DG_ENONPHYS"   # or, without it, the run broke down


@pytest.mark.parametrize("method", ["ssp_rk3", "rk4"])
@pytest.mark.parametrize("p,ne,rule,n", [(1, 0, "collapsed", 41), (1, 0, "symmetric", 41), (1, 0, "collapsed", 55),
                                         (1, 0, "symmetric", 55), (2, 0, "collapsed", 41), (2, 0, "symmetric", 41),
                                         (3, 0, "collapsed", 41), (3, 3, "collapsed", 41), (3, 0, "symmetric", 41),
                                         (4, 0, "collapsed", 41), (4, 0, "symmetric", 41), (5, 0, "collapsed", 41)])
def test_fused_equals_separate_launches_8_element_tiles(dgmod, p, ne, rule, n, method):
    """The stepper's second variant (meshes beyond 4 elements in each of 4 blocks per
    SM), with a ragged last tile; at p = 1 up to 6,080 elements (five blocks per SM)."""
    import torch
    mesh = I.periodic_mesh(n)
    m = dgmod.Mesh.from_mesh(mesh, p, n_edge_pts=ne, vol_rule=rule)
    assert m.N > 16 * torch.cuda.get_device_properties(0).multi_processor_count and m.N % 8 == 2
    c0 = m.project_function(I.perturbed_vortex)
    dt = I.fixed_dt(mesh, I.perturbed_vortex, p)
    a, kta = _run(m, c0, dt, 5, method, True)
    b, ktb = _run(m, c0, dt, 5, method, False)
    assert "stepper" in kta and "element" not in kta
    assert "stepper" not in ktb and "element" in ktb
    assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [41, 55])
def test_fused_with_limiter_8_element_tiles(dgmod, n):
    mesh = I.periodic_mesh(n)
    m = dgmod.Mesh.from_mesh(mesh, 1)
    c0 = m.limit(m.project_function(I.density_steps))
    dt = I.fixed_dt(mesh, I.density_steps, 1)
    m.set_limiter(True)
    a, kta = _run(m, c0, dt, 5, "rk2", True)
    b, ktb = _run(m, c0, dt, 5, "rk2", False)
    assert "stepper" in kta and "element" not in kta and "stepper" not in ktb
    assert np.array_equal(a, b)


def test_fused_matches_oracle(dgmod, oracle_mod):
    """The fused path against the oracle's SSP-RK3 run (relative L2 <= 1e-12)."""
    mesh = I.periodic_mesh(12)
    p = 3
    m = dgmod.Mesh.from_mesh(mesh, p)
    o = oracle_mod.OracleDG.from_mesh(mesh, p)
    dt = I.fixed_dt(mesh, I.perturbed_vortex, p)
    c = m.project_function(I.perturbed_vortex)
    m.set_timing(True)
    m.rk_step(c, dt, 25)
    assert "stepper" in m.kernel_times()
    m.set_timing(False)
    ref = o.ssp_rk3(o.project_ic(I.perturbed_vortex), dt, 25)
    got = _host(c)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 1e-12


def test_large_mesh_keeps_separate_launches(dgmod):
    """The fused stepper's tiles hold 4 or 8 elements, at most 4 blocks per SM;
    9,800 elements at p = 3 need 1,225 blocks of 8, more than one wave on 152 SMs:
    the separate launches run."""
    import torch
    mesh = I.periodic_mesh(70)
    m = dgmod.Mesh.from_mesh(mesh, 3)
    props = torch.cuda.get_device_properties(0)
    assert (m.N + 7) // 8 > 4 * props.multi_processor_count
    c = m.project_function(I.vortex)
    m.set_timing(True)
    m.rk_step(c, I.fixed_dt(mesh, I.vortex, 3), 2)
    kt = m.kernel_times()
    m.set_timing(False)
    assert "stepper" not in kt and kt["element"][0] == 6


THREADS = r'''
import sys, threading
import torch
sys.path.insert(0, ROOT)
from paper_1601_07944_gb300 import dg, inputs as I
dg.load()
mesh = I.periodic_mesh(12)
torch.zeros(1, device="cuda")
go = threading.Barrier(8)
made = [None] * 8

def make(i):
    torch.cuda.set_device(0)
    go.wait()
    made[i] = dg.Mesh.from_mesh(mesh, 2)

threads = [threading.Thread(target=make, args=(i,)) for i in range(8)]
for t in threads:
    t.start()
for t in threads:
    t.join()
first = None
for m in made:
    states = []
    for fused in (True, False):
        m.set_small_mesh_stepper(fused)
        c = m.project_function(I.vortex)
        m.set_timing(True)
        m.rk_step(c, 1e-3, 3)
        assert ("stepper" in m.kernel_times()) == fused
        m.set_timing(False)
        states.append(c)
    first = states[0] if first is None else first
    assert all(torch.equal(s, first) for s in states)
print("threads agree")
'''


def test_meshes_created_by_threads_at_once():
    """Whether a mesh fits the stepper is asked once per process, at the first mesh; eight
    threads create theirs at once, and every one keeps the stepper and its bits."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % root + THREADS], cwd=root, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and "threads agree" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
