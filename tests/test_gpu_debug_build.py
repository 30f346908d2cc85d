"""The index-checking build (libdg_debug.so, -DDG_DEBUG): every kernel checks each
connectivity index it reads before using it and records a bad one, which
dg_device_status reports as DG_EMESH (compute-sanitizer is not available, so this
build stands in for a memory checker).  A fresh process loads that build and runs
every kind of call -- all precisions, steppers, the limiter, boundary faces, the
adjoint and the no-allocation RHS, on both volume rules -- on meshes with ragged
last tiles, then
requires a clean device record and parity with the oracle.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r'''
import sys
import numpy as np
import torch
sys.path.insert(0, ROOT)
import oracle
from paper_1601_07944_gb300 import dg, inputs as I
lib = dg.load()
assert lib._name.endswith("libdg_debug.so"), lib._name

def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))

for mesh, ic in ((I.periodic_mesh(6), I.perturbed_vortex),
                 (I.box_mesh(6, x_code=I.BC_WALL, y_code=I.BC_STATE), I.steady_vortex)):
    for p, rule in ((1, "collapsed"), (3, "collapsed"), (5, "collapsed"), (2, "symmetric"), (5, "symmetric")):
        m = dg.Mesh.from_mesh(mesh, p, vol_rule=rule)
        o = oracle.OracleDG.from_mesh(mesh, p, vol_rule=rule)
        if m.n_boundary:
            xy = m.boundary_points().cpu().numpy()
            m.set_boundary_state(torch.from_numpy(ic(xy[..., 0], xy[..., 1])).cuda())
            oxy = o.boundary_points()
            o.set_boundary_state(ic(oxy[..., 0], oxy[..., 1]))
        c0 = o.project_ic(ic)
        c = torch.from_numpy(c0).cuda()
        assert rel(m.rhs(c).cpu().numpy(), o.rhs(c0)) < 1e-12
        r = torch.empty_like(c)
        m.rhs_noalloc(c, out=r)
        for prec in ("tf32x3", "tf32x1"):
            m.rhs(c, precision=prec)
        dt = I.fixed_dt(mesh, ic, p)
        for method in ("ssp_rk3", "rk2", "rk4"):
            x = c.clone()
            m.rk_step(x, dt, 18, method=method)
            assert rel(x.cpu().numpy(), getattr(o, method)(c0, dt, 18)) < 1e-12
            y = c.clone()
            m.rk_step(y, dt, 3, precision="tf32x3", method=method)
        m.adjoint_step(c, dt, torch.randn_like(c))
        if p == 1:
            m.set_limiter(True)
            z = c.clone()
            m.limit(z)
            m.rk_step(z, dt, 5)
            m.set_limiter(False)
        m.device_status()                 # raises on DG_EMESH (an index out of range)
print("debug build clean")
'''


def test_index_checking_build_runs_clean(oracle_mod):
    from paper_1601_07944_gb300 import _build
    lib = _build.build(debug=True)
    env = dict(os.environ, DG_LIB=lib)
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % ROOT + SCRIPT], env=env, cwd=ROOT,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and "debug build clean" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]


def test_index_checking_build_runs_clean_on_large_meshes(oracle_mod):
    """The same calls on 7,442 elements: the split-product kernels, their traces mode
    and the adjoint's, a ragged last tile, for two steps."""
    from paper_1601_07944_gb300 import _build
    lib = _build.build(debug=True)
    large = SCRIPT
    for small, big in (("periodic_mesh(6)", "periodic_mesh(61)"), ("box_mesh(6,", "box_mesh(61,"), ("dt, 18", "dt, 2")):
        assert small in large
        large = large.replace(small, big)
    env = dict(os.environ, DG_LIB=lib)
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % ROOT + large], env=env, cwd=ROOT,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and "debug build clean" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]


# Waits that expire, on a mesh of the split-product kernels (61 x 61 squares).
EXPIRE_SCRIPT = r'''
import os, sys
import numpy as np
import torch
sys.path.insert(0, ROOT)
from paper_1601_07944_gb300 import dg, inputs as I
lib = dg.load()
assert lib._name.endswith("libdg_debug.so"), lib._name
mesh = I.periodic_mesh(61)

# A completed wait of every tile group is reported as expired, the nth of each thread:
# DG_ETIMEOUT, and nothing of the kernel's last stores.  With one tile a group the
# right-hand side's element kernel has GEMM 1's wait and one for each batch of GEMM 2,
# the last of them before its stores; the adjoint's last kernel has one.
def expire(nth, p, call):
    os.environ["DG_DEBUG_EXPIRE"] = str(nth)
    m = dg.Mesh.from_mesh(mesh, p)
    del os.environ["DG_DEBUG_EXPIRE"]
    c = m.project_function(I.perturbed_vortex)
    out = torch.full_like(c, 7.0)
    call(m, c, out)
    try:
        m.device_status()
        expired = False
    except dg.DGError as e:
        assert dg.STATUS[e.status] == "DG_ETIMEOUT", e
        expired = True
    untouched = bool((out == 7.0).all())
    call(m, c, out)                       # the request ended with the status: a call as usual
    m.device_status()
    return expired, untouched, out.cpu().numpy(), m

for p in (1, 2, 3, 5):
    ref = None
    seen = []
    for nth in range(9):
        expired, untouched, got, m = expire(nth, p, lambda m, c, out: m.rhs(c, out=out))
        assert untouched == expired, (p, nth, expired, untouched)
        seen.append(expired)
        ref = got if ref is None else ref
        assert np.array_equal(got, ref)
    assert seen[0] and seen[1] and not seen[-1], seen
    if p <= 3:
        lam = torch.randn((m.N, 4, m.np), dtype=torch.float64, device="cuda")
        expired, untouched, _, _ = expire(0, p, lambda m, c, out: m.rhs_adjoint(c, lam, out=out))
        assert expired and untouched
print("debug build clean")
'''


def test_expired_waits_store_nothing():
    from paper_1601_07944_gb300 import _build
    lib = _build.build(debug=True)
    env = dict(os.environ, DG_LIB=lib)
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % ROOT + EXPIRE_SCRIPT], env=env, cwd=ROOT,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and "debug build clean" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
