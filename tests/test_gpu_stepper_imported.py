"""The time stepper on contacts whose stiffnesses the caller set (dem_set_contacts): shear
stiffer than normal by orders of magnitude, and negative values that cancel in a body's sums,
where FP32 estimates would choose the wrong bodies.  The step must be the one with every body
in FP64 (an unused material with a Poisson's ratio above 1 turns the estimates off)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2301_00611_gb300 as pkg
    return pkg


def _steps(pkg, make, full, steps):
    s = make()
    if full:
        s.set_material(7, 2600.0, 5e7, 2.0, 0.5)
    s.set_timestepper(safety=0.7, interval=1)
    out = []
    for _ in range(steps):
        s.step(1)
        out.append(s.dt())
    s.close()
    return out


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("ratio", [1.0, 1e4])
def test_shear_stiffer_than_normal(pkg, mixed, ratio):
    w = workloads.periodic_cloud(1500, 57, phi=0.34, inflate=1.05, vel_scale=0.05)
    prec = pkg.DEM_MIXED if mixed else pkg.DEM_FP64
    a = pkg.Scene.from_workload(w, precision=prec, dt=1e-8)
    a.step(2)
    c = a.contacts()
    a.close()
    assert len(c["id1"]) > 300
    phys = c["phys"].copy()
    phys[:, 1] = phys[:, 0] * ratio * (0.5 + workloads.uniform(len(phys), 3))

    def make():
        s = pkg.Scene.from_workload(w, precision=prec, dt=1e-8)
        s.set_contacts(c["id1"], c["id2"], c["c"], c["fs"], c["normal"], phys)
        return s
    got, want = (_steps(pkg, make, full, 5) for full in (False, True))
    assert got == want


@pytest.mark.parametrize("mixed", [False, True])
def test_negative_stiffnesses_that_cancel(pkg, mixed):
    """A closed row of spheres along a periodic cell: each has two contacts on its axis, whose
    shear stiffnesses have opposite signs and cancel to 2 or 3 units of FP32's last place.
    Truncated to FP32, the stiffest body (2.99 units) looks softer than two others."""
    n, r = 12, 1e-2
    a = 1.98 * r
    pos = np.column_stack([(np.arange(n) + 0.5) * a, np.full(n, 0.1), np.full(n, 0.1)])
    left = np.arange(n)                                     # contact k: spheres k and k + 1
    id1 = np.where(left == n - 1, 0, left)
    id2 = np.where(left == n - 1, n - 1, left + 1)
    shift = np.zeros((n, 3), np.int32)
    shift[n - 1, 0] = -1
    units = np.tile([9.99, 7.0, 9.5, 7.9, 10.0, 7.5], n // 6)
    ks = (1.0 - 2.0 * (left % 2)) * (2.0 ** 17 + 2.0 ** -6 * units)
    phys = np.column_stack([np.full(n, 1e-9), ks, np.full(n, 0.5)])
    normal = np.zeros((n, 3))
    normal[:, 0] = np.where(left == n - 1, -1.0, 1.0)
    order = np.lexsort((id2, id1))

    def make():
        s = pkg.Scene(periodic=True, cell=np.diag([n * a, 0.2, 0.2]),
                      precision=pkg.DEM_MIXED if mixed else pkg.DEM_FP64)
        s.set_material(0, 2600.0, 1e7, 0.3, 0.5)
        s.add_spheres(pos, np.full(n, r))
        s.set_dt(1e-8)
        s.set_contacts(id1[order], id2[order], shift[order], np.zeros((n, 3)), normal[order], phys[order])
        return s
    got, want = (_steps(pkg, make, full, 1) for full in (False, True))
    assert got == want and got[0] > 0.1
