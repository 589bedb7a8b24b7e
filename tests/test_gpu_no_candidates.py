"""Scenes whose collider runs find no candidate pair: a single sphere, spheres out of each
other's range, and a scene emptied by a removal.  The contact table then has no rows (its row
arrays may not exist), and every step, query and export must work all the same."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

R, GAP, V, DT = 0.01, 0.06, 1.0, 1e-5


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2301_00611_gb300 as pkg
    return pkg


def _scene(pkg, n, periodic, mixed, **kw):
    """n spheres (1 or 2) on a line, 2 R + GAP apart, approaching at V each."""
    kind = dict(periodic=True, cell=np.eye(3) * 0.3) if periodic else \
        dict(box_hi=(0.3, 0.3, 0.3), wall_mask=0x3F)
    s = pkg.Scene(precision=pkg.DEM_MIXED if mixed else pkg.DEM_FP64, damping=0.0, **kind, **kw)
    s.set_material(0, 2600.0, 1e7, 0.3, 0.5)
    x = 0.15 + (R + GAP / 2) * np.array([-1.0, 1.0])
    pos = np.column_stack([x, np.full(2, 0.15), np.full(2, 0.15)])[:n]
    vel = np.array([[V, 0, 0], [-V, 0, 0]])[:n]
    s.add_spheres(pos, np.full(n, R), vel=vel)
    s.set_dt(DT)
    return s, pos, vel


def _check_free(s, pos, vel, t):
    st = s.state()
    assert np.abs(st["pos"] - (pos + t * vel)).max() <= 1e-12      # 3000 sums of 1e-5, rounded
    assert np.array_equal(st["vel"], vel) and not st["force"].any() and not st["torque"].any()
    stats = s.stats()
    assert stats["n_contacts"] == stats["n_candidates"] == stats["n_wall_contacts"] == 0
    assert stats["kinetic_energy"] > 0 and not stats["stress"].any()
    assert s.count_contacts() == 0 and len(s.contacts()["id1"]) == 0


@pytest.mark.parametrize("graphs", [0, 1])
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("periodic", [False, True])
def test_single_sphere(pkg, periodic, mixed, graphs):
    s, pos, vel = _scene(pkg, 1, periodic, mixed)
    s.set_tuning(step_graphs=graphs)
    s.step(1)
    _check_free(s, pos, vel, DT)
    s.step(1500)                                  # several collider runs
    _check_free(s, pos, vel, 1501 * DT)
    assert s.stats()["n_rebuilds"] > 1
    s.close()


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("periodic", [False, True])
def test_spheres_that_meet_later(pkg, periodic, mixed):
    s, pos, vel = _scene(pkg, 2, periodic, mixed)
    s.step(100)
    _check_free(s, pos, vel, 100 * DT)
    touch = int(GAP / 2 / V / DT)
    s.step(touch + 30 - 100)                      # a contact lasts about 73 steps
    assert s.count_contacts() == 1 and s.contacts()["pen"][0] > 0
    s.step(170)
    v = s.state()["vel"]
    assert s.count_contacts() == 0
    assert np.abs(v + vel).max() <= 0.05 * V      # restitution 1 up to the step's share of a contact
    s.step(2000)                                  # out of range again
    assert s.stats()["n_candidates"] == 0
    s.close()


@pytest.mark.parametrize("mixed", [False, True])
def test_time_stepper_without_contacts(pkg, mixed):
    s, pos, vel = _scene(pkg, 1, True, mixed)
    s.set_timestepper(safety=0.5, interval=1, default_dt=2 * DT)
    s.step(10)
    assert s.dt() == 2 * DT
    s.close()


@pytest.mark.parametrize("mixed", [False, True])
def test_served_single_sphere(pkg, mixed):
    w = workloads.scaled_deposition(60, 5, 0.5, 1e7, steps=0)
    w.pos, w.radius, w.mat_id = w.pos[:1], w.radius[:1], w.mat_id[:1]
    w.vel = w.angvel = None
    with pkg.Server(precision=pkg.DEM_MIXED if mixed else pkg.DEM_FP64) as srv:
        t = srv.submit(w, 50, keep_state=True, dt=1e-5)
        srv.wait(t)
        z = srv.result(t, state=True)["state"]["pos"][0, 2]
        srv.release(t)
    fall = 0.5 * np.linalg.norm(w.gravity) * (50 * 1e-5) ** 2
    assert 0.5 * fall < w.pos[0, 2] - z < 1.1 * fall


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("stepper", [False, True])
def test_scene_emptied_by_a_removal(pkg, stepper, mixed):
    """The step after the removal of the last bodies runs on none; the scene then takes new
    ones, which advance as in a scene of their own."""
    a = workloads.box_cloud(300, 61, phi=0.3, inflate=1.04, vel_scale=0.05)
    b = workloads.scaled_deposition(200, 62, 0.4, 1e7, steps=0)
    prec = pkg.DEM_MIXED if mixed else pkg.DEM_FP64
    s, alone = pkg.Scene(precision=prec), pkg.Scene(precision=prec)
    for k in (s, alone):
        k.set_dt(1e-5)
        if stepper:
            k.set_timestepper(safety=0.5, interval=1, default_dt=2e-5)
    q = s.add_workload(a, 0, dt=1e-5)
    s.step(3)
    s.remove_subscene(q)
    s.step(1)
    assert s.n == 0 and s.count_contacts() == 0 and s.stats()["n_bodies"] == 0
    assert s.clock()[0] == 4 and s.stats()["dt"] == (2e-5 if stepper else 1e-5)
    s.step(5)
    assert s.clock()[0] == 9
    for k in (s, alone):
        k.add_workload(b, 8, dt=1e-5)
        k.step(20)
    x, y = s.state(force=False), alone.state(force=False)
    assert all(np.array_equal(x[k], y[k]) for k in x)
    s.close()
    alone.close()
