"""The collider where its partner lists can go wrong: spheres with more partners than a list
holds, in scenes small enough for a warp per body and large enough for a thread per body.
The contacts of a step must be the pairs dem_find_pairs gives for the same configuration
(its set is checked against brute force elsewhere), with their cell shifts, and a collider
run between two steps must carry every contact's history over unchanged."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2301_00611_gb300 as pkg
    return torch, pkg


def _scene(pkg, w, **kw):
    s = pkg.Scene.from_workload(w, dt=1e-9, **kw)
    return s


def _cloud(n, periodic):
    """n small spheres, some overlapping, and 24 large ones that touch dozens of them."""
    r = 0.42 * n ** (-1 / 3)
    rad = np.full(n, r)
    rad[5:5 + 24 * 7:7] = 3.5 * r
    L = 1.0
    pos = workloads.uniform(3 * n, 17).reshape(n, 3) * L
    w = workloads.periodic_cloud(64, 1, phi=0.1) if periodic else workloads.box_cloud(64, 1, phi=0.1)
    w.pos, w.radius, w.mat_id = pos, rad, np.zeros(n, dtype=np.int32)
    w.vel = (workloads.uniform(3 * n, 19).reshape(n, 3) - 0.5)
    w.angvel = None
    w.cell, w.box_lo, w.box_hi, w.wall_mask = np.eye(3) * L, np.zeros(3), np.full(3, L), 0
    w.gravity = np.zeros(3)
    return w


@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("n", [3000, 70000])
def test_contacts_of_long_lists_are_the_pairs(env, n, periodic):
    torch, pkg = env
    w = _cloud(n, periodic)
    s = _scene(pkg, w, verlet_dist=0.5 * w.radius.min())
    s.step(1)
    c = s.contacts()
    got = np.column_stack([c["id1"], c["id2"], c["c"]])
    I, J, C = pkg.find_pairs(torch.tensor(w.pos, device="cuda"), torch.tensor(w.radius, device="cuda"),
                             periodic=periodic, cell=w.cell)
    want = np.column_stack([I.cpu().numpy(), J.cpu().numpy(), C.cpu().numpy()])
    want = want[np.lexsort((want[:, 1], want[:, 0]))]
    deg = np.bincount(np.concatenate([want[:, 0], want[:, 1]]), minlength=n)
    assert len(want) > n / 2 and deg.max() > 20      # candidates of that sphere: well beyond 32
    assert np.array_equal(got, want)
    s.close()


@pytest.mark.parametrize("mixed", [False, True])
def test_collider_run_carries_every_history(env, mixed):
    torch, pkg = env
    w = _cloud(3000, True)
    prec = pkg.DEM_MIXED if mixed else pkg.DEM_FP64
    a, b = (_scene(pkg, w, precision=prec, verlet_dist=0.5 * w.radius.min()) for _ in range(2))
    for s in (a, b):
        s.step(3)
    b.set_state(pos=b.state(force=False)["pos"])     # forces a collider run, same positions
    for s in (a, b):
        s.step(1)
    ca, cb = a.contacts(), b.contacts()
    assert np.array_equal(ca["id1"], cb["id1"]) and np.array_equal(ca["id2"], cb["id2"])
    assert a.stats()["n_rebuilds"] == 1 and b.stats()["n_rebuilds"] == 2
    scale = np.linalg.norm(ca["fs"], axis=1).max()
    if mixed:   # the reference positions moved: FP32 increments differ in their last bits
        assert np.abs(ca["fs"] - cb["fs"]).max() <= 1e-5 * scale
    else:
        assert np.array_equal(ca["fs"], cb["fs"]) and np.array_equal(ca["fn"], cb["fn"])
    for s in (a, b):
        s.close()


@pytest.mark.parametrize("mixed", [False, True])
def test_integrated_force_is_the_sum_over_all_rows(env, mixed):
    """Undamped, without gravity, a step changes a velocity by dt F / m: the integrator's sum
    over a body's real rows (masks of 32 rows; some bodies have more) against the query's sum
    over all of them."""
    torch, pkg = env
    w = _cloud(3000, True)
    w.damping = 0.0
    s = _scene(pkg, w, precision=pkg.DEM_MIXED if mixed else pkg.DEM_FP64,
               verlet_dist=0.5 * w.radius.min())
    for _ in range(3):
        v0 = s.state(force=False)["vel"]
        s.step(1)
        st = s.state()
        m = w.materials[0].density * 4 / 3 * np.pi * w.radius ** 3
        dv = 1e-9 * st["force"] / m[:, None]
        # the velocity's own rounding, and in mixed precision the FP32 rounding of dt F / m
        bound = 4e-16 * np.abs(st["vel"]) + (1e-6 if mixed else 1e-14) * np.abs(dv).max()
        assert np.abs(dv).max() > 1e-6
        assert np.all(np.abs(st["vel"] - v0 - dv) <= bound)
    s.close()
