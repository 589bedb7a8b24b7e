"""Sweep margins and gradings that give most bodies more partners than a list of 32, some more
than the 512 that are ranked on chip, in scenes that take a warp per body and in larger ones:
the contacts must be the pairs of the configuration on the first run (which sizes the spill
buffer) and on later ones (which may choose another pass), and in FP64 a trajectory must not
depend on the margin at all."""
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


def _cloud(n, periodic, giants=0, size=1.0):
    """n spheres of equal size, many overlapping, `giants` of them `size` times larger."""
    r = 0.42 * n ** (-1 / 3)
    rad = np.full(n, r)
    rad[7:7 + 11 * giants:11] *= size
    w = workloads.periodic_cloud(64, 1, phi=0.1) if periodic else workloads.box_cloud(64, 1, phi=0.1)
    w.pos, w.radius, w.mat_id = workloads.uniform(3 * n, 23).reshape(n, 3), rad, np.zeros(n, np.int32)
    w.vel = workloads.uniform(3 * n, 29).reshape(n, 3) - 0.5
    w.angvel = None
    w.cell, w.box_lo, w.box_hi, w.wall_mask = np.eye(3), np.zeros(3), np.ones(3), 0
    w.gravity = np.zeros(3)
    return w


def _want(env, w):
    torch, pkg = env
    I, J, C = pkg.find_pairs(torch.tensor(w.pos, device="cuda"), torch.tensor(w.radius, device="cuda"),
                             periodic=w.periodic, cell=w.cell)
    want = np.column_stack([I.cpu().numpy(), J.cpu().numpy(), C.cpu().numpy()])
    return want[np.lexsort((want[:, 1], want[:, 0]))]


@pytest.mark.parametrize("n,periodic,giants,size,margin", [
    (3000, True, 0, 1, 1.0), (3000, False, 0, 1, 2.0), (70000, True, 0, 1, 1.0),
    (70000, True, 0, 1, 2.0), (70000, False, 40, 4, 1.25),
    (3000, False, 2, 12, 0.5), (70000, True, 3, 12, 0.5)])
def test_contacts_are_the_pairs_on_every_run(env, n, periodic, giants, size, margin):
    torch, pkg = env
    w = _cloud(n, periodic, giants, size)
    want = _want(env, w)
    s = pkg.Scene.from_workload(w, dt=1e-12, verlet_dist=margin * w.radius.min())
    for run in range(3):
        if run:
            s.set_state(pos=w.pos)          # another collider run, same positions
        s.step(1)
        c = s.contacts()
        assert np.array_equal(np.column_stack([c["id1"], c["id2"], c["c"]]), want)
    st = s.stats()
    assert st["n_rebuilds"] == 3 and 2 * st["n_candidates"] > (16 if margin >= 1 else 8) * n
    s.close()


@pytest.mark.parametrize("n", [3000, 70000])
def test_trajectory_does_not_depend_on_the_margin(env, n):
    torch, pkg = env
    w = _cloud(n, True, 20, 2.5)
    out = []
    for margin in (0.5, 1.25, 2.0):
        s = pkg.Scene.from_workload(w, dt=1e-7, verlet_dist=margin * w.radius.min())
        s.step(4)
        s.set_state(pos=s.state(force=False)["pos"])
        s.step(4)
        c = s.contacts()
        out.append([s.state()[k] for k in ("pos", "vel", "angvel", "force")] + [c[k] for k in ("id1", "id2", "c", "fs", "fn")])
        s.close()
    for other in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(out[0], other))


@pytest.mark.parametrize("n", [65537, 92683])
def test_more_candidate_pairs_than_a_table_can_hold(env, n):
    """Every pair within the margin: n (n - 1) / 2 is just above 2^31 and just above 2^32, where
    a 32-bit sum comes out negative and small.  Both are an error, not a table."""
    torch, pkg = env
    s = pkg.Scene(box_hi=(1, 1, 1), verlet_dist=10.0)
    s.set_material(0, 2600.0, 1e7, 0.3, 0.5)
    s.add_spheres(workloads.uniform(3 * n, 31).reshape(n, 3), np.full(n, 1e-6))
    s.set_dt(1e-9)
    with pytest.raises(pkg.DemError) as e:
        s.step(1)
    assert e.value.code == 4 and "pairs" in str(e.value)
    s.close()
