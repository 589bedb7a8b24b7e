"""Contacts exported through the spare part of the collider's list buffer (a scene with room for
many more bodies than it has) and through memory of their own must be the same records."""
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


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("n", [1000, 1023, 6001])
def test_both_buffers_give_the_same_records(pkg, n, walls, mixed):
    mk = workloads.box_cloud if walls else workloads.periodic_cloud
    w = mk(n, 73, phi=0.33 if not walls else 0.3, inflate=1.05, vel_scale=0.05, angvel_scale=10.0)
    out = []
    for capacity in (0, 64 * n):
        s = pkg.Scene.from_workload(w, precision=pkg.DEM_MIXED if mixed else pkg.DEM_FP64,
                                    capacity_bodies=capacity)
        s.step(3)
        out.append(s.contacts())
        before = s.state(force=False)
        s.step(2)                       # the lists are scratch: the scene goes on as before
        out[-1]["pos"] = s.state(force=False)["pos"]
        assert not np.array_equal(before["pos"], out[-1]["pos"])
        s.close()
    m = len(out[0]["id1"])
    # at least 148 m bytes: more than the 56 a body that the tight scene has to spare, less than the
    # other has
    assert 148 * m < 56 * 64 * n and (n != 6001 or 148 * m > 56 * 6001)
    assert all(np.array_equal(out[0][k], out[1][k]) for k in out[0])
