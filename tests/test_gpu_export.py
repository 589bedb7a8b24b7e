"""State and contact export: packed on the device, small results through pinned staging, larger
ones copied array by array.  Both routes and every subset of arrays must give the same rows."""
import ctypes

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


def _scene(pkg, n, mixed, walls):
    mk = workloads.box_cloud if walls else workloads.periodic_cloud
    w = mk(n, 71, phi=0.33 if not walls else 0.3, inflate=1.05, vel_scale=0.05, angvel_scale=10.0)
    s = pkg.Scene.from_workload(w, precision=pkg.DEM_MIXED if mixed else pkg.DEM_FP64)
    s.step(3)
    return s


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("n", [60, 2520, 2521, 6000])
def test_ranges_and_subsets_match_the_whole(pkg, n, mixed, walls):
    s = _scene(pkg, max(n, 300) if not walls else n, mixed, walls)
    n = s.n
    st = s.state()
    for first, m in ((0, n), (n // 3, 17), (n - 1, 1)):
        part = s.state_range(first, m)
        for k in ("pos", "vel", "angvel", "ori"):
            assert np.array_equal(part[k], st[k][first:first + m])
    only = np.empty((n, 3))
    for k in ("vel", "angvel", "pos", "torque", "force"):
        s.get_state_into(**{k: only})
        assert np.array_equal(only, st[k])
    # contacts: the forces of the rows add up to the body forces; prefixes agree
    c = s.contacts()
    m = len(c["id1"])
    assert m == s.count_contacts() and m > 20
    key = c["id1"].astype(np.int64) * (n + 8) + c["id2"]
    assert np.all(np.diff(key) > 0)
    F = np.zeros((n, 3))
    f = c["fn"] + c["fs"]
    np.add.at(F, c["id2"], f)
    ball = c["id1"] >= 0
    np.add.at(F, c["id1"][ball], -f[ball])
    assert np.abs(F - st["force"]).max() <= 1e-5 * np.abs(f).max()
    if walls:
        assert (~ball).any()
    names = ("id1", "id2", "c", "fn", "fs", "normal", "cpoint", "phys", "pen")
    for cap in (0, 1, min(m, 1700)):
        out = {k: np.empty_like(c[k][:cap]) for k in names}
        cnt = ctypes.c_longlong()
        ptr = [out[k].ctypes.data if k != "normal" else None for k in names]   # one array left out
        assert s._lib.dem_get_contacts(s._h, cap, ctypes.byref(cnt), *ptr) == 0
        assert cnt.value == m
        for k in names:
            if k != "normal":
                assert np.array_equal(out[k], c[k][:cap])
    s.close()
