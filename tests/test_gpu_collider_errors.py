"""A collider run that ends in an error leaves the scene as it was: when the cause is gone, the
next run carries every contact's history over, as if the failed one had not been."""
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


def _far(w, pos):       # one sphere's neighbours see it more than 511 cells away
    bad = pos.copy()
    bad[len(pos) // 2] += 600 * np.diag(w.cell)
    return bad


def _one_place(w, pos):   # every pair overlaps: more than 2^31 candidates
    return np.zeros_like(pos) + pos[:1]


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("n,spoil,word", [(3000, _far, "shift"), (65600, _one_place, "pairs")])
def test_histories_survive_a_failed_run(pkg, n, spoil, word, mixed):
    w = workloads.periodic_cloud(n, 47, phi=0.34, inflate=1.05, vel_scale=0.2, angvel_scale=20.0)
    out = []
    for fail in (False, True):
        s = pkg.Scene.from_workload(w, precision=pkg.DEM_MIXED if mixed else pkg.DEM_FP64)
        s.step(20)
        st = s.state(force=False)
        pos, vel = st["pos"], st["vel"]
        pos += 40 * s.dt() * vel           # a new order of slots at the next run
        if fail:
            s.set_state(pos=spoil(w, pos))
            for _ in range(2):
                with pytest.raises(pkg.DemError) as e:
                    s.step(1)
                assert e.value.code == 4 and word in str(e.value)
            assert np.array_equal(s.state(force=False)["vel"], vel)   # by id, in the old order
        s.set_state(pos=pos)
        s.step(1)
        c, a = s.contacts(), s.state()
        out.append([c[k] for k in ("id1", "id2", "c", "fn", "fs")] + [a[k] for k in a])
        s.close()
    assert np.abs(out[0][4]).max() > 0 and len(out[0][0]) > n / 10
    assert all(np.array_equal(x, y) for x, y in zip(*out))
