"""The contact shapes the autotuner tries are different launches: per-SM block counts up to
what an SM holds (larger settings launch that many), so its choice is one of those, and any
setting gives the same trajectory."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

TRIED = {False: {128: {2, 3, 5, 6}, 256: {1, 2}}, True: {128: {2, 4, 6, 8}, 256: {2, 4}}}


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2301_00611_gb300 as pkg
    return pkg


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("n", [3000, 120000])
def test_autotuner_chooses_a_launch_of_its_own(pkg, n, mixed):
    w = workloads.periodic_cloud(n, 43, phi=0.3, inflate=1.05, vel_scale=0.05)
    kw = dict(precision=pkg.DEM_MIXED if mixed else pkg.DEM_FP64)
    a = pkg.Scene.from_workload(w, **kw)
    chosen = a.autotune(steps_per_trial=1)
    assert chosen["contact_blocks_per_sm"] in TRIED[mixed][chosen["contact_block"]]
    n = a.clock()[0]
    want = a.state()
    a.close()
    for per_sm in (1, 64):
        b = pkg.Scene.from_workload(w, **kw)
        b.set_tuning(contact_blocks_per_sm=per_sm)
        assert b.tuning()["contact_blocks_per_sm"] == per_sm
        b.step(n)
        got = b.state()
        assert all(np.array_equal(got[k], want[k]) for k in ("pos", "vel", "angvel", "ori"))
        b.close()
