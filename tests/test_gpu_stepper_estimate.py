"""The time stepper's FP32 estimates only choose which bodies are computed in FP64, so the step
must be the same bits as with every body in FP64 (an unused material with ks > kn turns
the estimates off), for both laws and precisions, in walled boxes and periodic cells, and
for sub-scenes of very different stiffness."""
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


@pytest.mark.parametrize("law", [0, 1])
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("kind", ["periodic", "box"])
@pytest.mark.parametrize("n", [40, 2500])
def test_estimated_and_full_steps_agree(pkg, law, mixed, kind, n):
    if kind == "periodic":
        w = workloads.periodic_cloud(max(n, 300), 51, phi=0.34, inflate=1.05, vel_scale=0.05)
    else:
        w = workloads.box_cloud(n, 52, phi=0.3, inflate=1.04, vel_scale=0.05)
    dts = []
    for full in (False, True):
        s = pkg.Scene.from_workload(w, precision=pkg.DEM_MIXED if mixed else pkg.DEM_FP64)
        if full:
            s.set_material(7, 2600.0, 5e7, 2.0, 0.5)
        s.set_law(law)
        s.set_timestepper(safety=0.7, interval=1)
        out = []
        for _ in range(20):
            s.step(1)
            out.append(s.dt())
        dts.append((out, s.state(force=False)["vel"]))
        s.close()
    assert len(set(dts[0][0])) > 5          # the step does change
    assert dts[0][0] == dts[1][0]
    assert np.array_equal(dts[0][1], dts[1][1])


def test_subscenes_keep_their_own_minimum(pkg):
    ws = [workloads.scaled_deposition(n, 60 + n, 0.5, E, steps=0) for n, E in ((60, 1e6), (900, 1e8), (33, 1e7))]
    got = []
    for full in (False, True):
        s = pkg.Scene()
        subs = [s.add_workload(w, k, dt=1e-5) for k, w in enumerate(ws)]
        if full:
            s.set_material(99, 2600.0, 5e7, 2.0, 0.5)
        for q in subs:
            s.set_timestepper(safety=0.5, interval=2, sub=q)
        s.step(300)
        got.append([s.subscene(q)["dt"] for q in subs])
        s.close()
    assert got[0] == got[1] and len(set(got[0])) == 3
