"""dem_find_pairs where the warp-per-cell walk can go wrong: fewer spheres than lanes, a
single cell, cells with more bodies than lanes, spheres with more pairs than a list
keeps, lattice spacings exactly at the threshold (decided in FP64), and sizes whose
squares leave FP32's range.  The pairs must be the oracle's brute-force set."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import oracle
    import paper_2301_00611_gb300 as pkg
    return torch, oracle, pkg


def _check(env, pos, rad, periodic=False, H=None, margin=0.0):
    torch, oracle, pkg = env
    P = torch.tensor(pos, dtype=torch.float64, device="cuda")
    R = torch.tensor(rad, dtype=torch.float64, device="cuda")
    I, J, C = (x.cpu().numpy() for x in pkg.find_pairs(P, R, periodic=periodic, cell=H, margin=margin))
    oi, oj, oc = oracle.pairs(pos, rad, periodic=periodic, H=H, margin=margin, method="brute")
    got = sorted(zip(I.tolist(), J.tolist(), map(tuple, C.tolist())))
    want = sorted(zip(oi.tolist(), oj.tolist(), map(tuple, np.asarray(oc).tolist())))
    assert got == want
    return len(got)


@pytest.mark.parametrize("n", [2, 31, 32, 33, 257])
@pytest.mark.parametrize("scale", [1.0, 1e-3])
def test_few_spheres(env, n, scale):
    u = workloads.uniform(4 * n, 5 + n).reshape(n, 4)
    _check(env, u[:, :3] * scale * n ** (1 / 3), (0.3 + 0.4 * u[:, 3]) * scale)


def test_crowded_cells_and_long_lists(env):
    """Large spheres among many small ones: cells of hundreds of bodies, hundreds of pairs each."""
    n = 3000
    u = workloads.uniform(3 * n, 11).reshape(n, 3)
    rad = np.full(n, 0.012)
    rad[:12] = 0.11
    assert _check(env, u, rad) > 400
    assert _check(env, u, rad, periodic=True, H=np.eye(3), margin=1e-3) > 400


@pytest.mark.parametrize("periodic", [False, True])
def test_lattice_at_the_threshold(env, periodic):
    """A cubic lattice of spacing exactly 2 r (no pair: the test is strict), with every
    third sphere moved by one ulp or by 1e-9 of the spacing either way."""
    m, a = 8, 0.25
    g = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3) * a
    rad = np.full(len(g), a / 2)
    H = np.eye(3) * m * a
    assert _check(env, g, rad, periodic=periodic, H=H) == 0
    p = g.copy()
    p[::3, 0] = np.nextafter(p[::3, 0], 10.0)
    p[1::3, 1] -= a * 1e-9
    assert _check(env, p, rad, periodic=periodic, H=H) > 100


@pytest.mark.parametrize("scale", [1e-14, 1e12])
def test_sizes_near_the_ends_of_fp32(env, scale):
    w = workloads.periodic_cloud(400, 9, phi=0.33, inflate=1.05)
    assert _check(env, w.pos * scale, w.radius * scale, periodic=True, H=w.cell * scale) > 100
