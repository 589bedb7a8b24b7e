"""dem_find_pairs and its form without allocation at the limits of their inputs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2301_00611_gb300 as pkg
    return torch, pkg


@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("row", [(np.inf, 0, 0, 1), (0, np.nan, 0, 1), (0, 0, -np.inf, 1), (0, 0, 0, 0.0),
                                 (0, 0, 0, -1), (0, 0, 0, np.nan), (0, 0, 0, -np.nan), (0, 0, 0, np.inf),
                                 (1e308, 1e308, 0, 1), (-1e308, 0, -1e308, 1), (0, 0, 1e308, 1e308),
                                 (6e307, 6e307, 6e307, 1)])
def test_refused_inputs(env, row, noalloc):
    """Not finite, not positive, or a sum x + y + z + r beyond the range of a double."""
    torch, pkg = env
    a = np.ones((40, 4))
    a[:, 0] = 3 * np.arange(40)
    a[17] = row
    P, R = (torch.tensor(np.ascontiguousarray(x), device="cuda") for x in (a[:, :3], a[:, 3]))
    with pytest.raises(pkg.DemError) as e:
        pkg.find_pairs(P, R, noalloc=noalloc)
    assert e.value.code == 5 and "non-finite" in str(e.value)
