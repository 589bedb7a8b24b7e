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


def _query(env, n, cap, noalloc=False):
    """n spheres in one place, so every two are a pair: (error code, count, I, J, C)."""
    import ctypes
    torch, pkg = env
    lib = pkg.load_library()
    P = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    R = torch.full((n,), 1e-3, dtype=torch.float64, device="cuda")
    I, J = (torch.full((cap + 8,), -7, dtype=torch.int32, device="cuda") for _ in range(2))
    C = torch.full((cap + 8, 3), -7, dtype=torch.int32, device="cuda")
    cnt = ctypes.c_longlong(-1)
    fn = lib.dem_find_pairs_noalloc if noalloc else lib.dem_find_pairs
    ptr = [x.data_ptr() if cap else None for x in (I, J, C)]
    rc = fn(P.data_ptr(), R.data_ptr(), n, 0, np.eye(3).ctypes.data, 0.0, cap, *ptr, ctypes.byref(cnt),
            torch.cuda.current_stream().cuda_stream)
    return rc, cnt.value, I.cpu().numpy(), J.cpu().numpy(), C.cpu().numpy()


@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("n", [65536, 65537])
@pytest.mark.parametrize("cap", [0, 1000])
def test_pair_counts_around_a_signed_sum(env, n, cap, noalloc):
    """n (n - 1) / 2 is 2^31 - 2^15 and 2^31 + 2^15: counted exactly, rows within the capacity."""
    if noalloc and n > 65536:
        pytest.skip("more spheres than the fixed scratch holds")
    rc, count, I, J, C = _query(env, n, cap, noalloc)
    assert rc == 0 and count == n * (n - 1) // 2
    assert np.all(I[:cap] >= 0) and np.all(I[:cap] < J[:cap]) and np.all(J[:cap] < n) and not C[:cap].any()
    assert len(set(zip(I[:cap].tolist(), J[:cap].tolist()))) == cap
    assert np.all(I[cap:] == -7) and np.all(J[cap:] == -7) and np.all(C[cap:] == -7)


def test_more_pairs_than_can_be_counted(env):
    rc, count, I, J, C = _query(env, 92683, 16)       # n (n - 1) / 2 just above 2^32
    assert rc == 4 and count == 0
    assert np.all(I[16:] == -7) and np.all(J[16:] == -7)
