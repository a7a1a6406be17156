"""A cell of a (3+1)-d FP32 run whose density no frame can hold (the conversions
of the frame take finite values only) is counted, and the cells that it cannot
have reached yet are bitwise those of the run without it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rl():
    from paper_1909_04502_gb300 import rlbm
    return rlbm


@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("n", [1e12, 1e30, np.inf, np.nan])
def test_cell_without_frame_is_counted_and_stays_apart(rl, order, n):
    nx, ny, nz = 40, 17, 18
    rng = np.random.default_rng(order)
    fields = [1 + 0.1 * rng.random((nz, ny, nx))] + [0.05 * rng.random((nz, ny, nx)) for _ in range(3)]
    fields.append(1 + 0.1 * rng.random((nz, ny, nx)))
    got = []
    for bad in (False, True):
        f = [a.copy() for a in fields]
        if bad:
            f[0][9, 8, 20] = n
        lat = rl.Lattice3(nx, ny, nz, tau=0.9, precision="fp32", order=order)
        lat.init(*f)
        lat.step(1)
        got.append((lat.populations(), lat.sync_status()[1]))
        lat.close()
    reach = 8 if order == 3 else 3
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    far = np.maximum(np.maximum(abs(z - 9), abs(y - 8)), abs(x - 20)) > reach
    assert far.any()
    assert got[0][1] == 0 and got[1][1] > 0
    assert np.array_equal(got[0][0][:, far], got[1][0][:, far])
