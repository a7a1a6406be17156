"""States at the limits of the FP64 steps in 64-bit fixed point: frames without a
temperature, rates and equilibria outside the fixed-point range, non-finite
populations, slow relaxation.  What the arithmetic there cannot hold is either
computed in FP64 or counted."""
import numpy as np
import pytest

from tests.cases import rel_linf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rl():
    from paper_1909_04502_gb300 import rlbm
    return rlbm


def _frame2(g, p):
    """(n, eps) of the frame of the populations g."""
    N, T = g @ p, np.einsum("i,ia,ib->ab", g, p, p)
    w, v = np.linalg.eig(T * np.array([1.0, -1.0, -1.0]))
    assert np.abs(np.imag(w)).max() == 0
    for k in range(3):
        x = v[:, k].real
        nn = x[0] ** 2 - x[1] ** 2 - x[2] ** 2
        if nn > 1e-3:
            U = x * np.sign(x[0]) / np.sqrt(nn)
            return N @ (U * np.array([1.0, -1.0, -1.0])), w[k].real
    raise AssertionError("no timelike eigenvector")


def _states_without_temperature(p, m):
    """eps/n = r m from a rest population 1 and -s in all on the highest shell, each
    population changed by up to 1 %."""
    p0, top = p[:, 0], p[:, 0].max()
    shell = p0 > top - 1e-9
    out = []
    for r in (0.1, 0.3, 0.5, 0.7):
        s = m * m * (1 - r) / (top * top - r * m * top)
        g = np.where(p0 < m + 1e-9, 1.0, np.where(shell, -s / shell.sum(), 0.0))
        g = g * (1 + 0.01 * np.random.default_rng(len(out)).random(len(p0)))
        n, eps = _frame2(g, p)
        assert n > 0 and 0 < eps < 0.8 * m * n
        out.append(g)
    return out


@pytest.mark.parametrize("order", [2, 3])
def test_frames_without_a_temperature_are_counted(rl, order):
    """m > 0: below eps/n = (2 sqrt 2 - 2) m the equation of state has no real T.
    Uniform states (streaming moves nothing), positive at rest and negative on a
    shell of higher energy, with n, eps > 0 and eps/n up to 0.8 m: every cell is
    counted and left bitwise unrelaxed."""
    m, nx, ny = 5.0, 33, 6
    lat = rl.Lattice(nx, ny, m=m, order=order, tau=0.9, precision="fp64")
    states = _states_without_temperature(lat.p, m)
    for g in states:
        G = np.ascontiguousarray(np.broadcast_to(g[:, None, None], (lat.Q, ny, nx)))
        lat.set_populations(G)
        lat.step(1)
        assert lat.sync_status(raise_on_error=False) == (-4, nx * ny)
        assert np.array_equal(lat.populations(), G)
    lat.close()
