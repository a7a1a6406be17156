"""make_params: a stencil given by its groups and a force do not mix."""
import numpy as np
import pytest

from tests.cases import generators


@pytest.fixture(scope="module")
def rl():
    from paper_1909_04502_gb300 import build, rlbm
    build.build()
    return rlbm


@pytest.mark.parametrize("groups", [[(0, 0), (1, 0), (2, 1)], [(2, 1), (1, 0), (0, 0)], None])
@pytest.mark.parametrize("g", [(1e-3, -2e-3), (0.0, 0.0)])
def test_force_and_groups(rl, groups, g):
    p, _keep = rl.make_params(8, 8, m=5.0, groups=groups, g=g)
    assert (p.gx, p.gy) == g
    assert p.n_groups == (len(groups) if groups else 0)
    if groups:
        assert [p.groups[i] for i in range(2 * len(groups))] == [c for v in groups for c in v]


@pytest.mark.gpu
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
def test_forced_run_on_explicit_groups(rl, precision, tol):
    """The built-in stencil and the same one given by its groups, whose solved
    weights agree to rounding: the same forced flow at the parity bars."""
    nx, ny, m, g = 40, 24, 5.0, (2e-3, 5e-3)
    d = rl.plan(m=m)
    rng = np.random.default_rng(1)
    one = np.ones((ny, nx))
    fields = [one + 0.1 * rng.random((ny, nx)), 0 * one, 0 * one, one]
    out = []
    for kw in (dict(), dict(groups=generators(d["n"]), v0=d["v0"])):
        lat = rl.Lattice(nx, ny, m=m, tau=0.9, precision=precision, g=g, boundary="eqwall_x", **kw)
        lat.init(*fields)
        lat.step(10)
        out.append(lat.moments())
        lat.close()
    for k in ("n", "ux", "uy", "T"):
        assert np.abs(out[0][k] - out[1][k]).max() <= tol
    assert out[0]["uy"].mean() > 1e-3
