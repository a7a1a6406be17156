"""The FP64 steps with their population sums in 64-bit fixed point against the
oracle where the scaling has work to do: densities far from one, temperatures
and speeds whose populations are far from the reference's (negative ones among
them), and grids of one warp and a tail.  The bar is the FP64 parity bar,
1e-12 of the largest value: both sides round a few hundred times per step at
2^-53, amplified by the equilibrium's condition number (below 2^10 on these
states)."""
import numpy as np
import pytest

from oracle import d3 as OD
from tests.cases import rel_linf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rl():
    from paper_1909_04502_gb300 import rlbm
    return rlbm


def _state3(nx, ny, nz, n0, T0, u0, seed):
    rng = np.random.default_rng(seed)
    z, y, x = np.meshgrid(*(2 * np.pi * np.arange(k) / k for k in (nz, ny, nx)), indexing="ij")
    p = rng.uniform(0, 2 * np.pi, 5)
    n = n0 * (1 + 0.3 * np.cos(x + p[0]) * np.cos(y + p[1]))
    T = T0 * (1 + 0.2 * np.sin(y + z + p[2]))
    return n, u0 * np.cos(y + p[3]), 0.1 * u0 * np.sin(x + z + p[4]), -0.3 * u0 * np.cos(x), T


@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("n0,T0,u0", [(1.0, 1.0, 0.0), (1e-150, 1.0, 0.2), (3e120, 0.7, 0.3), (1.0, 1.6, 0.2),
                                      (2.0, 0.5, 0.5), (1.0, 1.0, 0.7)])
def test_fixed_point_step3_matches_oracle(rl, order, n0, T0, u0):
    nx, ny, nz = 33, 7, 6
    fields = [np.ascontiguousarray(a) for a in _state3(nx, ny, nz, n0, T0, u0, order)]
    quad = OD.massless_quadrature_3d(order)
    sim = OD.Simulation3(quad, OD.Expansion3(quad, order), nx, ny, nz, tau=0.8)
    lat = rl.Lattice3(nx, ny, nz, tau=0.8, precision="fp64", order=order)
    pos = {(tuple(v), round(p, 9)): i for i, (v, p) in enumerate(zip(lat.n.tolist(), lat.p[:, 0]))}
    idx = [pos[(tuple(v), round(p, 9))] for v, p in zip(quad.n.tolist(), quad.p[:, 0])]
    lat.init(*fields)
    sim.init(*fields)
    lat.step(2)
    sim.step(2)
    assert lat.sync_status() == (0, 0)
    assert rel_linf(lat.populations()[idx], sim.fs) <= 1e-12
    mo = lat.moments()
    for name, want in (("n", sim.fields.n), ("T", sim.fields.T), ("eps", sim.fields.eps)):
        assert rel_linf(mo[name], want) <= 1e-12
    speed = max(np.abs(sim.fields.u(k)).max() for k in (1, 2, 3))
    for k, name in ((1, "ux"), (2, "uy"), (3, "uz")):
        assert np.abs(mo[name] - sim.fields.u(k)).max() <= 1e-12 * max(speed, 1e-3)
    lat.close()


@pytest.mark.parametrize("order", [2, 3])
def test_fields_of_fp32_storage_match_fp64_sums(rl, order):
    """The fields sum the stored 32-bit deviations and the reference exactly: they
    equal the oracle's on the same populations to FP64 rounding."""
    nx, ny, nz = 35, 6, 7
    lat = rl.Lattice3(nx, ny, nz, tau=0.9, precision="fp32", order=order)
    lat.init(*[np.ascontiguousarray(a) for a in _state3(nx, ny, nz, 1.2, 0.9, 0.3, 7)])
    lat.step(2)
    quad = OD.massless_quadrature_3d(order)
    pos = {(tuple(v), round(p, 9)): i for i, (v, p) in enumerate(zip(lat.n.tolist(), lat.p[:, 0]))}
    idx = [pos[(tuple(v), round(p, 9))] for v, p in zip(quad.n.tolist(), quad.p[:, 0])]
    before = lat.populations()[idx]
    lat.step(1)
    want = OD.macroscopic3(OD.stream3(before, quad.n), quad)
    mo = lat.moments()
    for name, w in (("n", want.n), ("T", want.T), ("eps", want.eps)):
        assert rel_linf(mo[name], w) <= 1e-13
    for k, name in ((1, "ux"), (2, "uy"), (3, "uz")):
        assert np.abs(mo[name] - want.u(k)).max() <= 1e-14
    lat.close()
