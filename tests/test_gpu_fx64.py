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
from tests.cases import oracle_quadrature, oracle_sim, permutation, rel_linf

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


def _state2(nx, ny, n0, T0, u0, seed):
    rng = np.random.default_rng(seed)
    y, x = np.meshgrid(*(2 * np.pi * np.arange(k) / k for k in (ny, nx)), indexing="ij")
    p = rng.uniform(0, 2 * np.pi, 4)
    n = n0 * (1 + 0.3 * np.cos(x + p[0]))
    T = T0 * (1 + 0.1 * np.sin(y + p[1]))
    return [np.ascontiguousarray(a) for a in (n, u0 * np.cos(y + p[2]), 0.5 * u0 * np.sin(x + p[3]), T)]


@pytest.mark.parametrize("m,order,nx,ny,n0,T0,u0", [
    (0.0, 2, 33, 5, 1.0, 1.0, 0.0), (0.0, 2, 200, 1, 1e-150, 1.3, 0.3), (0.0, 3, 3, 70, 2e100, 0.8, 0.4),
    (0.0, 3, 65, 9, 1.0, 1.0, 0.6), (1.0, 2, 34, 6, 1.0, 1.1, 0.2), (5.0, 3, 33, 5, 1e8, 1.0, 0.2),
    (10.0, 2, 31, 9, 1.0, 1.0, 0.1)])
@pytest.mark.parametrize("stream", ["onlattice", "bilinear"])
def test_fixed_point_step2_matches_oracle(rl, m, order, nx, ny, n0, T0, u0, stream):
    lam = 1.0 if stream == "bilinear" else 0.0
    lat = rl.Lattice(nx, ny, m=m, order=order, tau=0.8, precision="fp64", stream=stream, lam=lam)
    quad = oracle_quadrature(m, order, lat.n, rl.plan(m=m, order=order)["v0"])
    sim = oracle_sim(quad, nx, ny, tau=0.8, stream=stream, lam=lam or None)
    fields = _state2(nx, ny, n0, T0, u0, order)
    lat.init(*fields)
    sim.init(*fields)
    lat.step(2)
    sim.step(2)
    assert lat.sync_status() == (0, 0)
    idx = permutation(lat.n, lat.p, quad)
    assert rel_linf(lat.populations()[idx], sim.fs) <= 1e-12
    mo = lat.moments(full=True)
    assert rel_linf(mo["n"], sim.fields.n) <= 1e-12 and rel_linf(mo["T"], sim.fields.T) <= 1e-12
    assert rel_linf(mo["N"], sim.fields.N) <= 1e-12
    lat.close()


@pytest.mark.parametrize("m,order", [(0.0, 2), (5.0, 3)])
def test_cells_without_a_frame_are_counted_and_streamed(rl, m, order):
    """A cell of negative density and one with an infinite population: both
    counted, their finite populations streamed unrelaxed, an infinity turned NaN."""
    nx, ny = 40, 11
    lat = rl.Lattice(nx, ny, m=m, order=order, tau=0.9, precision="fp64")
    lat.init(*_state2(nx, ny, 1.0, 1.0, 0.1, 3))
    f = lat.populations()
    f[:] = f[:, :1, :1]                            # uniform, so that streaming moves nothing
    f[:, :, :] *= -1.0
    lat.set_populations(f)
    lat.step(1)
    rc, count = lat.sync_status(raise_on_error=False)
    assert rc == -4 and count == nx * ny
    assert np.array_equal(lat.populations(), f)
    f *= -1.0
    f[3] = np.inf                                  # every cell pulls it
    lat.set_populations(f)
    lat.step(1)
    rc, count = lat.sync_status(raise_on_error=False)
    got = lat.populations()
    assert rc == -4 and count == nx * ny
    assert np.isnan(got[3]).all() and np.array_equal(np.delete(got, 3, 0), np.delete(f, 3, 0))
    lat.close()


@pytest.mark.parametrize("order", [2, 3, 5])
@pytest.mark.parametrize("nx,n0,T0,u0,boundary", [(1, 1.0, 1.0, 0.0, "periodic"), (129, 1e-140, 1.0, 0.3, "periodic"),
                                                  (257, 1e90, 0.6, 0.6, "freeflow_x"), (40, 1.0, 1.5, 0.2, "eqwall_x")])
def test_fixed_point_step1_matches_oracle(rl, order, nx, n0, T0, u0, boundary):
    """The (1+1)-d step: f and the fields against the oracle.  At order 5 the
    equilibrium's condition number reaches 2^13 off the reference temperature,
    in the oracle's FP64 sums as in the step: 1e-11 there."""
    from oracle import d1 as O1
    x = 2 * np.pi * np.arange(nx) / nx
    fields = [np.ascontiguousarray(a) for a in (n0 * (1 + 0.2 * np.sin(x)), u0 * np.cos(x + 0.4) + 0 * x,
                                                T0 * (1 + 0.1 * np.cos(x)))]
    lat = rl.Lattice1(nx, order=order, tau=0.8, boundary=boundary, precision="fp64")
    sim = O1.Simulation1(O1.massless_quadrature_1d(order), nx, tau=0.8, boundary=boundary)
    lat.init(*fields)
    sim.init(*fields)
    lat.step(2)
    sim.step(2)
    assert lat.sync_status() == (0, 0)
    tol = 1e-12 if order < 5 else 1e-11
    q = sim.quad
    pos = {(int(s), round(float(p), 9)): i for i, (s, p) in enumerate(zip(lat.n, lat.p[:, 0]))}
    idx = [pos[(int(s), round(float(p), 9))] for s, p in zip(q.n, q.p[:, 0])]
    assert rel_linf(lat.populations()[idx], sim.fs) <= tol
    mo = lat.moments()
    assert rel_linf(mo["n"], sim.fields.n) <= tol and rel_linf(mo["T"], sim.fields.T) <= tol
    assert rel_linf(mo["eps"], sim.fields.eps) <= tol
    lat.close()
