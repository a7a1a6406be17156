"""Fast flows.  The Landau frame of a flow of Lorentz factor g is what remains of a
tensor g^2 times as large, so that a relative rounding e of T^ab changes eps by
about g^4 e and u by g^2 e; with populations of both signs e is 2^-53 (the stored
values being given) times k = sum |f| p0^2 / T^00.  The bars are 16 times
that, for the oracle's rounding and the library's together."""
import numpy as np
import pytest

from oracle import d3 as OD
from oracle import lattice as OL
from oracle import scheme as OS
from tests.cases import oracle_quadrature, permutation, rel_linf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rl():
    from paper_1909_04502_gb300 import rlbm
    return rlbm


def _order3(lat, quad):
    pos = {(tuple(v), round(p, 9)): i for i, (v, p) in enumerate(zip(lat.n.tolist(), lat.p[:, 0]))}
    return [pos[(tuple(v), round(p, 9))] for v, p in zip(quad.n.tolist(), quad.p[:, 0])]


def _bar(f, quad, u):
    p2 = (quad.p[:, 0] ** 2).reshape((-1,) + (1,) * (f.ndim - 1))
    k = float(((np.abs(f) * p2).sum(0) / (f * p2).sum(0)).max())
    return 16 * k * 2.0 ** -53 / (1 - u * u) ** 2


def _check_fields3(mo, want, bar, u):
    assert np.isfinite(mo["n"]).all()
    for name, w in (("n", want.n), ("T", want.T), ("eps", want.eps)):
        assert np.abs(mo[name] / w - 1).max() <= bar
    for k, name in ((1, "ux"), (2, "uy"), (3, "uz")):
        assert np.abs(mo[name] - want.u(k)).max() <= bar * (1 - u * u)


@pytest.mark.parametrize("order,precision,speeds", [
    (2, "fp64", (0.9, 0.95, 0.99, 0.993, 0.995, 0.999, 0.9995)), (3, "fp64", (0.9, 0.95, 0.99, 0.995, 0.999, 0.9995)),
    (2, "fp32", (0.9, 0.99, 0.995, 0.999)), (3, "fp32", (0.9, 0.99, 0.993))])
def test_fields3_of_fast_cells(rl, order, precision, speeds):
    """Cells of one speed and random directions: the fields of the stored populations."""
    quad = OD.massless_quadrature_3d(order)
    shape = (6, 7, 33)
    for u in speeds:
        rng = np.random.default_rng(order)
        v = rng.standard_normal((3,) + shape)
        v *= u / np.sqrt((v * v).sum(0))
        lat = rl.Lattice3(33, 7, 6, tau=0.8, precision=precision, order=order)
        lat.init(1 + 0.3 * rng.random(shape), *[np.ascontiguousarray(a) for a in v], 1 + 0.2 * rng.random(shape))
        f = lat.populations()[_order3(lat, quad)]
        _check_fields3(lat.moments(), OD.macroscopic3(f, quad), _bar(f, quad, u), u)
        lat.close()


def _draws(H, f):
    """f = H M, and 64 times with errors 2^-40 sum_k |H_ik M_k| of random sign."""
    M = np.linalg.lstsq(H, f, rcond=None)[0]
    out = f[:, None] + 2.0 ** -40 * np.abs(H * M).sum(1)[:, None] * np.sign(
        np.random.default_rng(1).random((len(f), 65)) - 0.5)
    out[:, 0] = f
    return out


@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("u", [0.9, 0.95, 0.99, 0.995, 0.999, 0.9999])
def test_step3_of_a_uniform_stream(rl, order, u):
    """A uniform equilibrium stream: a step of its stored populations against the
    oracle's.  The bar is the oracle's amplification of rounding errors of the
    terms H_ik M_k (e sum_k |H_ik M_k| of either sign, e = 2^-40, the largest of 64
    draws), at 16 roundings: 16 times that at e = 2^-53."""
    plan = rl.plan3(order)
    nx, ny, nz = 34, 7, 6
    one = np.ones((nz, ny, nx))
    v = u * np.array([2.0, -1.0, 0.5]) / np.sqrt(5.25)
    lat = rl.Lattice3(nx, ny, nz, tau=0.8, precision="fp64", order=order)
    lat.init(one, *[c * one for c in v], one)
    f = lat.populations()
    quad = OD.massless_quadrature_3d(order)
    idx = _order3(lat, quad)
    draws = _draws(plan["H"], f[:, 0, 0, 0])[idx]
    fs, fields = OD.collide3(draws, quad, OD.Expansion3(quad, order), 0.8)
    assert fields.ok.all()
    bar = 16 * 2.0 ** (40 - 53) * rel_linf(fs[:, 1:], fs[:, :1])
    lat.step(1)
    assert lat.sync_status() == (0, 0)
    assert rel_linf(lat.populations()[idx], fs[:, :1, None, None]) <= bar
    lat.close()


GASES = [(0.0, 2), (0.0, 3), (1.0, 2), (5.0, 3)]


@pytest.mark.parametrize("m,order", GASES)
def test_fields2_of_fast_cells(rl, m, order):
    """As in (3+1)-d; T follows eps / n with a factor of at most eps / (n T)."""
    for u in (0.9, 0.95, 0.99, 0.995, 0.998, 0.999):
        rng = np.random.default_rng(order)
        th, shape = rng.uniform(0, 2 * np.pi, (7, 33)), (7, 33)
        lat = rl.Lattice(33, 7, m=m, order=order, tau=0.8, precision="fp64")
        quad = oracle_quadrature(m, order, lat.n, rl.plan(m=m, order=order)["v0"])
        lat.init(1 + 0.3 * rng.random(shape), u * np.cos(th), u * np.sin(th), 1 + 0.2 * rng.random(shape))
        f = lat.populations()[permutation(lat.n, lat.p, quad)]
        want, mo, bar = OS.macroscopic(f, quad), lat.moments(), _bar(f, quad, u)
        assert lat.sync_status() == (0, 0)
        assert np.abs(mo["n"] / want.n - 1).max() <= bar and np.abs(mo["eps"] / want.eps - 1).max() <= bar
        assert np.abs(mo["T"] / want.T - 1).max() <= bar * (want.eps / (want.n * want.T)).max()
        for k, name in ((1, "ux"), (2, "uy")):
            assert np.abs(mo[name] - want.U[k] / want.U[0]).max() <= bar * (1 - u * u)
        lat.close()


@pytest.mark.parametrize("m,order", GASES)
@pytest.mark.parametrize("u", [0.9, 0.99, 0.995, 0.999])
def test_step2_of_a_uniform_stream(rl, m, order, u):
    plan = rl.plan(m=m, order=order)
    one = np.ones((6, 34))
    lat = rl.Lattice(34, 6, m=m, order=order, tau=0.8, precision="fp64")
    quad = oracle_quadrature(m, order, lat.n, plan["v0"])
    idx = permutation(lat.n, lat.p, quad)
    lat.init(one, 0.8 * u * one, -0.6 * u * one, one)
    draws = _draws(plan["H"], lat.populations()[:, 0, 0])[idx][:, :, None]
    fs, fields = OS.collide(draws, quad, OL.Expansion(quad), 0.8)
    assert fields.ok.all()
    bar = 16 * 2.0 ** (40 - 53) * rel_linf(fs[:, 1:], fs[:, :1])
    lat.step(1)
    assert lat.sync_status() == (0, 0)
    assert rel_linf(lat.populations()[idx], fs[:, :1]) <= bar
    lat.close()


@pytest.mark.parametrize("order,speeds", [(2, (0.9, 0.95, 0.98, 0.99, 0.993, 0.995)), (3, (0.9, 0.95, 0.98, 0.99))])
def test_fp32_step3_of_uniform_streams(rl, order, speeds):
    """FP32 storage, 24 directions: a step of the stored populations against the
    oracle's, the bar as for FP64 at four roundings of 2^-24 (each moment is one
    FP32 sum over 12 or 39 runs).  A frame is found in every cell."""
    plan = rl.plan3(order)
    quad = OD.massless_quadrature_3d(order)
    one = np.ones((6, 6, 6))
    for u in speeds:
        d = np.random.default_rng(3).standard_normal((24, 3))
        for v in u * d / np.linalg.norm(d, axis=1)[:, None]:
            lat = rl.Lattice3(6, 6, 6, tau=0.8, precision="fp32", order=order)
            idx = _order3(lat, quad)
            lat.init(one, *[c * one for c in v], one)
            draws = _draws(plan["H"], lat.populations()[:, 0, 0, 0])[idx]
            fs, fields = OD.collide3(draws, quad, OD.Expansion3(quad, order), 0.8)
            assert fields.ok.all()
            lat.step(1)
            assert lat.sync_status() == (0, 0)
            bar = 4 * 2.0 ** (40 - 24) * rel_linf(fs[:, 1:], fs[:, :1])
            err = rel_linf(lat.populations()[idx], fs[:, :1, None, None])
            assert err <= bar, (u, err, bar)
            lat.close()
