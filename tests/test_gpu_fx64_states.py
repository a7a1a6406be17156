"""States at the limits of the FP64 steps in 64-bit fixed point: frames without a
temperature, rates and equilibria outside the fixed-point range, non-finite
populations, slow relaxation.  What the arithmetic there cannot hold is either
computed in FP64 or counted."""
import numpy as np
import pytest

from oracle import lattice as OL
from oracle import scheme as OS
from tests.cases import oracle_quadrature, permutation, rel_linf

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


@pytest.mark.parametrize("m,order,stream", [(0.0, 2, "onlattice"), (5.0, 3, "onlattice"), (0.0, 3, "bilinear"),
                                            (1.0, 2, "bilinear")])
def test_relaxation_time_fields_of_any_value(rl, m, order, stream):
    """tau of 0, NaN, infinity, a negative one and some far below and above one, in an
    interior cell, at an edge and in a corner each: what the oracle's FP64 relaxation
    gives, to 1e-12 of f (1 + 1/tau); not finite where it is not."""
    nx, ny = 35, 9
    lam = 0.9 if stream == "bilinear" else 0.0
    lat = rl.Lattice(nx, ny, m=m, order=order, tau_mode="field", precision="fp64", stream=stream, lam=lam)
    quad = oracle_quadrature(m, order, lat.n, rl.plan(m=m, order=order)["v0"])
    idx = permutation(lat.n, lat.p, quad)
    rng = np.random.default_rng(order)
    lat.init(1 + 0.3 * rng.random((ny, nx)), *(0.2 * rng.random((2, ny, nx)) - 0.1), 1 + 0.1 * rng.random((ny, nx)))
    f = lat.populations()[idx]
    f = OS.stream_onlattice(f, quad.n) if stream == "onlattice" else OS.stream_bilinear(f, lam * quad.velocity(), "periodic")
    odd = [0.0, np.nan, np.inf, -1.0, 1e-12, 2.0 ** -26.5, 2.0 ** -28.5, 1e-5, 1e5, 1e300, 5e-324]
    for at in ([4] * len(odd), [0] * len(odd), [ny - 1] * len(odd)):
        tau = np.full((ny, nx), 0.9)
        tau[at, (np.arange(len(odd)) * 3) % nx] = odd
        with np.errstate(all="ignore"):
            want = OS.collide(f, quad, OL.Expansion(quad), tau)[0]
            bar = 1e-12 * np.abs(f).max() * (1 + 1 / np.abs(tau))
        start = lat.populations()
        lat.set_tau_field(tau)
        lat.step(1)
        got = lat.populations()[idx]
        assert lat.sync_status() == (0, 0)
        ok = np.isfinite(want).all(0)
        assert (~ok).sum() == 3 and np.array_equal(np.isfinite(got).all(0), ok)
        assert (np.abs(got - want).max(0)[ok] <= bar[ok]).all()
        lat.set_populations(start)
    lat.close()


@pytest.mark.parametrize("order", [2, 3, 4, 5])
@pytest.mark.parametrize("wall", [2.0, 1e4, 1e8, 1e12])
def test_walls_of_any_temperature(rl, order, wall):
    """(1+1)-d: the equilibrium of a wall cell is a polynomial of the prescribed
    temperature, whose terms are all positive or as large as f itself at T >> 1: each
    wall cell to 1e-13 of its largest value, as its few roundings make."""
    from oracle import d1 as O1
    nx = 40
    one = np.ones(nx)
    lat = rl.Lattice1(nx, order=order, tau=0.9, boundary="eqwall_x", wall_T=(wall, 0.5 * wall), precision="fp64")
    q = O1.massless_quadrature_1d(order)
    sim = O1.Simulation1(q, nx, tau=0.9, boundary="eqwall_x", wall_T=(wall, 0.5 * wall))
    for s in (lat, sim):
        s.init(one, 0 * one, one)
        s.step(1)
    assert lat.sync_status() == (0, 0)
    pos = {(int(d), round(float(p), 9)): i for i, (d, p) in enumerate(zip(lat.n, lat.p[:, 0]))}
    got = lat.populations()[[pos[(int(d), round(float(p), 9))] for d, p in zip(q.n, q.p[:, 0])]]
    for x in (0, nx - 1):
        assert rel_linf(got[:, x], sim.fs[:, x]) <= 1e-13 * (1 if order < 5 else 10)
    assert rel_linf(got[:, 1:-1], sim.fs[:, 1:-1]) <= 1e-12
    lat.close()


@pytest.mark.parametrize("order,u", [(2, 0.9), (2, 0.999), (2, 0.9999), (2, 0.99999), (3, 0.9), (3, 0.999), (3, 0.9999),
                                     (5, 0.9), (5, 0.999)])
def test_fast_streams_in_one_dimension(rl, order, u):
    """A uniform stream (rates from e^theta / tau, 400 at the last speed): a step of
    its stored populations against the oracle's, at 16 times the oracle's own
    amplification of roundings sum_k |H_ik M_k| 2^-53 (as in test_gpu_fast_flow.py)."""
    from oracle import d1 as O1
    from tests.test_gpu_fast_flow import _draws
    one = np.ones(37)
    lat = rl.Lattice1(37, order=order, tau=0.8, precision="fp64")
    q = O1.massless_quadrature_1d(order)
    pos = {(int(d), round(float(p), 9)): i for i, (d, p) in enumerate(zip(lat.n, lat.p[:, 0]))}
    idx = [pos[(int(d), round(float(p), 9))] for d, p in zip(q.n, q.p[:, 0])]
    lat.init(one, u * one, one)
    draws = _draws(rl.plan1(order)["H"], lat.populations()[:, 0])[idx]
    fs, fields = O1.collide1(draws, q, O1.Expansion1(q), 0.8)
    assert fields.ok.all()
    lat.step(1)
    assert lat.sync_status() == (0, 0)
    assert rel_linf(lat.populations()[idx], fs[:, :1]) <= 16 * 2.0 ** (40 - 53) * rel_linf(fs[:, 1:], fs[:, :1])
    lat.close()


def _row3(precision, order, n):
    """Fields of a line of cells at rest, T = 1, of densities n along x, at t = 0."""
    from paper_1909_04502_gb300 import rlbm
    shape = (6, 6, len(n))
    lat = rlbm.Lattice3(len(n), 6, 6, tau=0.9, precision=precision, order=order)
    one = np.ones(shape)
    lat.init(np.ascontiguousarray(n * one), 0 * one, 0 * one, 0 * one, one)
    mo = {k: v[2, 3] for k, v in lat.moments().items()}
    lat.close()
    return mo


def _row1(precision, order, n):
    from paper_1909_04502_gb300 import rlbm
    lat = rlbm.Lattice1(len(n), order=order, tau=0.9, precision=precision)
    lat.init(n, 0 * n, 1 + 0 * n)
    mo = lat.moments()
    lat.close()
    return mo


@pytest.mark.parametrize("row,order", [(_row3, 2), (_row3, 3), (_row1, 3), (_row1, 5)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_fields_up_to_the_largest_populations(rl, row, order, precision):
    """Densities to the end of the storage's range have their fields, to its
    rounding; from where a population is infinite no field is finite."""
    top = 1e37 if precision == "fp32" else 1e300
    n = np.array([1.0, 1e20, 1e30, 1e34, 1e35, 1e36, 5e36, top, 3.0, 1e45 if precision == "fp32" else np.inf, np.nan, 2.0])
    tol = 1e-4 if precision == "fp32" else 1e-10
    mo = row(precision, order, n)
    good = np.isfinite(n) & (n <= top)
    with np.errstate(invalid="ignore"):
        assert np.abs(mo["n"] / n - 1)[good].max() <= tol and np.abs(mo["T"] - 1)[good].max() <= tol
    for k in ("n", "T", "eps", "ux"):
        assert np.isfinite(mo[k][good]).all() and not np.isfinite(mo[k][~good]).any(), k


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("m,order,steps", [(0.0, 2, 0), (0.0, 2, 1), (5.0, 3, 0), (5.0, 3, 1)])
def test_full_moments_of_non_finite_populations(rl, m, order, steps, bad):
    """N^a and T^ab of a cell with a population that is not finite are not finite,
    as their sums in FP64 are; those of the cells that it has not reached are."""
    nx, ny = 40, 30
    lat = rl.Lattice(nx, ny, m=m, order=order, tau=0.9, precision="fp64")
    one = np.ones((ny, nx))
    lat.init(one, 0 * one, 0 * one, one)
    f = lat.populations()
    f[3, 15, 20] = bad
    lat.set_populations(f)
    lat.step(steps)
    mo = lat.moments(full=True)
    y, x = 15, 20
    if steps:
        x, y = x + lat.n[3][0], y + lat.n[3][1]          # where it has moved
    far = one.astype(bool)
    far[y, x] = False
    for k, v in mo.items():
        v = v.reshape(-1, ny, nx)
        assert not np.isfinite(v[:, y, x]).any(), k
        assert np.isfinite(v[:, far]).all(), k
    lat.close()


@pytest.mark.parametrize("boundary", ["periodic", "freeflow_x", "eqwall_x"])
@pytest.mark.parametrize("order", [2, 3, 5])
def test_cells_without_a_frame_in_one_dimension(rl, order, boundary):
    """(1+1)-d, FP64: cells of negative density, at both ends and inside, and one with
    infinite (order 2) or NaN populations are counted and their populations
    streamed as they are, infinities included."""
    nx = 41
    n, u, T = np.ones(nx), np.full(nx, 0.1), np.ones(nx)
    for x in (0, 13, nx - 1):
        n[x] = -1.0
    n[20], u[20], T[20] = 1.7e308, 0.3, 3.0                    # n T overflows
    lat = rl.Lattice1(nx, order=order, tau=0.9, boundary=boundary, precision="fp64")
    lat.init(n, u, T)
    lat.sync_status()
    f = lat.populations()
    assert np.isinf(f[:, 20]).any() if order == 2 else np.isnan(f[:, 20]).any()
    s = np.ravel(lat.n)
    src = np.arange(nx)[None] - s[:, None]
    src = src % nx if boundary == "periodic" else np.clip(src, 0, nx - 1)
    g = np.take_along_axis(f, src, 1)                          # streamed
    p = lat.p[:, :1]
    with np.errstate(invalid="ignore"):
        B = [(p * p * g)[s == k].sum(0) for k in (1, -1)]
        none = ~((B[0] > 0) & (B[1] > 0) & np.isfinite(g).all(0))
    lat.step(1)
    got = lat.populations()
    assert lat.sync_status() == (-4, none.sum()) and none.sum() >= 4
    assert np.array_equal(got[:, none], g[:, none], equal_nan=True)
    assert np.isfinite(got[:, ~none]).all()
    lat.close()


@pytest.mark.parametrize("m,order,stream", [(0.0, 2, "onlattice"), (0.0, 3, "onlattice"), (5.0, 3, "onlattice"),
                                            (10.0, 2, "onlattice"), (0.0, 2, "bilinear"), (0.0, 3, "bilinear")])
def test_flows_without_frames_only_stream(rl, m, order, stream):
    """Negative densities everywhere, on the faces too: each step only streams (on the
    lattice bit by bit, bilinear to its four roundings), through the images that the
    steps themselves have stored."""
    nx, ny, steps = 37, 7, 3
    lam = 0.9 if stream == "bilinear" else 0.0
    y, x = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    lat = rl.Lattice(nx, ny, m=m, order=order, tau=0.9, precision="fp64", stream=stream, lam=lam)
    lat.init(-1 - 0.1 * np.cos(x + y), 0.1 * np.cos(1.0 * y), 0.1 + 0.0 * x, 1 + 0.1 * np.sin(1.0 * x))
    lat.sync_status(raise_on_error=False)
    f = lat.populations()
    lat.step(steps)
    assert lat.sync_status(raise_on_error=False) == (-4, steps * nx * ny)
    for _ in range(steps):
        f = OS.stream_onlattice(f, lat.n) if lam == 0 else OS.stream_bilinear(f, lam * lat.p[:, 1:] / lat.p[:, :1], "periodic")
    if lam == 0:
        assert np.array_equal(lat.populations(), f)
    else:
        assert np.abs(lat.populations() - f).max() <= steps * 4 * 2.0 ** -53 * np.abs(f).max()
    lat.close()


@pytest.mark.parametrize("precision,order", [("fp64", 2), ("fp64", 3), ("fp32", 2), ("fp32", 3)])
def test_flows_without_frames_only_stream_in_three_dimensions(rl, precision, order):
    from oracle import d3 as OD
    nx, ny, nz, steps = 35, 7, 6, 3
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    lat = rl.Lattice3(nx, ny, nz, tau=0.9, precision=precision, order=order)
    lat.init(-3 - 0.1 * np.cos(x + y + z), 0.1 * np.cos(1.0 * y), 0.1 + 0.0 * x, 0.1 * np.sin(1.0 * z), 1 + 0.1 * np.sin(1.0 * x))
    lat.sync_status()
    f = lat.populations()
    lat.step(steps)
    assert lat.sync_status() == (-4, steps * nx * ny * nz)
    for _ in range(steps):
        f = OD.stream3(f, lat.n)
    assert np.array_equal(lat.populations(), f)
    lat.close()


@pytest.mark.parametrize("order", [2, 3])
def test_infinite_populations_in_three_dimensions(rl, order):
    """A corner cell of infinite density: the populations that are not finite arrive as
    NaN, each in a cell that is counted and keeps its others; the rest is finite."""
    nx, ny, nz = 35, 13, 14
    one = np.ones((nz, ny, nx))
    n = one.copy()
    n[0, 0, 0] = np.inf
    lat = rl.Lattice3(nx, ny, nz, tau=0.9, precision="fp64", order=order)
    lat.init(n, 0.1 * one, 0 * one, 0 * one, one)
    lat.sync_status()
    f = lat.populations()
    hit = np.zeros((nz, ny, nx), bool)
    for i in np.flatnonzero(~np.isfinite(f[:, 0, 0, 0])):
        hit[tuple(lat.n[i][::-1] % (nz, ny, nx))] = True
    assert hit.sum() > 10
    lat.step(1)
    got = lat.populations()
    assert lat.sync_status() == (-4, hit.sum())
    for i, s in enumerate(lat.n):
        g = np.roll(f[i], (int(s[2]), int(s[1]), int(s[0])), (0, 1, 2))
        assert np.array_equal(got[i][hit], np.where(np.isfinite(g), g, np.nan)[hit], equal_nan=True)
    assert np.isfinite(got[:, ~hit]).all()
    lat.close()
