"""FP64 steps at relaxation times from 0.8 to 10^6: a step of the
stored populations against the same step in extended precision.  Population i may be
off by its own last rounding, 2^-53 |f_i|, and by what the rate Omega_i leaves of
the equilibrium's rounding: 16 Omega_i 2^-53 sum_k |H_ik M_k|."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L = np.longdouble


@pytest.fixture(scope="module")
def rl():
    from paper_1909_04502_gb300 import rlbm
    return rlbm


def _frame(N, T):
    """n, eps, U (contravariant) of N [4, cells], T [4, 4, cells] by Newton on
    T00 - t.(S + l)^-1 t = l from the right."""
    t, S, l = T[0, 1:], T[1:, 1:], T[0, 0].copy()
    for _ in range(80):
        a, b, c = S[0, 0] + l, S[1, 1] + l, S[2, 2] + l
        A = [[b * c - S[1, 2] ** 2, S[0, 2] * S[1, 2] - S[0, 1] * c, S[0, 1] * S[1, 2] - S[0, 2] * b],
             [None, a * c - S[0, 2] ** 2, S[0, 1] * S[0, 2] - a * S[1, 2]], [None, None, a * b - S[0, 1] ** 2]]
        det = a * A[0][0] + S[0, 1] * A[0][1] + S[0, 2] * A[0][2]
        u = [sum(A[min(i, j)][max(i, j)] * t[j] for j in range(3)) / det for i in range(3)]
        w = 1 - sum(x * x for x in u)
        l = l + (T[0, 0] - sum(x * y for x, y in zip(t, u)) - l) / w
    g = 1 / np.sqrt(w)
    U = np.stack([g] + [g * x for x in u])
    return U[0] * N[0] - U[1] * N[1] - U[2] * N[2] - U[3] * N[3], l, U


def _moments(d, m, order, n, eps, U):
    """The Maxwell-Juttner moments of the basis of plan's (d = 2) or plan3's (d = 3) H."""
    e = eps / n
    T = e / 3 if d == 3 else 0.25 * (e - 2 * m + np.sqrt(e * e + 4 * m * (e - m)))
    r1 = 0.5 / T if d == 3 else 1 / (m + T)
    r2 = 4 * T if d == 3 else (m * m + 3 * m * T + 3 * T * T) / (m + T)
    r3 = 24 * T * T if d == 3 else (m ** 3 + 6 * m * m * T + 15 * m * T * T + 15 * T ** 3) / (m + T)
    q = T * (4 * T if d == 3 else r2)
    eta = lambda a, b: (1 if a == 0 else -1) if a == b else 0
    axes = range(1, d + 1)
    one, two = [()], [(a,) for a in axes]
    pairs = [(a, b) for a in axes for b in range(a, d + 1)]

    def mom(ix):
        if len(ix) == 0:
            return n * r1
        if len(ix) == 1:
            return n * U[ix[0]]
        if len(ix) == 2:
            return n * (r2 * U[ix[0]] * U[ix[1]] - T * eta(*ix))
        a, b, c = ix
        return n * (r3 * U[a] * U[b] * U[c] - q * (eta(a, b) * U[c] + eta(a, c) * U[b] + eta(b, c) * U[a]))

    # (d = 2, order 3: the members with p0 are p0 - m instead)
    sh = m if d == 2 and order == 3 else 0
    with0 = lambda ix: mom((0,) + ix) - sh * mom(ix)
    M = [mom(())] + [with0(())] + [mom(i) for i in two] + [with0(i) for i in two] + [mom(i) for i in pairs]
    if order == 3:
        M += [with0(i) for i in pairs]
        M += [mom((a, b, c)) for a in axes for b in range(a, d + 1) for c in range(b, d + 1)]
    return np.stack(M)


def _check(got, f, p, M, H, U, tau):
    H, p = H.astype(L), p.astype(L)
    om = (U[0][None] - (p[:, 1:] / p[:, :1]) @ U[1:]) / L(tau)
    want = f + om * (H @ M - f)
    bar = 2.0 ** -53 * (np.abs(f) + 16 * om * (np.abs(H) @ np.abs(M)))
    assert (np.abs(got - want) <= bar).all()
    return want


TAUS = [0.8, 3.0, 10.0, 1e3, 1e6]


@pytest.mark.parametrize("m,order", [(0.0, 2), (0.0, 3), (1.0, 2), (10.0, 2), (5.0, 3), (10.0, 3)])
@pytest.mark.parametrize("tau", TAUS)
def test_step2(rl, m, order, tau):
    nx, ny = 37, 9
    y, x = np.meshgrid(2 * np.pi * np.arange(ny) / ny, 2 * np.pi * np.arange(nx) / nx, indexing="ij")
    for tf in (False, True):
        lat = rl.Lattice(nx, ny, m=m, order=order, tau=tau, tau_mode="field" if tf else "const", precision="fp64")
        if tf:
            lat.set_tau_field(np.full((ny, nx), tau))
        lat.init(1 + 0.2 * np.cos(x), 0.3 * np.cos(y), 0.2 * np.sin(x + 1), 1 + 0.1 * np.sin(y + 2))
        f = lat.populations()
        f = np.stack([np.roll(a, (int(s[1]), int(s[0])), (0, 1)) for a, s in zip(f, lat.n)]).reshape(lat.Q, -1).astype(L)
        p = np.concatenate([lat.p, np.zeros((lat.Q, 1))], 1)
        N, T = p.T.astype(L) @ f, np.einsum("qa,qb,qc->abc", p.astype(L), p.astype(L), f)
        n, eps, U = _frame(N, T)
        lat.step(1)
        assert lat.sync_status() == (0, 0)
        _check(lat.populations().reshape(lat.Q, -1), f, p, _moments(2, L(m), order, n, eps, U),
               rl.plan(m=m, order=order)["H"], U, tau)
        lat.close()


@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("tau", TAUS)
def test_step3(rl, order, tau):
    nx, ny, nz = 33, 7, 6
    z, y, x = np.meshgrid(*(2 * np.pi * np.arange(k) / k for k in (nz, ny, nx)), indexing="ij")
    lat = rl.Lattice3(nx, ny, nz, tau=tau, precision="fp64", order=order)
    lat.init(1 + 0.2 * np.cos(x), 0.3 * np.cos(y), 0.2 * np.sin(z + 1), 0.1 * np.cos(x + y), 1 + 0.1 * np.sin(y + 2) + 0 * z)
    f = lat.populations()
    f = np.stack([np.roll(a, (int(s[2]), int(s[1]), int(s[0])), (0, 1, 2)) for a, s in zip(f, lat.n)])
    f, p = f.reshape(lat.Q, -1).astype(L), lat.p
    N, T = p.T.astype(L) @ f, np.einsum("qa,qb,qc->abc", p.astype(L), p.astype(L), f)
    n, eps, U = _frame(N, T)
    lat.step(1)
    assert lat.sync_status() == (0, 0)
    _check(lat.populations().reshape(lat.Q, -1), f, p, _moments(3, 0, order, n, eps, U), rl.plan3(order)["H"], U, tau)
    lat.close()


@pytest.mark.parametrize("order", [2, 3, 5])
@pytest.mark.parametrize("tau", TAUS)
def test_step1(rl, order, tau):
    nx = 131
    x = 2 * np.pi * np.arange(nx) / nx
    lat = rl.Lattice1(nx, order=order, tau=tau, precision="fp64")
    lat.init(1 + 0.2 * np.cos(x), 0.3 * np.cos(x + 1), 1 + 0.1 * np.sin(x + 2))
    f = np.stack([np.roll(a, int(s)) for a, s in zip(lat.populations(), np.ravel(lat.n))]).astype(L)
    p0, s = lat.p[:, 0].astype(L), np.sign(lat.p[:, 1]).astype(L)
    A, B = [[(w * f)[s == k].sum(0) for k in (1, -1)] for w in (p0[:, None], p0[:, None] ** 2)]
    eps, e2 = 2 * np.sqrt(B[0] * B[1]), np.sqrt(B[0] / B[1])          # e2 = e^(2 theta)
    E = np.sqrt(e2)
    n = A[0] / E + A[1] * E
    T, M, fact = eps / n, [], 1
    for a in range(1, order + 1):
        c = n * fact * T ** (a - 1) / 2
        M += [c * (E ** a + E ** -a), c * (E ** a - E ** -a)]
        fact *= a
    lat.step(1)
    assert lat.sync_status() == (0, 0)
    U = np.stack([(E + 1 / E) / 2, (E - 1 / E) / 2])
    _check(lat.populations(), f, lat.p, np.stack(M), rl.plan1(order)["H"], U, tau)
    lat.close()
