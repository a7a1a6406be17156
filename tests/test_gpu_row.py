"""Grids of one row in FP32 storage, whose steps share a kernel: against the
same flow on four equal rows, whose steps are launched one by one, over the
whole padded storage of both buffers (the images included).  Both run the same
operations per cell, so that only a contraction the compiler chose differently
can separate them: 2^-20 per step at populations that sum to one, where a wrong
image or a step too few is larger by orders of magnitude."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rl():
    from paper_1909_04502_gb300 import rlbm
    return rlbm


class _View:
    def __init__(self, owner, ptr, size):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (size,), "typestr": "<f4", "data": (ptr, False), "version": 3}


def _storage(lat):
    """The padded rows [Q][ny + 2 hy][nx + 2 hx] of f*(t) and f*(t - 1)."""
    import torch
    torch.cuda.synchronize()
    cur, prev, _elem, plane, (pitch, hx, hy, px) = lat.buffers()
    out = []
    for p in (cur, prev):
        raw = torch.as_tensor(_View(lat, p, lat.Q * plane), device="cuda")
        out.append(raw.as_strided((lat.Q, lat.ny + 2 * hy, lat.nx + 2 * hx), (plane, pitch, 1), px - hx).cpu().numpy())
    return out, hy


@pytest.mark.parametrize("nx", [1, 3, 33, 129, 2048, 2049])
@pytest.mark.parametrize("kw", [dict(), dict(stream="bilinear", lam=1.0), dict(boundary="freeflow_x"),
                                dict(m=1.0, boundary="eqwall_x", g=(1e-3, 2e-3)), dict(m=5.0, g=(0.0, 1e-3)),
                                dict(m=10.0, stream="bilinear", lam=0.8), dict(tau_mode="eta_over_s", eta_over_s=0.05, kappa=15.0)])
@pytest.mark.parametrize("steps", [1, 2, 7])
def test_row_equals_equal_rows(rl, nx, kw, steps):
    rng = np.random.default_rng(nx)
    row = [1 + 0.2 * rng.random(nx), 0.2 * rng.random(nx), 0.1 * rng.random(nx), 1 + 0.1 * rng.random(nx)]
    lats = []
    for ny in (1, 4):
        lat = rl.Lattice(nx, ny, precision="fp32", **{"tau": 0.8, **kw})
        lat.init(*[np.ascontiguousarray(np.tile(a, (ny, 1))) for a in row])
        lats.append(lat)
    (start, _), hy = _storage(lats[0])
    (want, _), _ = _storage(lats[1])
    tol = 2.0 ** -20
    for r in range(2 * hy + 1):
        assert np.abs(start[:, r] - want[:, hy]).max() <= tol
    for lat in lats:
        lat.step(steps)
        assert lat.sync_status() == (0, 0)
    got, _ = _storage(lats[0])
    want, _ = _storage(lats[1])
    for g, w in zip(got, want):
        tol = 2.0 ** -20 * (steps + 1)
        for r in range(2 * hy + 1):
            assert np.abs(g[:, r] - w[:, hy]).max() <= tol
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("kw", [dict(), dict(stream="bilinear", lam=1.0), dict(m=1.0, boundary="eqwall_x", g=(1e-5, 2e-5))])
@pytest.mark.parametrize("steps", [1024, 1025, 2048, 2051])
def test_long_calls_equal_short_ones(rl, kw, steps):
    """A call is split into launches of at most 1024 steps: both buffers, images
    included, are bit by bit those of calls of at most 100."""
    nx = 150
    rng = np.random.default_rng(5)
    row = [1 + 0.2 * rng.random((1, nx)), 0.2 * rng.random((1, nx)), 0.1 * rng.random((1, nx)), 1 + 0.1 * rng.random((1, nx))]
    out = []
    for size in (steps, 100):
        lat = rl.Lattice(nx, 1, precision="fp32", tau=0.8, **kw)
        lat.init(*row)
        for done in range(0, steps, size):
            lat.step(min(size, steps - done))
        assert lat.sync_status() == (0, 0) and lat.t == steps
        out.append(_storage(lat)[0])
        lat.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("shape", [0, 1, 2])
def test_rows_in_a_batch_and_by_the_direct_kernel(rl, shape):
    """One-row members of a batch (whose chains launch the row's kernel unchained) and the
    direct kernel: the same bits, and the batch's rows go on by themselves."""
    cfg = [dict(nx=150, ny=1, tau=0.8), dict(nx=33, ny=1, tau=1.1, m=1.0), dict(nx=2049, ny=1, tau=0.7, m=10.0),
           dict(nx=40, ny=24, tau=0.9), dict(nx=70, ny=1, tau=0.8, stream="bilinear", lam=1.0)]
    batch = rl.Batch([dict(c, precision="fp32") for c in cfg])
    lats = []
    for i, c in enumerate(cfg):
        rng = np.random.default_rng(i)
        s = (c["ny"], c["nx"])
        f = [1 + 0.2 * rng.random(s), 0.2 * rng.random(s), 0.1 * rng.random(s), 1 + 0.1 * rng.random(s)]
        lat = rl.Lattice(precision="fp32", **c)
        lat.set_step_kernel("direct")
        for x in (lat, batch[i]):
            x.init(*f)
        lats.append(lat)
    batch.config(shape, batch.info()["grid_max"][shape] if shape < 2 else 0)
    for k in (7, 4):
        batch.step(k)
        batch[0].step(3)
        for lat in lats:
            lat.step(k)
        lats[0].step(3)
        assert batch.sync_status() == (0, 0)
        for i, lat in enumerate(lats):
            assert np.array_equal(batch[i].populations(), lat.populations()), i
    batch.close()
