"""Which step kernel a handle launches: the fixed-point step wherever its tables
apply, the FP64 sums elsewhere."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _profiled(work):
    import torch
    torch.cuda.synchronize()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        work()
        torch.cuda.synchronize()
    return " ".join(e.key for e in prof.key_averages())


@pytest.fixture(scope="module")
def rl():
    import torch
    from paper_1909_04502_gb300 import rlbm
    _profiled(lambda: torch.zeros(8, device="cuda"))       # (the first trace of a process may come back empty)
    return rlbm


def _kernels(lat, fields):
    lat.init(*fields)
    lat.step(1)
    return _profiled(lambda: lat.step(1))


# every stencil with an orbit-symmetric evaluation: massless, the App. H tables of order 2 and
# columns A to D of order 3, and the 45-vector stencil of the paper's performance table
STENCILS = [(0.0, 2, None), (0.0, 3, None), (1.0, 2, None), (5.0, 2, None), (10.0, 2, None), (2.0, 3, None), (3.0, 3, None),
            (5.0, 3, None), (10.0, 3, None),
            (15.0, 3, [(0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2), (3, 0), (3, 2), (3, 3), (4, 0)])]


@pytest.mark.parametrize("m,order,groups", STENCILS)
@pytest.mark.parametrize("stream", ["onlattice", "bilinear"])
def test_fp64_steps_take_the_fixed_point_kernel(rl, m, order, groups, stream):
    one = np.ones((6, 40))
    lat = rl.Lattice(40, 6, m=m, order=order, groups=groups, tau=0.9, precision="fp64", stream=stream,
                     lam=0.9 if stream == "bilinear" else 0.0)
    names = _kernels(lat, [one, 0 * one, 0 * one, one])
    assert "k_step2x" in names and "k_step<" not in names
    lat.close()


def test_steps_without_fixed_point_tables_take_the_fp64_sums(rl):
    """Forces and walls, and a table whose orbits are in another order."""
    one = np.ones((6, 40))
    q = rl.plan(m=5.0, order=2)
    custom = np.concatenate([q["n"], q["p"], q["w"][:, None]], 1)[::-1]
    for kw in (dict(m=5.0, g=(1e-3, 0.0)), dict(m=0.0, boundary="eqwall_x"),
               dict(m=5.0, quadrature="custom", custom=custom)):
        lat = rl.Lattice(40, 6, tau=0.9, precision="fp64", **kw)
        names = _kernels(lat, [one, 0 * one, 0 * one, one])
        assert "k_step<" in names and "k_step2x" not in names
        lat.close()
