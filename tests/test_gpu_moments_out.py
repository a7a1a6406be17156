"""rlbm_moments into device memory: the kernel stores into the caller's planes where
it can (8-byte aligned memory of the current device), and copies where it cannot.
Both give the bits of the host call, in and out of graph capture."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NX, NY = 45, 7
PLANES = (("n", 1), ("ux", 1), ("uy", 1), ("T", 1), ("eps", 1), ("N", 3), ("Tab", 6))


@pytest.fixture(scope="module")
def rl():
    from paper_1909_04502_gb300 import rlbm
    return rlbm


def _lattice(rl, precision, m, order):
    lat = rl.Lattice(NX, NY, m=m, order=order, tau=0.8, precision=precision)
    rng = np.random.default_rng(1)
    lat.init(1 + 0.1 * rng.random((NY, NX)), *(0.1 * rng.random((2, NY, NX))), 1 + 0.1 * rng.random((NY, NX)))
    lat.step(2)
    return lat


@pytest.mark.parametrize("precision,m,order", [("fp32", 0.0, 2), ("fp64", 0.0, 2), ("fp64", 5.0, 3)])
@pytest.mark.parametrize("offset", [0, 4, 1])
def test_planes_at_any_byte(rl, precision, m, order, offset):
    import torch
    lat = _lattice(rl, precision, m, order)
    want = lat.moments(full=True)
    raw = {k: torch.zeros(NX * NY * c * 8 + 16, dtype=torch.uint8, device="cuda") for k, c in PLANES}
    ptr = {k: v.data_ptr() + offset for k, v in raw.items()}
    assert lib_moments(rl, lat, ptr) == 0
    torch.cuda.synchronize()
    for k, c in PLANES:
        got = raw[k][offset:offset + NX * NY * c * 8].cpu().numpy().copy().view(np.float64)
        assert np.array_equal(got, want[k].ravel()), k
        assert not raw[k][offset + NX * NY * c * 8:].any() and not raw[k][:offset].any()
    lat.close()


def lib_moments(rl, lat, ptr):
    return rl.lib().rlbm_moments(lat.h, *[ptr.get(k) for k, _ in PLANES], 1)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_device_planes_under_capture(rl, precision):
    import torch
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        lat = _lattice(rl, precision, 0.0, 2)
        out = {k: torch.zeros(c * NX * NY, dtype=torch.float64, device="cuda") for k, c in PLANES}
        lat.moments(full=True)                       # (kernels loaded)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            lat.step(2)
            lat.moments(out=out)
        graph.replay()
        torch.cuda.synchronize()
        want = lat.moments(full=True)
    for k, _ in PLANES:
        assert np.array_equal(out[k].cpu().numpy(), want[k].ravel()), k
    lat.close()
