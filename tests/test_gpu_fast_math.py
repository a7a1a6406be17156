"""The short quotients, square roots and conversions of the fixed-point steps and of
the (3+1)-d FP32 frame (rlbm_fast_math_f64, _f32) against correctly rounded results.

Bounds.  reciprocal and quotient end in one FMA whose correction is below 2^-19 of the
result, so that they round within 0.51 ulp: at most one ulp from the correctly rounded
value.  reciprocal_sqrt forms e = 1 - x y^2 from the rounded x y, an error of 2^-54 of
the result besides the last rounding: below 1.1 ulp, again one ulp from the rounded value."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rl():
    from paper_1909_04502_gb300 import rlbm
    return rlbm


def _f64(rl, a, b):
    import torch
    n = len(a)
    ta, tb = (torch.tensor(v, dtype=torch.float64, device="cuda") for v in (a, b))
    out = torch.empty(6 * n, dtype=torch.float64, device="cuda")
    assert rl.lib().rlbm_fast_math_f64(ta.data_ptr(), tb.data_ptr(), out.data_ptr(), n,
                                       torch.cuda.current_stream().cuda_stream) == 0
    return out.cpu().numpy().reshape(6, n)


def _f32(rl, a, b):
    import torch
    n = len(a)
    ta, tb = (torch.tensor(v, dtype=torch.float32, device="cuda") for v in (a, b))
    out = torch.empty(3 * n, dtype=torch.float64, device="cuda")
    assert rl.lib().rlbm_fast_math_f32(ta.data_ptr(), tb.data_ptr(), out.data_ptr(), n,
                                       torch.cuda.current_stream().cuda_stream) == 0
    return out.cpu().numpy().reshape(3, n)


def _ulps(a, b, kind):
    return np.abs(a.view(kind).astype(np.int64) - b.view(kind).astype(np.int64))


@pytest.mark.parametrize("span", [1, 30, 100, 500])
def test_quotients_and_roots_within_an_ulp(rl, span):
    """Random significands at exponents up to +-span, and those next to powers of two."""
    rng = np.random.default_rng(span)
    n = 1 << 20
    b = np.ldexp(1 + rng.random(n), rng.integers(-span, span + 1, n))
    edge = np.ldexp(1.0, np.arange(-span, span + 1))
    b = np.concatenate([b, edge, np.nextafter(edge, 0), np.nextafter(edge, np.inf)])
    a = np.ldexp(1 + rng.random(len(b)), rng.integers(-span, span + 1, len(b))) * rng.choice([-1, 1], len(b))
    got = _f64(rl, a, b)
    L = np.longdouble
    for k, want in enumerate((1 / b, a / b, (1 / np.sqrt(b.astype(L))).astype(np.float64))):
        assert _ulps(got[k], want, np.int64).max() <= 1, k


def test_cut_and_rounded_floats(rl):
    rng = np.random.default_rng(3)
    n = 1 << 18
    a = np.ldexp(1 + rng.random(n), rng.integers(-135, 127, n)) * rng.choice([-1, 1], n)
    edge = np.array([np.nextafter(s * np.ldexp(1.0, e), t) for e in (-149, -127, -126, -125, -121, -120, -119, -1, 0, 1, 126)
                     for s in (1, -1) for t in (-np.inf, 0, s * np.ldexp(1.0, e), np.inf)] + [0.0, -0.0])
    ties = np.float32(1 + rng.random(1000)).astype(np.float64) + 2.0 ** -24
    a = np.concatenate([a, edge, ties, -ties])
    got = _f64(rl, a, np.ones(len(a)))
    cut = (a.view(np.int64) & ~((1 << 29) - 1)).view(np.float64)         # the significand cut to 24 bits
    small = np.abs(a) < 2.0 ** -126
    assert np.array_equal(got[3], np.where(small, 0.0 * a, cut)) and np.array_equal(np.signbit(got[3]), np.signbit(a))
    half = (a.view(np.int64) + (1 << 28)).view(np.float64)               # ties away from zero
    away = (half.view(np.int64) & ~((1 << 29) - 1)).view(np.float64)
    assert np.array_equal(got[4], np.where(np.abs(away) < 2.0 ** -120, 0.0, away))
    assert not got[5].any()


def test_values_that_no_float_holds_are_reported(rl):
    top = np.ldexp(1.0, 127)
    a = np.array([top, -top, np.nextafter(top, np.inf), 1e39, -1e300, np.inf, -np.inf, np.nan, -np.nan,
                  np.nextafter(top, 0) * (1 - 2.0 ** -20), 1e37])
    assert _f64(rl, a, np.ones(len(a)))[5].tolist() == [1] * 9 + [0, 0]


def test_widened_floats(rl):
    rng = np.random.default_rng(4)
    bits = rng.integers(0, 2 ** 32, 1 << 18, dtype=np.uint64).astype(np.uint32)
    a = np.concatenate([bits.view(np.float32), np.array([0.0, -0.0, 1e-40, -3e-42, np.finfo(np.float32).tiny, 1.0], np.float32)])
    a = a[np.isfinite(a)]
    got = _f32(rl, a, np.ones(len(a), np.float32))
    normal = np.abs(a) >= np.finfo(np.float32).tiny
    for k in (1, 2):
        assert np.array_equal(got[k][normal], a[normal].astype(np.float64))
        assert (np.abs(got[k][~normal]) < 2.0 ** -126).all()
        assert np.array_equal(np.signbit(got[k]), np.signbit(a))
    zero = a == 0
    assert (np.abs(got[1][zero]) == 2.0 ** -127).all()


def test_float_quotient_within_an_ulp(rl):
    """Quotients that are normal, of normal divisors below 2^126."""
    rng = np.random.default_rng(5)
    n = 1 << 20
    b = np.ldexp(np.float32(1 + rng.random(n)), rng.integers(-60, 60, n)).astype(np.float32)
    a = (np.ldexp(np.float32(1 + rng.random(n)), rng.integers(-60, 60, n)) * rng.choice([-1, 1], n)).astype(np.float32)
    assert _ulps(_f32(rl, a, b)[0].astype(np.float32), a / b, np.int32).max() <= 1
