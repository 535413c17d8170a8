"""The FP64 face kernel forms its square root from an FP32 reciprocal square
root seed and two Newton (Heron) steps with the remainder from one fused
multiply-add.  This checks the error bound on the host, with seeds off by up to
2^-22 (the hardware approximation and the operand cut to 24 bits together): the
result stays within 0.51 units in the last place.  The fused multiply-adds are
emulated in extended precision.  And the algebra of the closure: (5 - 2 r) / 3
with r = sqrt(4 - 3 f^2) is (3 + 4 f^2) / (5 + 2 r), and 2 - r = 3 f^2 / (2 + r)."""
import numpy as np
import pytest


def _fma(x, y, z):
    return (np.longdouble(x) * np.longdouble(y) + np.longdouble(z)).astype(np.float64)


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 63, reason="needs an extended long double for the fma emulation")
def test_newton_square_root_within_half_ulp():
    rng = np.random.default_rng(2)
    n = 400_000
    t = rng.uniform(1, 4, n) * 4.0 ** rng.integers(-300, 300, n)
    exact = np.sqrt(np.longdouble(t))
    y = (1 / exact).astype(np.float64) * (1 + rng.uniform(-1, 1, n) * 2.0 ** -22)
    h, g = 0.5 * y, t * y
    for _ in range(2):
        g = _fma(_fma(-g, g, t), h, g)
    err = np.abs((np.longdouble(g) - exact).astype(np.float64)) / np.spacing(exact.astype(np.float64))
    assert err.max() < 0.51


def test_closure_forms_agree():
    f = np.concatenate([[0.0, 1e-8, 1.0], np.random.default_rng(3).uniform(0, 1, 1000)])
    r = np.sqrt(4 - 3 * f * f)
    assert np.allclose((5 - 2 * r) / 3, (3 + 4 * f * f) / (5 + 2 * r), rtol=0, atol=1e-15)
    assert np.allclose(2 - r, 3 * f * f / (2 + r), rtol=0, atol=1e-15)
