"""Inputs split into double-float parts from their bits: every significand
counts to 48 bits.  A transform of x times a unit vector is x times that of the
unit vector (both within rounding, far below 10 eps |x|; a low part lost or
rounded the wrong way would show at 6e-8 |x|), forward and adjoint, for ties,
carries into the exponent, signs and values outside the FP32 range.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from gpu_helpers import to_dev  # noqa: E402

VALUES = [1.0 + 2.0 ** -24, 1.0 + 2.0 ** -23 + 2.0 ** -24, 1.0 + 2.0 ** -24 + 2.0 ** -52, 2.0 - 2.0 ** -52,
          2.0 - 2.0 ** -25, -(2.0 - 2.0 ** -24), -np.pi, 1.0 / 3.0, -1e-200, 1e200 / 3.0, -7.0 * 2.0 ** -1040]


@pytest.mark.parametrize("nu,min_size", [(0, 1024), (1, 64), (4, 1024)])
@pytest.mark.parametrize("x", VALUES)
def test_scaled_unit_vector(x, nu, min_size):
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(3)
    n, m = 700, 800
    r, omega = np.sort(rng.uniform(0.0, 1.0, n)), np.sort(rng.uniform(0.0, 900.0, m))
    with Plan(nu, to_dev(r), to_dev(omega), 1e-14, min_size=min_size) as p:
        for apply, size in ((p.execute, n), (p.adjoint, m)):
            for at in (1, size // 2, size - 2):
                u = np.zeros(size)
                u[at] = 1.0
                ref = apply(to_dev(u)).cpu().numpy()
                got = apply(to_dev(x * u)).cpu().numpy()
                # the subnormal range's own spacing beside the rounding
                assert np.max(np.abs(got - x * ref)) <= 1e-13 * abs(x) + 2.0 ** -1074


@pytest.mark.parametrize("nu", [0, 3])
def test_wide_range_of_inputs(nu):
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(4)
    n, m = 300, 310
    r, omega = rng.uniform(0.0, 1.0, n), rng.uniform(0.0, 500.0, m)
    c = rng.standard_normal(n) * 2.0 ** rng.integers(-120, 1, n)
    with Plan(nu, to_dev(r), to_dev(omega), 1e-14) as p:
        parts = sum(p.execute(to_dev(np.where(k == np.arange(n) % 3, c, 0.0))).cpu().numpy() for k in range(3))
        whole = p.execute(to_dev(c)).cpu().numpy()
    assert np.max(np.abs(whole - parts)) <= 1e-13 * np.sum(np.abs(c))
