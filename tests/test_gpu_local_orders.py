"""Local blocks at orders above 0: the evaluation keeps the last nu + 1 Bessel
values of its sweep.

All-local transforms (omega r <= z) over the orders where that rule can go
wrong: the smallest, even and odd, and orders larger than the highest one the
expansion needs (loose tolerances); arguments from far below 1 (power series)
to z; one real component and a pair.  Against the oracle within the accuracy
contract.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

from gpu_helpers import to_dev, tol  # noqa: E402


@pytest.mark.parametrize("pair", [False, True])
@pytest.mark.parametrize("eps", [1e-1, 1e-4, 1e-8, 1e-12])
@pytest.mark.parametrize("nu", [1, 2, 3, 10, 19, 64, 99, 100])
def test_all_local_orders(nu, eps, pair):
    from paper_2411_09583_gb300 import Plan, choose_params
    rng = np.random.default_rng(1000 + nu)
    _, z, _ = choose_params(nu, eps)
    r = rng.uniform(0.0, 1.0, 150)
    omega = np.concatenate([rng.uniform(0.0, z, 150), 10.0 ** rng.uniform(-12, 0, 40), [0.0, z]])
    c = rng.standard_normal(r.size)
    if pair:
        c = c + 1j * rng.standard_normal(r.size)
    with Plan(nu, to_dev(r), to_dev(omega), eps) as p:
        info = p.info()
        assert info["n_local"] > 0 and info["n_asy"] == info["n_direct"] == 0
        g = p.execute(to_dev(c)).cpu().numpy()
    err = np.max(np.abs(g - oracle.direct(nu, r, omega, c)))
    assert err <= tol(eps, c), (err, tol(eps, c))
