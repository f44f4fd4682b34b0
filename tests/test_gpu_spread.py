"""The dense spreading paths (forward and adjoint) at the edges of their rules.

One asymptotic block whose points fill few cells, so that every tile takes a
moment path: one, two and more bins per tile (bins are formed in pairs), tiles
with a remainder, both accumulation variants (the anchored one from eps = 1e-11
on), few and many Hankel terms, and coefficients of very different size in one
tile.  Against the oracle's direct sum within the accuracy contract
max|error| <= 10 eps ||input||_1.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

from gpu_helpers import to_dev, tol  # noqa: E402


def _input(kind, n, rng):
    x = rng.standard_normal(n)
    if kind == "spike":
        x[rng.integers(0, n)] = 1e9
    elif kind == "zeros":
        x[rng.random(n) < 0.9] = 0.0
        x[n // 2] = 1e-30
    return x


@pytest.mark.parametrize("kind", ["normal", "spike", "zeros"])
@pytest.mark.parametrize("eps,nu", [(1e-8, 0), (1e-8, 17), (1e-11, 0), (9.9e-12, 0), (1e-12, 6), (1e-14, 1)])
@pytest.mark.parametrize("n,m,cells", [(33, 40, 1), (255, 257, 2), (256, 600, 3), (700, 129, 9), (1500, 1300, 30)])
def test_dense_block(n, m, cells, eps, nu, kind):
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(n + 7 * cells + nu)
    # r in [1, 2] spans 2 S / pi cells of the spreading grid (S the half-width in omega)
    s = 0.5 * np.pi * cells
    r = rng.uniform(1.0, 2.0, n)
    omega = rng.uniform(600.0, 600.0 + 2 * s, m)
    c, e = _input(kind, n, rng), _input(kind, m, rng)
    with Plan(nu, to_dev(r), to_dev(omega), eps) as p:
        info = p.info()
        assert (info["n_local"], info["n_asy"], info["n_direct"]) == (0, 1, 0)
        g = p.execute(to_dev(c)).cpu().numpy()
        ca = p.adjoint(to_dev(e)).cpu().numpy()
    err = np.max(np.abs(g - oracle.direct(nu, r, omega, c)))
    assert err <= tol(eps, c), (err, tol(eps, c))
    err = np.max(np.abs(ca - oracle.direct(nu, omega, r, e)))
    assert err <= tol(eps, e), (err, tol(eps, e))
