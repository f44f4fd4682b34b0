"""The sparse spreading path (forward and adjoint) at the edges of its passes.

One asymptotic block whose points lie apart, from a window of little more than
the kernel's width (two lanes per output) to one of many passes with gaps
between the points, short and long last tiles, few and many Hankel terms, one
and several members, and the deterministic sums.  Against the oracle's direct
sum within the accuracy contract max|error| <= 10 eps ||input||_1.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

from gpu_helpers import to_dev, tol  # noqa: E402


def _check(nu, r, omega, eps, nvec, seed, **opt):
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(seed)
    c, e = rng.standard_normal((r.size, nvec)), rng.standard_normal((omega.size, nvec))
    with Plan(nu, to_dev(r), to_dev(omega), eps, **opt) as p:
        info = p.info()
        assert info["n_asy"] >= 1 and info["n_local"] == 0
        g = p.execute(to_dev(c)).cpu().numpy()
        ca = p.adjoint(to_dev(e)).cpu().numpy()
    for v in range(nvec):
        err = np.max(np.abs(g[:, v] - oracle.direct(nu, r, omega, c[:, v])))
        assert err <= tol(eps, c[:, v]), (err, tol(eps, c[:, v]))
        err = np.max(np.abs(ca[:, v] - oracle.direct(nu, omega, r, e[:, v])))
        assert err <= tol(eps, e[:, v]), (err, tol(eps, e[:, v]))


@pytest.mark.parametrize("nvec", [1, 2])
@pytest.mark.parametrize("eps,nu", [(1e-3, 0), (1e-8, 17), (1e-12, 0), (1e-14, 6)])
@pytest.mark.parametrize("cells", [3, 14, 60, 400, 1500])
@pytest.mark.parametrize("n,m", [(33, 35), (100, 257), (257, 90), (700, 520)])
def test_sparse_block(n, m, cells, eps, nu, nvec):
    rng = np.random.default_rng(n + 7 * cells + nu)
    # r in [1, 2] spans 2 S / pi cells of the spreading grid (S the half-width in omega)
    s = 0.5 * np.pi * cells
    r = rng.uniform(1.0, 2.0, n)
    omega = rng.uniform(3000.0, 3000.0 + 2 * s, m)
    _check(nu, r, omega, eps, nvec, n)


@pytest.mark.parametrize("det", [False, True])
def test_clusters_and_gaps(det):
    rng = np.random.default_rng(5)
    # three far clusters (many points on one cell each) and a few points between
    r = np.concatenate([1.0 + 1e-4 * rng.random(90), 1.5 + 1e-4 * rng.random(80), 2.0 - 1e-4 * rng.random(60),
                        rng.uniform(1.0, 2.0, 12)])
    omega = 3000.0 + 4000.0 * np.sort(rng.random(200)) ** 3
    _check(0, r, omega, 1e-10, 1, 6, **({"deterministic": True} if det else {}))
