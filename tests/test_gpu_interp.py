"""Sparse interpolation tiles (forward and adjoint) at the edges of their window.

One asymptotic block whose outputs lie several cells apart, so that every tile
sums the taps of each output from a window of the grid: windows within a dense
tile's room, ones that run over the room of the per-bin sums, and ones too wide
to be staged, for few and many Hankel terms, short and long last tiles, one and
several members.  Against the oracle's direct sum within the accuracy contract
max|error| <= 10 eps ||input||_1.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

from gpu_helpers import to_dev, tol  # noqa: E402


@pytest.mark.parametrize("nvec", [1, 3])
@pytest.mark.parametrize("eps,nu", [(1e-5, 0), (1e-8, 17), (1e-12, 6), (1e-14, 1)])
@pytest.mark.parametrize("cells", [20, 45, 70, 100, 150, 210, 330, 1100])
@pytest.mark.parametrize("n,m", [(40, 257), (129, 33), (300, 150)])
def test_sparse_tiles(n, m, cells, eps, nu, nvec):
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(n + 7 * cells + nu)
    # r in [1, 2] spans 2 S / pi cells of the spreading grid (S the half-width in omega)
    s = 0.5 * np.pi * cells
    r = rng.uniform(1.0, 2.0, n)
    omega = rng.uniform(2000.0, 2000.0 + 2 * s, m)
    c, e = rng.standard_normal((n, nvec)), rng.standard_normal((m, nvec))
    with Plan(nu, to_dev(r), to_dev(omega), eps) as p:
        info = p.info()
        assert info["n_asy"] >= 1 and info["n_local"] == 0
        g = p.execute(to_dev(c)).cpu().numpy()
        ca = p.adjoint(to_dev(e)).cpu().numpy()
    for v in range(nvec):
        err = np.max(np.abs(g[:, v] - oracle.direct(nu, r, omega, c[:, v])))
        assert err <= tol(eps, c[:, v]), (err, tol(eps, c[:, v]))
        err = np.max(np.abs(ca[:, v] - oracle.direct(nu, omega, r, e[:, v])))
        assert err <= tol(eps, e[:, v]), (err, tol(eps, e[:, v]))
