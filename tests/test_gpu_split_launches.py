"""Small tiles in launches of their own (plans of at least 2048 asymptotic blocks):
with the components of a group, with pairs, in the deterministic mode and in mixed
precision, forward and adjoint, against the oracle's direct sum per problem within
10 eps ||input||_1; and the order-0 derivative plan through groups of vectors."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

from gpu_helpers import to_dev  # noqa: E402


@pytest.mark.parametrize("eps,comps,opts", [(1e-10, 3, dict(vec_group=3)), (1e-10, 5, dict(vec_group=2)),
                                            (1e-12, 2, dict(deterministic=True)),
                                            (1e-5, 3, dict(precision="mixed", vec_group=3))])
def test_members_and_modes(eps, comps, opts):
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(int(-np.log10(eps)) + comps)
    count = 2100
    n, m = rng.integers(2, 40, count), rng.integers(2, 40, count)
    n[:4], m[:4] = (64, 65, 300, 513), (300, 64, 65, 513)   # full tiles among the small ones
    nus = rng.integers(0, 6, count)
    r, omega = rng.uniform(0.5, 1.0, n.sum()), rng.uniform(900.0, 1200.0, m.sum())
    c, e = rng.standard_normal((r.size, comps)), rng.standard_normal((omega.size, comps))
    with Plan.many(nus, to_dev(r), n, to_dev(omega), m, eps, **opts) as p:
        assert p.info()["n_asy"] >= 2048
        g, a = p.execute(to_dev(c)).cpu().numpy(), p.adjoint(to_dev(e)).cpu().numpy()
        if opts.get("deterministic"):
            assert np.array_equal(g, p.execute(to_dev(c)).cpu().numpy())
            assert np.array_equal(a, p.adjoint(to_dev(e)).cpu().numpy())
    ro, wo = np.concatenate([[0], np.cumsum(n)]), np.concatenate([[0], np.cumsum(m)])
    for i in list(range(60)) + list(range(60, count, 41)):
        jr, jw = slice(ro[i], ro[i + 1]), slice(wo[i], wo[i + 1])
        err = np.max(np.abs(g[jw] - oracle.direct(int(nus[i]), r[jr], omega[jw], c[jr])), axis=0)
        assert np.all(err <= 10 * eps * np.abs(c[jr]).sum(axis=0)), (i, err)
        err = np.max(np.abs(a[jr] - oracle.direct(int(nus[i]), omega[jw], r[jr], e[jw])), axis=0)
        assert np.all(err <= 10 * eps * np.abs(e[jw]).sum(axis=0)), (i, err)


@pytest.mark.parametrize("nvec,group", [(3, 3), (5, 4), (17, 16), (4, 1)])
def test_order_zero_gradients_of_groups(nvec, group):
    # J_0' = -J_1: grad_r[j] = -sum_v c[j, v] sum_k e[k, v] omega_k J_1(omega_k r_j)
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(nvec)
    eps, n, m = 1e-10, 900, 800
    r, omega = rng.uniform(0.0, 1.0, n), rng.uniform(0.0, 2000.0, m)
    c, e = rng.standard_normal((n, nvec)), rng.standard_normal((m, nvec))
    with Plan(0, to_dev(r), to_dev(omega), eps, vec_group=group) as p, p.deriv() as d:
        gr, gw = d.grad_r(to_dev(c), to_dev(e)).cpu().numpy(), d.grad_omega(to_dev(c), to_dev(e)).cpu().numpy()
    we, rc = omega[:, None] * e, r[:, None] * c
    ref_r = -np.sum(c * oracle.direct(1, omega, r, we), axis=1)
    ref_w = -np.sum(e * oracle.direct(1, r, omega, rc), axis=1)
    assert np.all(np.abs(gr - ref_r) <= 10 * eps * np.abs(c) @ np.abs(we).sum(axis=0))
    assert np.all(np.abs(gw - ref_w) <= 10 * eps * np.abs(e) @ np.abs(rc).sum(axis=0))
