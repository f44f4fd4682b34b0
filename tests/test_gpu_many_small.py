"""A batch of very many small problems: the host's work per problem."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from gpu_helpers import to_dev  # noqa: E402


def test_tables_of_many_problems():
    # 30000 problems of 21 orders: the precision split of an order's Hankel terms is
    # formed once, not per problem.  Before the split listed its items it took 0.3 us
    # a problem (0.5 with the lists formed for each)
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(4)
    count, n = 30000, 6
    nus, sizes = rng.integers(0, 21, count), np.full(count, n)
    r, omega = to_dev(rng.uniform(0.0, 1.0, count * n)), to_dev(rng.uniform(0.0, 100.0, count * n))
    best = np.inf
    for _ in range(5):
        with Plan.many(nus, r, sizes, omega, sizes, 1e-8) as p:
            best = min(best, p.info()["plan_ms"][2])
    assert 1e3 * best / count <= 0.3, best


@pytest.mark.parametrize("nus", [[0, 3, 3, -3, 17, 0, 17], [100, 1, 100, -1, 2]])
def test_repeated_orders_in_a_batch(nus):
    # the problems of an order that share its tables give what they give alone
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(len(nus))
    n = rng.integers(150, 400, len(nus))
    m = rng.integers(150, 400, len(nus))
    r, omega = rng.uniform(0.0, 1.0, n.sum()), rng.uniform(0.0, 4000.0, m.sum())
    c = rng.standard_normal(n.sum())
    eps = 1e-10
    with Plan.many(nus, to_dev(r), n, to_dev(omega), m, eps) as p:
        g = p.execute(to_dev(c)).cpu().numpy()
    ro, wo = np.concatenate([[0], np.cumsum(n)]), np.concatenate([[0], np.cumsum(m)])
    for i, nu in enumerate(nus):
        jr, jw = slice(ro[i], ro[i + 1]), slice(wo[i], wo[i + 1])
        with Plan(nu, to_dev(r[jr]), to_dev(omega[jw]), eps) as p:
            alone = p.execute(to_dev(c[jr])).cpu().numpy()
        # both within the contract of the direct sum
        assert np.max(np.abs(g[jw] - alone)) <= 20 * eps * np.abs(c[jr]).sum()
