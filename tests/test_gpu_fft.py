"""The double-float FFT of the asymptotic blocks at the edges of its pass rule.

One block (r in [1, 2], omega r far above z) whose spreading grid just fills an
FFT of 2^LN points: one pass up to 2^9, two up to 2^18, three above, lines of
5..9 bits, and every way the 2M Hankel terms are cut into chunks.  Forward and
adjoint against the oracle's direct sum, within the accuracy contract
max|error| <= 10 eps ||input||_1.
"""
import math

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

from gpu_helpers import to_dev, tol  # noqa: E402


def _block(LN, w, n, m, seed):
    # N1 = ceil(2 X S / pi + w / 2) + 1 with X = 1/2; the FFT has the smallest
    # power of two >= 2 (2 N1 + 1) points
    s = math.pi * (2 ** (LN - 2) - w / 2 - 3)
    rng = np.random.default_rng(seed)
    r = rng.uniform(1.0, 2.0, n)
    omega = rng.uniform(500.0, 500.0 + 2 * s, m)
    r[:2] = 1.0, 2.0
    omega[:2] = 500.0, 500.0 + 2 * s
    return r, omega, rng.standard_normal(n), rng.standard_normal(m)


@pytest.mark.parametrize("LN,eps,m_terms,members", [
    (6, 1e-8, 0, 1), (7, 1e-12, 0, 1), (8, 1e-12, 20, 1), (9, 1e-12, 0, 1), (9, 1e-10, 7, 3), (10, 1e-12, 0, 1),
    (11, 1e-4, 1, 1), (13, 1e-12, 5, 2), (15, 1e-12, 13, 1), (16, 1e-8, 0, 1), (17, 1e-12, 6, 1),
    (18, 1e-12, 0, 1), (19, 1e-12, 0, 1), (20, 1e-10, 9, 1)])
def test_one_block_at_every_pass_count(LN, eps, m_terms, members):
    from paper_2411_09583_gb300 import Plan
    w = math.ceil(-math.log10(eps)) + 1
    r, omega, c, e = _block(LN, w, 257, 301, 70 + LN)
    if members > 1:
        rng = np.random.default_rng(170 + LN)
        c, e = rng.standard_normal((r.size, members)), rng.standard_normal((omega.size, members))
    with Plan(1, to_dev(r), to_dev(omega), eps, m_terms=m_terms, vec_group=members) as p:
        info = p.info()
        assert (info["n_local"], info["n_asy"], info["n_direct"]) == (0, 1, 0)
        assert info["fft_points"] == 1 << LN
        g = p.execute(to_dev(c)).cpu().numpy()
        ca = p.adjoint(to_dev(e)).cpu().numpy()
    err = np.max(np.abs(g - oracle.direct(1, r, omega, c)), axis=0)
    assert np.all(err <= tol(eps, c)), (err, tol(eps, c))
    err = np.max(np.abs(ca - oracle.direct(1, omega, r, e)), axis=0)
    assert np.all(err <= tol(eps, e)), (err, tol(eps, e))


@pytest.mark.parametrize("count,n", [(1, 60), (3, 4000), (40, 500), (60, 1500)])
def test_mixed_blocks_of_both_size_classes(count, n):
    # mixed precision transforms a block's grids whole in one CTA, small and
    # large ones in launches of their own: none, few or many of either kind
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(count)
    ns, ms = rng.integers(n // 2, n + 1, count), rng.integers(n // 2, n + 1, count)
    r, omega = rng.uniform(0.0, 1.0, ns.sum()), rng.uniform(0.0, 1.0, ms.sum()) * n
    c = rng.standard_normal(r.size)
    nus = np.arange(count) % 4
    with Plan.many(nus, to_dev(r), ns, to_dev(omega), ms, 1e-5, precision="mixed", min_size=64) as p:
        g = p.execute(to_dev(c)).cpu().numpy()
    jo = io = 0
    for nu, a, b in zip(nus, ns, ms):
        ref = oracle.direct(int(nu), r[jo:jo + a], omega[io:io + b], c[jo:jo + a])
        assert np.max(np.abs(g[io:io + b] - ref)) <= tol(1e-5, c[jo:jo + a])
        jo += a
        io += b


@pytest.mark.parametrize("precision,eps", [("mixed", 1e-5), ("fp64", 1e-8)])
def test_many_small_tiles(precision, eps):
    # enough blocks that the spreading and interpolation run small and large tiles
    # in launches of their own
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(9)
    count, big = 500, 3
    ns = np.r_[np.full(count, 700), np.full(big, 6000)]
    nus = np.arange(ns.size) % 3
    r, omega = rng.uniform(0.0, 1.0, ns.sum()), rng.uniform(0.0, 1.0, ns.sum()) * np.repeat(ns, ns)
    c, e = rng.standard_normal(r.size), rng.standard_normal(r.size)
    with Plan.many(nus, to_dev(r), ns, to_dev(omega), ns, eps, precision=precision, min_size=32) as p:
        assert p.info()["n_asy"] >= 8192
        g = p.execute(to_dev(c)).cpu().numpy()
        ca = p.adjoint(to_dev(e)).cpu().numpy()
    at = 0
    for nu, n in zip(nus, ns):
        sl = slice(at, at + n)
        rows = rng.integers(0, n, 8)
        ref = oracle.direct(int(nu), r[sl], omega[sl][rows], c[sl])
        assert np.max(np.abs(g[sl][rows] - ref)) <= tol(eps, c[sl])
        ref = oracle.direct(int(nu), omega[sl], r[sl][rows], e[sl])
        assert np.max(np.abs(ca[sl][rows] - ref)) <= tol(eps, e[sl])
        at += n
