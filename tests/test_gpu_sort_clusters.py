"""The plan's sort where values lie far closer than their range spans.

Radii of points on a few circles, computed from Cartesian coordinates, differ in
their last bits and share the sort's 32-bit key: the order is numpy's stable sort,
and the plan takes no more than three times a plan of evenly spread values (four
passes over the key; where equal keys are out of order, at most five over the bits
below and four over the key again, a part of the plan each time).
"""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from gpu_helpers import dev, to_dev  # noqa: E402


def _circles(rng, n, k, outlier):
    a, rad = rng.uniform(0.0, 2.0 * np.pi, n), rng.choice(np.array([1.0, 0.4, 0.7, 0.25])[:k], n)
    v = np.hypot(rad * np.cos(a), rad * np.sin(a))
    if outlier:
        v[n // 3] = outlier
    return v


def _plan_us(r, omega, reps=7):
    import torch
    from paper_2411_09583_gb300 import Plan
    ts = []
    for _ in range(reps):
        torch.cuda.synchronize(dev())
        t = time.perf_counter()
        Plan(0, r, omega, 1e-8).close()
        torch.cuda.synchronize(dev())
        ts.append(time.perf_counter() - t)
    return 1e6 * min(ts)


def _check(n, k, outlier):
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(n + k)
    r, omega = _circles(rng, n, k, outlier), rng.uniform(0.0, 1.0, n)   # omega r <= 1: all local
    with Plan(0, to_dev(r), to_dev(omega), 1e-8) as p:
        pr, pw = p.permutations()
    assert np.array_equal(pr, np.argsort(r, kind="stable"))
    assert np.array_equal(pw, np.argsort(omega, kind="stable"))
    base, t = _plan_us(to_dev(rng.uniform(0.0, 1.0, n)), to_dev(omega)), _plan_us(to_dev(r), to_dev(omega))
    assert t <= 3.0 * base, (t, base)


@pytest.mark.parametrize("n", [1000, 1024, 4000, 8000, 8192])
@pytest.mark.parametrize("k,outlier", [(1, 1e-3), (4, 0.0), (2, 1e-300)])
def test_clusters_in_one_cta(n, k, outlier):
    _check(n, k, outlier)


@pytest.mark.parametrize("n", [8193, 100003, 1000003])
@pytest.mark.parametrize("k,outlier", [(1, 1e-3), (4, 0.0), (2, 1e-300)])
def test_clusters_over_many_ctas(n, k, outlier):
    _check(n, k, outlier)


@pytest.mark.parametrize("nprob,top", [(2, 9000), (300, 3000), (700, 400)])
def test_clusters_in_segments(nprob, top):
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(nprob)
    n, m = rng.integers(0, top, nprob), rng.integers(0, 90, nprob)
    n[0] = top
    r, omega = _circles(rng, int(n.sum()), 2, 1e-3), _circles(rng, int(m.sum()), 1, 1e-5)
    with Plan.many(rng.integers(0, 4, nprob), to_dev(r), n, to_dev(omega), m, 1e-6) as p:
        pr, pw = p.permutations()

    def want(x, cnt):
        off = np.concatenate([[0], np.cumsum(cnt)])
        return np.concatenate([off[i] + np.argsort(x[off[i]:off[i + 1]], kind="stable") for i in range(len(cnt))])
    assert np.array_equal(pr, want(r, n))
    assert np.array_equal(pw, want(omega, m))


@pytest.mark.parametrize("n", [5000, 60000])
def test_short_runs_beside_a_long_one(n):
    # pairs and triples of equal keys that differ in other bits than the long run's
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(n)
    v = np.concatenate([rng.uniform(0.5, 0.6, n), 1.0 + 2.0 ** -52 * rng.integers(0, 5, n), [1e-300]])
    r, omega = rng.permutation(v), rng.uniform(0.0, 1.0, 9000)
    with Plan(0, to_dev(r), to_dev(omega), 1e-8) as p:
        pr, _ = p.permutations()
    assert np.array_equal(pr, np.argsort(r, kind="stable"))
