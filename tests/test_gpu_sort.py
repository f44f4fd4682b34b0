"""The plan's sort against numpy's stable sort, entry for entry.

The device sorts by a 32-bit key formed from the range of the values and orders
equal keys by their full patterns: sizes around the one-CTA / many-CTA and the
tile boundaries, and values that share keys (duplicates, a narrow band beside
far smaller values, zeros, subnormals, a negative zero).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from gpu_helpers import to_dev  # noqa: E402


def _values(kind, n, rng):
    if kind == "uniform":
        return rng.uniform(0.0, 1.0, n)
    if kind == "equal":
        return np.full(n, 0.37)
    if kind == "duplicates":
        return rng.integers(0, 7, n) / 7.0
    if kind == "zeros":
        v = rng.uniform(0.0, 1.0, n)
        v[rng.random(n) < 0.4] = 0.0
        v[rng.random(n) < 0.1] = -0.0
        return v
    if kind == "band":
        # most values within 2^-40 of one another, the range spans decades
        v = 1.0 + rng.integers(0, 4096, n) * 2.0 ** -52
        v[rng.random(n) < 0.1] = 10.0 ** rng.uniform(-200, -1)
        v[rng.random(n) < 0.05] = 0.0
        return v
    if kind == "tiny":
        return rng.integers(0, 1000, n) * 5e-324
    return 10.0 ** rng.uniform(-300, 0, n)


@pytest.mark.parametrize("kind", ["uniform", "equal", "duplicates", "zeros", "band", "tiny", "decades"])
@pytest.mark.parametrize("n,m", [(1, 2), (33, 1), (1024, 1025), (4096, 4097), (8192, 5), (8193, 300), (131072, 40),
                                 (50, 131073), (300001, 200001)])
def test_permutations_are_numpys_stable_sort(kind, n, m):
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(n + m)
    r, omega = _values(kind, n, rng), _values(kind, m, rng)
    with Plan(0, to_dev(r), to_dev(omega), 1e-6) as p:   # omega r <= 1: all local
        pr, pw = p.permutations()
    # -0.0 sorts as 0.0
    assert np.array_equal(pr, np.argsort(r + 0.0, kind="stable"))
    assert np.array_equal(pw, np.argsort(omega + 0.0, kind="stable"))


@pytest.mark.parametrize("nprob", [2, 300])
@pytest.mark.parametrize("kind", ["uniform", "duplicates", "band"])
def test_segments_are_sorted_on_their_own(nprob, kind):
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(nprob)
    n, m = rng.integers(0, 400, nprob), rng.integers(1, 300, nprob)
    r, omega = _values(kind, int(n.sum()), rng), _values(kind, int(m.sum()), rng)
    with Plan.many(rng.integers(0, 4, nprob), to_dev(r), n, to_dev(omega), m, 1e-6) as p:
        pr, pw = p.permutations()

    def want(x, cnt):
        off = np.concatenate([[0], np.cumsum(cnt)])
        return np.concatenate([off[i] + np.argsort(x[off[i]:off[i + 1]] + 0.0, kind="stable")
                               for i in range(len(cnt))])
    assert np.array_equal(pr, want(r, n))
    assert np.array_equal(pw, want(omega, m))
