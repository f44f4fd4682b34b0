"""Host threads that execute plans of different shapes side by side.

Every kernel's dynamic shared memory follows the plan (Hankel terms, tile sizes,
groups) and, from 2048 asymptotic blocks on, is launched at two sizes per call:
threads on streams of their own get the results that they get alone.
"""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from gpu_helpers import dev, to_dev  # noqa: E402


def _plans(torch):
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(12)
    out = []
    for k, (eps, opts) in enumerate([(1e-12, {}), (1e-4, {}), (1e-8, {}), (1e-5, dict(precision="mixed"))]):
        # 2500 problems with an asymptotic block each, at least
        n = np.full(2500, 40)
        r, omega = rng.uniform(0.5, 1.0, 100000), rng.uniform(0.0, 400.0, 100000)
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            p = Plan.many(np.full(2500, k), to_dev(r), n, to_dev(omega), n, eps, stream=s, **opts)
            x = to_dev(rng.standard_normal(100000))
        assert p.info()["n_asy"] >= 2048
        out.append((p, s, x))
    # one far-field block: FFT passes of different tiles
    r, omega = rng.uniform(1.0, 2.0, 3000), rng.uniform(2e5, 4e5, 3000)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        out.append((Plan(0, to_dev(r), to_dev(omega), 1e-12, stream=s), s, to_dev(rng.standard_normal(3000))))
    return out


def test_threads_with_plans_of_different_shapes():
    import torch
    torch.cuda.synchronize(dev())
    plans = _plans(torch)
    want = []
    for p, s, x in plans:
        with torch.cuda.stream(s):
            want.append((p.execute(x), p.adjoint(x)))
    torch.cuda.synchronize(dev())
    failures = []

    def work(i):
        p, s, x = plans[i]
        try:
            with torch.cuda.stream(s):
                for _ in range(60):
                    g, a = p.execute(x), p.adjoint(x)
                s.synchronize()
            for got, ref in ((g, want[i][0]), (a, want[i][1])):
                # the order of the atomics: far below any tolerance
                if not float((got - ref).abs().max()) <= 1e-6 * float(ref.abs().max()):
                    failures.append((i, "result"))
        except Exception as e:   # noqa: BLE001
            failures.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(plans))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize(dev())
    assert not failures, failures
    for p, _, _ in plans:
        p.close()
