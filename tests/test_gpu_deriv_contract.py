"""What a derivative plan reports, as the header states it: two problems (orders
nu - 1 and nu + 1) over two copies of the base plan's points and frequencies -- at
order 0 too, where one transform of order 1 stands for both."""
import ctypes

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

from gpu_helpers import to_dev  # noqa: E402


def _report(d, n, m):
    from paper_2411_09583_gb300 import _native as N
    lib = N.lib()
    info = N.NuhtPlanInfo()
    N.check(lib.nuht_info(d._h, ctypes.byref(info)), "nuht_info")
    pr, pw = np.full(2 * n, -1, np.int32), np.full(2 * m, -1, np.int32)
    N.check(lib.nuht_get_permutations(d._h, pr.ctypes.data_as(ctypes.c_void_p), pw.ctypes.data_as(ctypes.c_void_p)),
            "nuht_get_permutations")
    blocks = []
    for cls in range(3):
        cnt = ctypes.c_int64()
        N.check(lib.nuht_get_blocks(d._h, cls, None, 0, ctypes.byref(cnt)), "nuht_get_blocks")
        b = np.full((cnt.value, 4), -1, np.int64)
        N.check(lib.nuht_get_blocks(d._h, cls, b.ctypes.data_as(ctypes.c_void_p), cnt.value, ctypes.byref(cnt)),
                "nuht_get_blocks")
        # a shorter buffer takes the first of them
        if cnt.value > 1:
            part = np.full((cnt.value // 2 + 1, 4), -1, np.int64)
            N.check(lib.nuht_get_blocks(d._h, cls, part.ctypes.data_as(ctypes.c_void_p), part.shape[0],
                                        ctypes.byref(cnt)), "nuht_get_blocks")
            assert cnt.value == b.shape[0] and np.array_equal(part, b[:part.shape[0]])
        blocks.append(b)
    return info, pr, pw, blocks


@pytest.mark.parametrize("nu", [0, 1, -2])
def test_sizes_permutations_and_blocks(nu):
    from paper_2411_09583_gb300 import Plan
    rng = np.random.default_rng(31)
    n, m = 700, 600
    r, omega = rng.uniform(0.0, 1.0, n), rng.uniform(0.0, 900.0, m)
    with Plan(nu, to_dev(r), to_dev(omega), 1e-8) as p, p.deriv() as d:
        info, pr, pw, blocks = _report(d, n, m)
    assert (info.n, info.m) == (2 * n, 2 * m)
    assert np.array_equal(pr, np.tile(np.argsort(r, kind="stable"), 2))
    assert np.array_equal(pw, np.tile(np.argsort(omega, kind="stable"), 2))
    assert (info.n_local, info.n_asy, info.n_direct) == tuple(b.shape[0] for b in blocks)
    cover = np.zeros((2 * m, 2 * n), dtype=np.int8)
    rc = [0, 0]
    for cls, b in enumerate(blocks):
        for k0, k1, j0, j1 in b:
            cover[k0:k1 + 1, j0:j1 + 1] += 1
            if cls < 2:
                rc[cls] += k1 - k0 + 1 + j1 - j0 + 1
    assert np.all(cover[:m, :n] == 1) and np.all(cover[m:, n:] == 1)
    assert np.all(cover[:m, n:] == 0) and np.all(cover[m:, :n] == 0)
    assert (info.local_rows_cols, info.asy_rows_cols) == tuple(rc)
    assert info.direct_entries == sum((k1 - k0 + 1) * (j1 - j0 + 1) for k0, k1, j0, j1 in blocks[2])
