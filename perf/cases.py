"""The transforms that a user of this library runs, as measurable cases.

    g_k = sum_j c_j J_nu(omega_k r_j),  and its adjoint and gradients

Each case goes through the package's public entry points: ``nuht`` (plan, apply,
release), ``Plan.execute`` / ``Plan.adjoint`` on a kept plan, ``Plan.many`` for
batches, ``nuht_autograd`` for gradients and ``transform_host`` for host buffers.

A case's fields:
  call   oneshot | execute | solver | adjoint | batch | gradient | host
  n, m   points r_j and frequencies omega_k (of the whole batch's largest problem for "batch")
  nu, eps, dist, omega_max, min_size, precision, complex, nvec, group, count, sizes
dist: "uniform" r ~ U[0, 1], omega ~ U[0, omega_max]; "log" r = 10^U[-3, 0];
"grid" the exponential grid omega_j = r_j; "shell" r ~ U[1, 2],
omega ~ U[omega_max / 2, omega_max] (one asymptotic block).
"""
import math

import numpy as np
import torch

from paper_2411_09583_gb300 import Plan, nuht, transform_host
from paper_2411_09583_gb300.autograd import nuht_autograd
from paper_2411_09583_gb300.workloads import exponential_grid

# entries of the matrix J_nu(omega_k r_j) up to which exact() forms the direct sum
EXACT_ENTRIES = 2.1e10


def _case(name, call, n, m, nu, eps, dist="uniform", omega_max=0.0, min_size=1024, precision="fp64",
          is_complex=False, nvec=1, group=0, count=1, sizes=0):
    c = dict(call=call, n=n, m=m, nu=nu, eps=eps, dist=dist, omega_max=float(omega_max), min_size=min_size,
             precision=precision, complex=is_complex, nvec=nvec, group=group, count=count, sizes=sizes)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one small transform from unsorted points, start to end: a script's or a test's call
        _case("oneshot_2e3", "oneshot", 2000, 2000, 0, 1e-8, omega_max=2000),
        # one iteration (forward, then adjoint) of a small least-squares solve on a kept plan
        _case("solver_3e3", "solver", 3001, 2500, 1, 1e-10, omega_max=4000),
        # an ordinary transform of the method's hardest grid (already sorted, all scales)
        _case("grid_1e5", "oneshot", 100003, 100003, 0, 1e-8, dist="grid"),
        # the adjoint at an ordinary ragged size and a higher order, as in an inverse problem
        _case("adjoint_1e5", "adjoint", 90001, 110003, 10, 1e-10, omega_max=1e5),
        # several radial profiles on one set of points (one plan, one grouped call)
        _case("vectors_1e5", "execute", 150000, 120000, 0, 1e-12, omega_max=1e5, nvec=16, group=16),
        # a call on host buffers: upload, plan, transform, download
        _case("host_2e5", "host", 200003, 100001, 0, 1e-8, omega_max=1e5),
        # the benchmark's transform on a kept plan (repeated right-hand sides)
        _case("forward_1e6", "execute", 1000000, 1000000, 0, 1e-12, omega_max=1e5, min_size=4096),
        # the benchmark's step: a new set of points each time
        _case("oneshot_1e6", "oneshot", 1000000, 1000000, 0, 1e-12, omega_max=1e5, min_size=4096),
        # one training step with learned points: value, gradients in c and r
        _case("gradient_1e6", "gradient", 1000000, 1000000, 0, 1e-10, omega_max=1e5),
        # complex coefficients at engineering accuracy, points clustered at the origin
        _case("mixed_4e6", "execute", 4000000, 4000000, 1, 1e-5, dist="log", omega_max=4e4,
              precision="mixed", is_complex=True),
        # an uneven batch of many orders and sizes in one plan
        _case("batch_256", "batch", 100000, 100000, 20, 1e-8, count=256, sizes=5),
        # far field: every product large, grids beyond the L2 cache
        _case("farfield_4e6", "execute", 4000000, 4000000, 0, 1e-12, dist="shell", omega_max=2e7),
    ]


def _size(rng, lo, hi):
    """Log-uniform, odd ones among them."""
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    call = rng.choice(["oneshot", "oneshot", "execute", "execute", "solver", "adjoint", "batch", "gradient", "host",
                       "mixed", "farfield"])
    nu = rng.choice([0, 0, 1, 2, rng.randint(3, 20)])
    eps = rng.choice([1e-8, 1e-10, 1e-12])
    min_size = rng.choice([1024, 1024, 2048, 4096])
    if call == "batch":
        top = _size(rng, 2000, 100000)
        return _case(None, "batch", top, top, rng.randint(0, 20), 1e-8, count=_size(rng, 4, 200),
                     sizes=rng.randrange(1 << 30))
    if call == "mixed":
        n, m = _size(rng, 4e3, 3.5e6), _size(rng, 4e3, 3.5e6)
        return _case(None, "execute", n, m, nu if nu < 3 else 1, rng.choice([1e-5, 1e-6]),
                     dist=rng.choice(["log", "uniform"]), omega_max=_size(rng, 4e3, 1e5), precision="mixed",
                     is_complex=rng.random() < 0.5)
    if call == "farfield":
        n, m = _size(rng, 1e4, 3.5e6), _size(rng, 1e4, 3.5e6)
        return _case(None, "execute", n, m, 0, eps, dist="shell", omega_max=_size(rng, 1e5, 1.8e7))
    if call == "gradient":
        n, m = _size(rng, 2e3, 9e5), _size(rng, 2e3, 9e5)
        return _case(None, "gradient", n, m, min(nu, 10), rng.choice([1e-8, 1e-10]),
                     omega_max=_size(rng, 2e3, 1e5))
    top = 1e6 if call in ("oneshot", "execute") else 5e5
    n, m = _size(rng, 500, top), _size(rng, 500, top)
    dist = rng.choice(["uniform", "uniform", "uniform", "log", "grid"])
    nvec = group = 1
    if call == "execute":
        nvec = rng.choice([1, 1, 2, 5, 16])
        group = 0 if nvec < 5 else rng.choice([0, nvec])
        if nvec > 1:
            n, m = min(n, 200001), min(m, 200001)
    if dist == "grid":
        m = n
    return _case(None, call, n, m, nu, eps, dist=dist, omega_max=_size(rng, 1e3, 1e5), min_size=min_size,
                 nvec=nvec, group=group if nvec > 1 else 0)


def _device():
    return torch.device("cuda:0" if torch.cuda.is_available() else "cpu")


def _batch_sizes(case):
    """(nus, n, m) of a batch: fixed by the case, log-uniform sizes from 1 % of the largest on."""
    rng = np.random.default_rng(case["sizes"])
    lo, hi = math.log10(max(20.0, case["n"] / 100.0)), math.log10(case["n"])
    n = (10.0 ** rng.uniform(lo, hi, case["count"])).astype(np.int64)
    m = (10.0 ** rng.uniform(lo, hi, case["count"])).astype(np.int64)
    return rng.integers(0, case["nu"] + 1, case["count"]), n, m


def _inputs(case, seed):
    """Points, frequencies, coefficients and the upstream vector, from the seed alone."""
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(int(seed))

    def u(size, lo, hi):
        return torch.rand(size, generator=gen, device=dev, dtype=torch.float64) * (hi - lo) + lo

    if case["call"] == "batch":
        _, ns, ms = _batch_sizes(case)
        n, m = int(ns.sum()), int(ms.sum())
        r = u(n, 0.0, 1.0)
        top = torch.as_tensor(np.repeat(ms.astype(np.float64), ms), device=dev)
        w = u(m, 0.0, 1.0) * top
    else:
        n, m = case["n"], case["m"]
        if case["dist"] == "grid":
            r, w = (torch.as_tensor(v, device=dev) for v in exponential_grid(n))
        elif case["dist"] == "shell":
            r, w = u(n, 1.0, 2.0), u(m, 0.5 * case["omega_max"], case["omega_max"])
        else:
            r = 10.0 ** u(n, -3.0, 0.0) if case["dist"] == "log" else u(n, 0.0, 1.0)
            w = u(m, 0.0, case["omega_max"])
    kind = torch.complex128 if case["complex"] else torch.float64
    tail = (case["nvec"],) if case["nvec"] > 1 else ()
    c = torch.randn((n,) + tail, generator=gen, device=dev, dtype=kind)
    e = torch.randn((m,) + tail, generator=gen, device=dev, dtype=kind)
    return r, w, c, e


def prepare(case, seed):
    r, w, c, e = _inputs(case, seed)
    opts = dict(min_size=case["min_size"], precision=case["precision"])
    s = dict(case=case, r=r, w=w, c=c, e=e, opts=opts)
    if case["group"]:
        opts["vec_group"] = case["group"]
    if case["call"] in ("execute", "solver", "adjoint"):
        s["plan"] = Plan(case["nu"], r, w, case["eps"], **opts)
    elif case["call"] == "batch":
        nus, ns, ms = _batch_sizes(case)
        s["plan"] = Plan.many(nus, r, ns, w, ms, case["eps"], **opts)
    elif case["call"] == "gradient":
        c.requires_grad_(True)
        r.requires_grad_(True)
    elif case["call"] == "host":
        # page-locked buffers, as a program that streams data keeps them
        pin = torch.cuda.is_available()
        for k in ("r", "w", "c"):
            t = s[k].cpu()
            s[k] = (t.pin_memory() if pin else t).numpy()
        out = torch.empty(w.shape[0], dtype=torch.float64, pin_memory=pin)
        s["out"] = out.numpy()
        s.pop("e")
    return s


def run(s):
    case, call = s["case"], s["case"]["call"]
    if call == "oneshot":
        return nuht(case["nu"], s["r"], s["w"], s["c"], case["eps"], **s["opts"])
    if call == "host":
        return transform_host(case["nu"], s["r"], s["w"], s["c"], case["eps"], out=s["out"], **s["opts"])
    if call == "gradient":
        # loss = |g - e|^2 / 2 against the data e
        g = nuht_autograd(s["c"], s["r"], s["w"], case["nu"], case["eps"], **s["opts"])
        dc, dr = torch.autograd.grad(g, (s["c"], s["r"]), grad_outputs=g.detach() - s["e"])
        return {"g": g.detach(), "dc": dc, "dr": dr}
    if call == "adjoint":
        return s["plan"].adjoint(s["e"])
    g = s["plan"].execute(s["c"])
    if call == "solver":
        return {"g": g, "c": s["plan"].adjoint(g - s["e"])}
    return g


def work(case):
    """Inputs read once, outputs written once; arithmetic: every point spread
    and every frequency interpolated once for the leading term alone, at the
    w taps (two FLOP each, complex) that the tolerance needs."""
    if case["call"] == "batch":
        _, ns, ms = _batch_sizes(case)
        n, m = int(ns.sum()), int(ms.sum())
    else:
        n, m = case["n"], case["m"]
    comps = case["nvec"] * (2 if case["complex"] else 1)
    passes = {"solver": 2, "gradient": 3}.get(case["call"], 1)
    taps = math.ceil(-math.log10(case["eps"])) + 1
    vectors = {"solver": (n + 3 * m) + n, "gradient": 2 * n + 2 * m + n}.get(case["call"], n + m)
    return {"bytes": 8.0 * (n + m + comps * vectors), "flops": 4.0 * taps * (n + m) * comps * passes}


# ---- the direct sum in 64 bits ------------------------------------------------

def _two_prod(a, b):
    """x = fl(a b) and the rounding error a b - x (Dekker's product)."""
    x = a * b
    f = 134217729.0
    t = f * a
    ah = t - (t - a)
    al = a - ah
    t = f * b
    bh = t - (t - b)
    bl = b - bh
    return x, ((ah * bh - x) + ah * bl + al * bh) + al * bl


def _hankel_from(nu):
    return max(30.0, 0.5 * nu * nu)


def _bessel_small(nu, x):
    """J_nu(x) for x below _hankel_from(nu): power series below 2, else the
    backward recurrence normalised by J_0 + 2 sum J_2k = 1."""
    n0 = int(_hankel_from(nu)) + 60 + nu
    n0 += n0 % 2
    y = x.clamp_min(2.0)
    hi, lo = torch.zeros_like(y), torch.full_like(y, 1e-200)
    total, want = 2.0 * lo, torch.zeros_like(y)
    # lo holds J_k (scaled), hi J_{k+1}
    for k in range(n0, 0, -1):
        if k == nu:
            want = lo.clone()
        hi, lo = lo, (2.0 * k / y) * lo - hi
        if (k - 1) % 2 == 0:
            total = total + (lo if k == 1 else 2.0 * lo)
        if k % 8 == 0:
            f = torch.where(lo.abs() > 1e100, torch.full_like(y, 1e-150), torch.ones_like(y))
            hi, lo, total, want = hi * f, lo * f, total * f, want * f
    if nu == 0:
        want = lo
    big = want / total
    z = -0.25 * x * x
    term = torch.ones_like(x)
    s = torch.ones_like(x)
    for k in range(1, 24):
        term = term * z / (k * (k + nu))
        s = s + term
    small = s * torch.exp(nu * torch.log(0.5 * x) - math.lgamma(nu + 1)) if nu else s
    small = torch.where(x > 0, small, torch.full_like(x, 1.0 if nu == 0 else 0.0))
    return torch.where(x < 2.0, small, big)


def _bessel_large(nu, x, d):
    """J_nu(x + d) for x from _hankel_from(nu) on, |d| a rounding error of x."""
    a = [1.0]
    for k in range(1, 26):
        a.append(a[-1] * (4.0 * nu * nu - (2 * k - 1) ** 2) / (8.0 * k))
    i1 = 1.0 / x
    i2 = i1 * i1
    p = torch.full_like(x, a[24])
    q = torch.full_like(x, a[25])
    for k in range(11, -1, -1):
        sgn = 1.0 if k % 2 == 0 else -1.0
        p.mul_(i2).add_(sgn * a[2 * k])
        q.mul_(i2).add_(sgn * a[2 * k + 1])
    q.mul_(i1)
    c, s = torch.cos(x), torch.sin(x)
    c, s = c - d * s, s + d * c
    # cos and sin of (2 nu + 1) pi / 4
    h = math.sqrt(0.5)
    cp = (h, -h, -h, h)[nu % 4]
    sp = (h, h, -h, -h)[nu % 4]
    cc, ss = c * cp + s * sp, s * cp - c * sp
    return (p * cc - q * ss) * torch.sqrt(i1 * (2.0 / math.pi))


def _bessel(nu, w, r):
    """J_nu(w_k r_j) for a column of w and a row of r."""
    x, d = _two_prod(w, r)
    low = x < _hankel_from(nu)
    j = _bessel_large(nu, x.clamp_min(_hankel_from(nu)), torch.where(low, torch.zeros_like(d), d))
    if bool(low.any()):
        j[low] = _bessel_small(nu, x[low])
    return j


def _direct(nu, w, r, c):
    """sum_j J_nu(w_k r_j) c_j, some rows of the matrix at a time."""
    rows = max(1, int(6e6) // max(1, r.numel()))
    c2 = c.reshape(r.numel(), -1)
    out = torch.empty((w.numel(), c2.shape[1]), dtype=c2.dtype, device=w.device)
    for k in range(0, w.numel(), rows):
        out[k:k + rows] = _bessel(nu, w[k:k + rows, None], r[None, :]).to(c2.dtype) @ c2
    return out.reshape((w.numel(),) + tuple(c.shape[1:]))


def exact(case, seed):
    call = case["call"]
    per = {"solver": 2, "gradient": 4}.get(call, 1)
    if call == "batch":
        nus, ns, ms = _batch_sizes(case)
        # (many short rows: slower per entry)
        if per * float((ns * ms).sum()) > EXACT_ENTRIES / 4:
            return None
    elif per * case["n"] * case["m"] > EXACT_ENTRIES:
        return None
    r, w, c, e = _inputs(case, seed)
    nu = case["nu"]
    if call == "batch":
        ro, wo = np.concatenate([[0], np.cumsum(ns)]), np.concatenate([[0], np.cumsum(ms)])
        return torch.cat([_direct(int(nus[i]), w[wo[i]:wo[i + 1]], r[ro[i]:ro[i + 1]], c[ro[i]:ro[i + 1]])
                          for i in range(case["count"])])
    if call == "adjoint":
        return _direct(nu, r, w, e)
    g = _direct(nu, w, r, c)
    if call == "solver":
        return {"g": g, "c": _direct(nu, r, w, g - e)}
    if call == "gradient":
        u = g - e
        below = (-1.0 if nu == 0 else 1.0) * _direct(abs(nu - 1), r, w, w * u)
        return {"g": g, "dc": _direct(nu, r, w, u), "dr": 0.5 * c * (below - _direct(nu + 1, r, w, w * u))}
    if call == "host":
        return g.cpu().numpy()
    return g
