"""The eigenvalue kernels' reciprocal, root and rotation against exact rational arithmetic, over the whole
exponent range, pivot-sized and very large arguments among them.

Bounds: 2^-52 relative for 1 / x and 1 / sqrt(x) (the last rounding, 2^-53, and less than that again from the series
and the intermediate one).  For a rotation with u = 1 + t^2: |c^2 u - 1| <= 2^-50 (c within 2^-52 of 1 / sqrt(u), u itself
rounded); what is left of a_pq, c^2 (a_pq (1 - t^2) - t (a_qq - a_pp)), at most 2^-20 |a_pq|, since t is the exact
tangent to 2^-21 (float32 arguments truncated to 2^-23 each, four float32 roundings) and the remainder moves
by |t'/t - 1| |a_pq| at most; but all of a_pq where it is below 2^-60 |a_qq - a_pp| or 2^-990."""
import ctypes
from fractions import Fraction as F

import numpy as np
import pytest
import torch

import kernel_unit
from gpu_util import t as cuda

pytestmark = pytest.mark.gpu


def _call(name, ins, outs):
    lib = kernel_unit.load("fp64_unit")
    n = ins[0].shape[0]
    di = [cuda(np.asarray(a, np.float64)) for a in ins]
    do = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(outs)]
    torch.cuda.synchronize()
    p = lambda a: ctypes.c_void_p(a.data_ptr())
    assert getattr(lib, name)(*[p(a) for a in di], n, *[p(a) for a in do]) == 0
    return [a.cpu().numpy() for a in do]


def _arguments(lo, hi, seed):
    rng = np.random.default_rng(seed)
    e = np.concatenate([rng.integers(lo, hi, 3000), np.arange(lo, hi)])
    x = np.ldexp(1.0 + rng.random(e.shape[0]), e)
    near = np.ldexp(1.0 + 2.0 ** -52 * rng.integers(0, 4, 200), rng.integers(lo, hi, 200))
    return np.concatenate([x, near, np.ldexp(1.0, np.arange(lo, hi + 1)), np.ldexp(2 - 2.0 ** -52, np.arange(lo, hi))])


def test_reciprocal():
    x = _arguments(-1022, 1021, 1)
    x = np.concatenate([x, -x[:500]])
    (y,) = _call("fp64_rcp", [x], 1)
    for a, b in zip(x.tolist(), y.tolist()):
        assert abs(F(a) * F(b) - 1) <= F(1, 2 ** 52), (a, b)
    (z,) = _call("fp64_rcp", [np.array([np.ldexp(1.5, 1023), -np.ldexp(1.0, 1023)])], 1)
    assert (np.abs(z) <= 2.0 ** -1022).all()


def test_reciprocal_root():
    x = _arguments(-1022, 1023, 2)
    (y,) = _call("fp64_rsqrt", [x], 1)
    tol = 2 * F(1, 2 ** 52)  # x y^2 moves twice as far as y
    for a, b in zip(x.tolist(), y.tolist()):
        assert abs(F(a) * F(b) ** 2 - 1) <= tol + F(1, 2 ** 100), (a, b)


@pytest.mark.parametrize("scale", [0, -900, 900])
def test_rotation(scale):
    rng = np.random.default_rng(3 + abs(scale))
    n = 4000
    app, aqq = rng.standard_normal(n), rng.standard_normal(n)
    aqq[:500] = app[:500] * (1 + 2.0 ** -52 * rng.integers(-4, 5, 500))  # nearly equal or equal
    apq = rng.standard_normal(n) * 2.0 ** rng.integers(-90, 10, n)
    apq[rng.integers(0, n, 50)] = 0.0
    app, aqq, apq = (np.ldexp(v, scale) for v in (app, aqq, apq))
    t, c = _call("fp64_angle", [app, aqq, apq], 2)
    assert (np.abs(t) <= 1).all()
    for a, b, o, tt, cc in zip(app.tolist(), aqq.tolist(), apq.tolist(), t.tolist(), c.tolist()):
        T, C, d = F(tt), F(cc), F(b) - F(a)
        assert abs(C * C * (1 + T * T) - 1) <= F(1, 2 ** 50)
        left = abs(C * C * (F(o) * (1 - T * T) - T * d))
        small = abs(F(o)) <= F(1, 2 ** 60) * abs(d) or abs(o) < 2.0 ** -990
        rounding = F(1, 2 ** 52) * (abs(F(a)) + abs(F(b)))  # a_qq - a_pp is rounded
        assert left <= F(1, 2 ** 20) * abs(F(o)) + rounding or (small and tt == 0.0), (a, b, o, tt, cc)
    t0, c0 = _call("fp64_angle", [app, aqq, np.zeros(n)], 2)
    assert (t0 == 0).all() and (np.abs(c0 - 1) <= 2.0 ** -52).all()
    bad = np.array([np.nan, np.inf, -np.inf])
    for args in ((bad, np.ones(3), np.ones(3)), (np.ones(3), bad, np.ones(3)), (np.ones(3), np.zeros(3), bad)):
        t0, c0 = _call("fp64_angle", list(args), 2)
        assert (t0 == 0).all() and (np.abs(c0 - 1) <= 2.0 ** -52).all()
