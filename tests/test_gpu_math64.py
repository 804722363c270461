"""FP64 exp, sin, cos, division and square root of the generated kernels and the
interpreter (csrc/math64.cuh), at the edges of their fixed-point ranges.

Division and square root are rounded to nearest, so they equal numpy's bit for
bit.  exp, sin and cos round a value known to 2^-57 or better once: at most
0.6 ulp from the extended-precision value.  Outside the ranges (special
values, subnormals, large arguments) the library's 2 ulp hold."""
import numpy as np
import pytest
import torch

from paper_2408_09662_gb300 import programs
from paper_2408_09662_gb300.api import Function
from paper_2408_09662_gb300.ir import Op

pytestmark = pytest.mark.gpu

PI2 = np.longdouble("1.57079632679489661923132169163975144")


def around(v):
    """v and its neighbours in double precision, both signs."""
    v = np.asarray(v, dtype=np.float64).ravel()
    v = np.concatenate([v, np.nextafter(v, np.inf), np.nextafter(v, -np.inf)])
    return np.concatenate([v, -v])


def evaluate(op, path, *rows):
    fn = Function(programs.single_op(op).to_bytes(), dtype="f64", path=path)
    x = torch.tensor(np.stack(rows), device="cuda")
    return fn(x)[0].cpu().numpy()


def ulps(y, ref):
    e = np.frexp(ref)[1]
    return np.abs(y.astype(np.longdouble) - ref) / np.ldexp(np.longdouble(1), np.maximum(e, -1021) - 53)


@pytest.mark.parametrize("path", ["compiled", "interp"])
@pytest.mark.parametrize("op", [Op.EXP, Op.SIN, Op.COS], ids=lambda o: o.name)
def test_functions_within_their_ulp(op, path):
    rng = np.random.default_rng(int(op))
    n = 20000
    x = [rng.uniform(-1, 1, n), rng.standard_normal(n) * 4, rng.uniform(-708, 708, n),
         np.ldexp(rng.uniform(1, 2, n), rng.integers(-60, 9, n)), around(np.ldexp(1.0, np.arange(-130, 10)))]
    if op == Op.EXP:
        step = np.log(np.longdouble(2)) / 256       # table steps: the index may be one off there
        x += [around((np.arange(-3000, 3000) * step).astype(np.float64)), around([708.0, 709.7, 745.0, 64.0])]
        ref_fn = np.exp
    else:
        k = np.concatenate([np.arange(1, 3000), rng.integers(3000, 160000, 2000)])
        x += [rng.uniform(-2.0 ** 18, 2.0 ** 18, n), around((k * PI2).astype(np.float64)),
              around((k * PI2 / 2).astype(np.float64)), around([2.0 ** 18, 2.0 ** -27, 0.5, 1e6, 1e15, 1e22])]
        ref_fn = np.sin if op == Op.SIN else np.cos
    x = np.concatenate(x)
    y = evaluate(op, path, x)
    ref = ref_fn(x.astype(np.longdouble))
    err = ulps(y, ref)
    ax = np.abs(x)
    fast = ax < 708 if op == Op.EXP else ax < 2.0 ** 18
    # next to a zero the library answers (the remainder keeps too few bits)
    fast &= np.abs(ref) > 2.0 ** -18 if op != Op.EXP else True
    assert err[fast].max() <= 0.6, (float(err[fast].max()), float(x[fast][np.argmax(err[fast])]))
    with np.errstate(over="ignore"):
        rest = ~fast & np.isfinite(ref.astype(np.float64))
    if np.finfo(np.longdouble).nmant > 100 or op == Op.EXP:   # extended sin of large arguments needs 113 bits
        assert err[rest].max() <= 2.0, float(err[rest].max())
    s = evaluate(op, path, np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e308, 800.0, -800.0]))
    if op == Op.EXP:
        np.testing.assert_array_equal(s, [1, 1, np.inf, 0, np.nan, 1, np.inf, np.inf, 0])
    else:
        assert np.all(np.isnan(s[2:5]))
        np.testing.assert_array_equal(s[[0, 1, 5]], [1, 1, 1] if op == Op.COS else [0.0, -0.0, 5e-324])
        assert op == Op.COS or np.signbit(s[1])


def bit_patterns(rng, n, lo, hi):
    """Doubles with exponent fields in [lo, hi]: random, trailing-zero and trailing-one mantissas."""
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    cut = rng.integers(0, 52, n).astype(np.uint64)
    low = (np.uint64(1) << cut) - np.uint64(1)
    pick = rng.integers(0, 4, n)
    m = np.where(pick == 0, m & ~low, np.where(pick == 1, m | low, m)) & np.uint64((1 << 52) - 1)
    e = rng.integers(lo, hi + 1, n).astype(np.uint64)
    s = rng.integers(0, 2, n).astype(np.uint64)
    return (s << np.uint64(63) | e << np.uint64(52) | m).view(np.float64)


@pytest.mark.parametrize("path", ["compiled", "interp"])
def test_division_and_square_root_round_to_nearest(path):
    rng = np.random.default_rng(7)
    n = 1 << 20
    a, b = bit_patterns(rng, n, 1, 2046), bit_patterns(rng, n, 1, 2046)
    a[: n // 2], b[: n // 2] = bit_patterns(rng, n // 2, 900, 1100), bit_patterns(rng, n // 2, 900, 1100)
    near = slice(0, n // 8)
    a[near] = b[near] * (1.0 + rng.integers(-2, 3, n // 8) * 2.0 ** -52)        # quotients next to 1
    exact = slice(n // 8, n // 4)
    a[exact] = b[exact] * rng.integers(1, 1 << 20, n // 8)                      # short quotients
    edge = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 2.0 ** -1022, 2.0 ** -509, 2.0 ** 512, 2.0 ** 513,
                     2.0 ** -510, 1.7976931348623157e308, 1.0, -3.0])
    ea, eb = (g.ravel() for g in np.meshgrid(edge, edge))
    a, b = np.concatenate([a, ea]), np.concatenate([b, eb])
    with np.errstate(all="ignore"):
        np.testing.assert_array_equal(evaluate(Op.DIV, path, a, b), a / b)
        q = evaluate(Op.DIV, path, ea, eb)
        np.testing.assert_array_equal(np.signbit(q[~np.isnan(q)]), np.signbit((ea / eb)[~np.isnan(q)]))
        np.testing.assert_array_equal(evaluate(Op.INV, path, b), 1.0 / b)
        r = np.abs(np.concatenate([a, b, np.square(rng.integers(1, 1 << 26, n).astype(np.float64)),
                                   np.square(1.0 + rng.integers(0, 1000, 4096) * 2.0 ** -52)]))
        np.testing.assert_array_equal(evaluate(Op.SQRT, path, r), np.sqrt(r))
        s = evaluate(Op.SQRT, path, np.array([-1.0, -0.0, 0.0, np.nan, -np.inf]))
        assert np.isnan(s[0]) and s[1] == 0 and np.signbit(s[1]) and s[2] == 0 and np.all(np.isnan(s[3:]))
