"""Which multiplies round on their own in the generated kernels.  A program with
kernels for few, for most and for many instances has it decided before any of them
is written (and the compiler's contraction off), so that every instance has the same
bits whatever the batch's size: the statements of one value agree between the forms."""
import re

import pytest

from paper_2408_09662_gb300 import programs, tracer as T
from paper_2408_09662_gb300.api import Function


def values(fn, adjoint=False):
    """value -> expression, without the warp that a cooperative kernel loads it for."""
    src = fn.source(adjoint)
    src = src[src.index('extern "C" __global__'):]
    found = {}
    for v, e in re.findall(r"^\s*(?:const )?(?:double )?(v\d+) = (.*);$", src, flags=re.M):
        e = re.sub(r"(v\d+)_\d+", r"\1", e)
        if not re.search(r"\b(X|X2|Xb|X2b|W|cs_x)\[", e):      # loads
            found[v] = e
    return found


@pytest.mark.parametrize("make", [programs.cartpole_rk4, programs.srb_step, lambda: programs.ldlt_spd_solve(10),
                                  lambda: programs.random_program(800, seed=3)], ids=["cartpole", "srb", "ldlt10", "random"])
def test_forms_of_one_program_round_the_same_values(make):
    ir = make()
    one = Function(ir, dtype="f64", adjoint=1, cache_dir=None)
    eight = Function(ir, dtype="f64", adjoint=1, ways=8, cache_dir=None)
    for adjoint in (False, True):
        a, b = values(one, adjoint), values(eight, adjoint)
        plain = {v: e for v, e in a.items() if re.search(r" [-+*] |fma\(", e)}
        assert len(plain) > 100 and sum("fma(" in e for e in plain.values()) > 30
        assert {v: b[v] for v in plain} == plain


def test_multiplies_join_adds_where_every_reader_is_one():
    x = T.Graph().symbols(6)
    a, b, c, d, e, f = x
    two, out, third = a * b, c * d, e * f       # read by two adds; an output; read by an add and a product
    y = [two + c, e - two, out, out + f, third - a, third * b, a * a + b]
    for _ in range(64):                         # long enough for a form for few instances
        f = T.sin(f)
    y.append(f)
    fn = Function(T.Function([("x", x)], [("y", y)]).to_ir(), dtype="f64", cache_dir=None, schedule=0)
    found = list(values(fn).values())
    assert sum(e.startswith("fma(") for e in found) == 3
    assert sum(" * " in e for e in found) == 3
    assert sum(re.match(r"v\d+ [-+] v\d+$", e) is not None for e in found) == 2
    off = Function(T.Function([("x", x)], [("y", y)]).to_ir(), dtype="f64", fmad=0, cache_dir=None, schedule=0)
    assert "fma(" not in off.source()
