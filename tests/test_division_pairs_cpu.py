"""Pairs of FP64 quotients by one divisor (one call for two) in the generated
kernels: every program compiles, whichever of its divisions share a divisor.
path="compiled" throughout, so that no failure hides behind the interpreter."""
import pytest

from paper_2408_09662_gb300 import tracer as T
from paper_2408_09662_gb300.api import Batch, Function


def program(f, n):
    x = T.Graph().symbols(n)
    return T.Function([("x", x)], [("y", f(*x))]).to_ir()


def load(ir, **options):
    return Function(ir, dtype="f64", path="compiled", cache_dir=None, **options)


M, P = 1.5, 0.7     # divisors that are no powers of two


def test_a_quotient_belongs_to_one_pair():
    """Of three quotients by m, the second needs the first and is read by the third's
    sum: the third pairs with the first and must not pair again with the second."""
    ir = program(lambda a, b, c: [(a / M + b) / M + c / M], 3)
    assert load(ir).source().count("cs_divr2_d(") == 2          # the function and one call
    Batch([ir], [64], dtype="f64", cache_dir=None)


def test_the_same_in_a_reverse_sweep():
    ir = program(lambda a, b, c, p: [(a / p + b) / p + c / p, a / p * c], 4)
    load(ir, adjoint=1)
