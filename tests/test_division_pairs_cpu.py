"""Pairs of FP64 quotients by one divisor (one call for two) in the generated
kernels: every program compiles, whichever of its divisions share a divisor.
path="compiled" throughout, so that no failure hides behind the interpreter."""
import random
from concurrent.futures import ThreadPoolExecutor

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


def test_a_quotient_that_waits_is_no_numerator_before_its_turn():
    """v1 is evaluated with v3; its own quotient v4 must not move up to v2."""
    def f(a, b, c, d):
        v1, v2, v3 = a / M, b / P, (c * d) / M
        return [v1 + v3, v2, v1 / P]
    load(program(f, 4), schedule=0)


def test_a_quotient_that_waits_is_no_argument_before_its_turn():
    def f(a, b, c, d):
        v1, v2, v3 = a / M, T.sin(b), (c * d) / M
        return [v3, v2, T.sin(v1)]
    load(program(f, 4), schedule=0, pair_calls=64)


def random_program(seed, ops, sines=True):
    """Sums, products, sines and quotients by two inputs and two constants; outputs are
    the values read last."""
    rng = random.Random(seed)
    x = T.Graph().symbols(6)
    v = list(x)
    for _ in range(ops):
        a, b = rng.choice(v[-12:]), rng.choice(v[-12:])
        v.append(rng.choice([lambda: a + b, lambda: a - b, lambda: a * b, lambda: T.sin(a) if sines else b - a, lambda: a / x[0],
                             lambda: a / x[1], lambda: a / M, lambda: a / P, lambda: a / P])())
    return T.Function([("x", list(x))], [("y", v[-8:])]).to_ir()


def test_random_programs_compile():
    cases = [(s, ops, opt) for s, ops in enumerate([12] * 20 + [30] * 20 + [80] * 10)
             for opt in ({"adjoint": 1}, {"pair_calls": 64})]

    def one(case):
        seed, ops, opt = case
        load(random_program(seed, ops), compile_threads=1, **opt)
    with ThreadPoolExecutor(8) as ex:
        list(ex.map(one, cases))
    Batch([random_program(s, 80) for s in range(50, 54)], [64] * 4, dtype="f64", cache_dir=None)
