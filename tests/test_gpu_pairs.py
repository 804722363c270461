"""Functions evaluated two to a call in the generated kernels give the bits of the
functions one by one: FP64 quotients by one divisor, FP32 sin and cos of one
argument."""
import numpy as np
import pytest
import torch

from oracle import Oracle
from paper_2408_09662_gb300 import programs, tracer as T
from paper_2408_09662_gb300.api import Batch, Function
from paper_2408_09662_gb300.ir import Op
from test_division_pairs_cpu import random_program

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed,ops", [(s, 12 + 17 * (s % 5)) for s in range(20)])
def test_quotients_by_shared_divisors(seed, ops):
    """Sums, products and quotients, contraction off: every value is rounded as IEEE 754
    asks, so the results equal the oracle's bit for bit."""
    irb = random_program(seed, ops, sines=False).to_bytes()
    X = np.random.default_rng(seed).standard_normal((6, 257))
    x = torch.tensor(X, device="cuda")
    want = Oracle(irb).eval(X)
    for options in ({}, {"ways": 2}, {"inst_per_thread": 2}):
        fn = Function(irb, dtype="f64", path="compiled", fmad=0, **options)
        np.testing.assert_array_equal(fn(x).cpu().numpy(), want, err_msg=str(options))
    y = torch.empty((8, 257), dtype=torch.float64, device="cuda")
    Batch([irb], [257], dtype="f64", fmad=0)([x], [y])
    np.testing.assert_array_equal(y.cpu().numpy(), want)


def test_single_precision_sin_and_cos_together_on_every_argument():
    (x,) = T.Graph().symbols(1)
    both = Function(T.Function([("x", [x])], [("y", [T.sin(x), T.cos(x)])]).to_ir(), dtype="f32")
    assert "cs_sincos_f(v" in both.source()
    apart = [Function(programs.single_op(op).to_bytes(), dtype="f32") for op in (Op.SIN, Op.COS)]
    n = 1 << 26
    for k in range(64):
        bits = torch.arange(n, device="cuda", dtype=torch.int64) + (k * n - (1 << 31))
        v = bits.to(torch.int32).view(torch.float32)[None]
        y = both(v)
        for row, fn in enumerate(apart):
            w = fn(v)[0]
            same = (y[row].view(torch.int32) == w.view(torch.int32)) | (torch.isnan(y[row]) & torch.isnan(w))
            assert bool(same.all()), (k, fn)
