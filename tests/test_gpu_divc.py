"""FP32 division by a constant in the generated kernels: rounded to nearest, the
bits of numpy's x / c, for constants that need one and two corrections; subnormal
quotients within one step of the grid."""
import numpy as np
import pytest
import torch

from paper_2408_09662_gb300 import tracer as T
from paper_2408_09662_gb300.api import Function

pytestmark = pytest.mark.gpu

CONSTANTS = [12.0, 0.07, 0.26, 0.28, 3.0, 7.0, 0.1, -5.0, 1e-3, 1e10, 2.0, 1.0 / 3.0, 16777215.0, 8388609.0, 1.9999999,
             1.0000001, 49.0, -0.3, 2.0 ** -40, 2.0 ** 40, 2.0 ** 41]      # the last takes the plain division


@pytest.mark.parametrize("ways", [0, 2])
def test_division_by_constants_rounds_to_nearest(ways):
    g = T.Graph()
    (x,) = g.symbols(1)
    ir = T.Function([("x", [x])], [("y", [x / c for c in CONSTANTS])]).to_ir()
    fn = Function(ir, dtype="f32", ways=ways)
    src = fn.source()
    assert "cs_divc_f(" in src and "cs_divc2_f(" in src
    rng = np.random.default_rng(3)
    n = 1 << 20
    bits = rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)                # every exponent, NaNs
    mant = (rng.integers(0, 1 << 23, n, dtype=np.uint64).astype(np.uint32) | np.uint32(0x3f800000))
    edge = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1e-45, -1e-45, 1.1754944e-38, 3.4028235e38, -3.4028235e38,
                     2.0 ** -60, np.nextafter(np.float32(2.0 ** -60), np.float32(0)), 1.0, -1.0], dtype=np.float32)
    short = (rng.integers(1, 1 << 12, 1 << 16)[:, None] * np.array(CONSTANTS)).astype(np.float32).ravel()   # near-exact
    X = np.concatenate([bits.view(np.float32), mant.view(np.float32), edge, short])
    y = fn(torch.tensor(X[None], device="cuda")).cpu().numpy()
    with np.errstate(all="ignore"):
        for k, c in enumerate(CONSTANTS):
            want = X / np.float32(c)
            sub = (np.abs(want) < np.float32(2.0 ** -126)) & (want != 0)
            np.testing.assert_array_equal(y[k][~sub], want[~sub], err_msg=str(c))
            zero = want == 0
            np.testing.assert_array_equal(np.signbit(y[k][zero]), np.signbit(want[zero]), err_msg=str(c))
            assert np.all(np.abs(y[k][sub].astype(np.float64) - want[sub]) <= 2.0 ** -149), c


@pytest.mark.parametrize("ways", [0, 2])
def test_division_by_constants_at_both_ends_of_the_range(ways):
    """Subnormal quotients, and quotients next to overflow: the bits of x / c."""
    (x,) = T.Graph().symbols(1)
    ir = T.Function([("x", [x])], [("y", [x / c for c in CONSTANTS])]).to_ir()
    rng = np.random.default_rng(4)
    c = np.abs(np.array(CONSTANTS))
    half = (rng.integers(0, 1 << 23, 1 << 14) + 0.5) * 2.0 ** -149
    near = (half[:, None] * c).astype(np.float32).ravel()
    top = np.minimum(c * 2.0 ** 128, 3.4028234e38).astype(np.float32)
    X = np.concatenate([near, np.nextafter(near, np.float32(0)), -near, np.arange(1 << 16, dtype=np.uint32).view(np.float32)]
                       + [(top.view(np.int32) + np.int32(i)).view(np.float32) for i in range(-32, 33)])
    y = Function(ir, dtype="f32", ways=ways)(torch.tensor(X[None], device="cuda")).cpu().numpy()
    with np.errstate(all="ignore"):
        for k, v in enumerate(CONSTANTS):
            want = X / np.float32(v)
            same = (y[k].view(np.uint32) == want.view(np.uint32)) | (np.isnan(y[k]) & np.isnan(want))
            assert np.all(same), (v, X[~same][:3])
