"""Double-precision programs evaluated on few instances (as many groups of 32 as the
GPU holds at once, one to four per SM) run in their cooperative form: same bits as
ways = 8, same results as the one-thread form within the FP64 rule, on both sides
of the limit, through every call that picks the form by the batch's size."""
import numpy as np
import pytest
import torch

from oracle import Oracle, tolerance
from paper_2408_09662_gb300 import inputs, programs
from paper_2408_09662_gb300.api import Function

pytestmark = pytest.mark.gpu

FEW, MANY = 152 * 32, 4 * 152 * 32


@pytest.mark.parametrize("n", [1, 31, 33, 1000, FEW, MANY + 1])
def test_form_by_batch_size(n):
    irb = programs.cartpole_rk4().to_bytes()
    X = inputs.cartpole(n, seed=n)
    x = torch.tensor(X, device="cuda")
    fn = Function(irb, dtype="f64")
    buf = torch.full((24, n + 7), 5.0, dtype=torch.float64, device="cuda")
    y = fn(x, out=buf[:, :n])
    same = Function(irb, dtype="f64", ways=8) if n <= FEW else Function(irb, dtype="f64", maxrregcount=128)
    assert torch.equal(y, same(x))
    assert torch.all(buf[:, n:] == 5.0)
    orc = Oracle(irb)
    ref = orc.eval(X)
    assert np.all(np.abs(y.cpu().numpy() - ref) <= tolerance(orc, X, ref, 1e-12, kind=0))
    host = fn.eval_host(torch.tensor(X).pin_memory(), chunks=3)     # the whole batch decides
    assert torch.equal(host, y.cpu())


def test_adjoint_with_shared_gradient():
    irb = programs.srb_step().to_bytes()
    n = 1000
    rng = np.random.default_rng(4)
    X = np.vstack([np.tile(rng.normal(0, 0.1, (144, 1)), (1, n)), rng.uniform(-0.1, 0.1, (12, n)), np.zeros((1, n))])
    B = rng.standard_normal((13, n))
    x, b = torch.tensor(X, device="cuda"), torch.tensor(B, device="cuda")
    got = []
    for fn in (Function(irb, dtype="f64"), Function(irb, dtype="f64", ways=8)):
        g = torch.ones(157, dtype=torch.float64, device="cuda")
        got.append((fn.adjoint(x, b, shared_out=g, accumulate_broadcast=True)[144:], g))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    ref = Oracle(irb).adjoint(X, B)
    np.testing.assert_allclose(got[0][1][:144].cpu().numpy() - 1.0, ref[:144].sum(1), rtol=1e-9, atol=1e-10)


@pytest.mark.parametrize("n", [38912, 38913, 50001])
def test_many_instances_at_128_registers(n):
    """Values past a thread's registers: the 128-register form runs when the batch
    no longer fits the GPU at 255.  The compiler may contract differently under
    another register bound, so the bits are compared with contraction off."""
    irb = programs.random_program(3000, seed=21).to_bytes()
    X = inputs.normal(64, n, seed=2)
    x = torch.tensor(X, device="cuda")
    fn = Function(irb, dtype="f64", fmad=0)
    y, b = fn(x), torch.tensor(inputs.normal(32, n, seed=3), device="cuda")
    for cap in (128, 255):
        other = Function(irb, dtype="f64", fmad=0, maxrregcount=cap)
        assert torch.equal(y, other(x))
    assert torch.equal(fn.adjoint(x, b), other.adjoint(x, b))
    idx = np.arange(0, n, 997)
    orc = Oracle(irb)
    ref = orc.eval(X[:, idx])
    got = Function(irb, dtype="f64")(x)[:, idx].cpu().numpy()
    assert np.all(np.abs(got - ref) <= tolerance(orc, X[:, idx], ref, 1e-12, kind=0))


@pytest.mark.parametrize("n", [1, 45000, 65537])
def test_single_precision_many_at_128_registers(n):
    """FP32 programs of 129 to 168 registers: the compiler's count while the batch fits
    the GPU at once, 128 beyond; the same bits on both sides (contraction off)."""
    irb = programs.random_program(5000, seed=101).to_bytes()
    x = torch.tensor(inputs.normal(64, n, seed=n), dtype=torch.float32, device="cuda")
    fn = Function(irb, dtype="f32", fmad=0)
    assert "__launch_bounds__(128) cs_fwd" in fn.source()
    assert torch.equal(fn(x), Function(irb, dtype="f32", fmad=0, maxrregcount=128)(x))


@pytest.mark.parametrize("name,dtype", [("cartpole", "f64"), ("srb", "f64"), ("random3k", "f64"), ("random5k", "f32")])
def test_bits_do_not_depend_on_the_batch_size(name, dtype):
    """The first n columns of a large batch have the bits of a batch of n: one form for
    few instances, one for most, one beyond one wave; contraction on (the default)."""
    ir = {"cartpole": programs.cartpole_rk4, "srb": programs.srb_step, "random3k": lambda: programs.random_program(3000, seed=21),
          "random5k": lambda: programs.random_program(5000, seed=101)}[name]()
    fn = Function(ir, dtype=dtype, adjoint=1)
    N = 65537
    g = torch.Generator(device="cuda").manual_seed(2)
    x = (torch.randn((fn.nnz_in, N), generator=g, device="cuda", dtype=torch.float64) * 0.3).to(fn.torch_dtype)
    b = torch.randn((fn.nnz_out, N), generator=g, device="cuda", dtype=torch.float64).to(fn.torch_dtype)
    y, xb = fn(x), fn.adjoint(x, b)
    acc = fn.adjoint(x, b, out=torch.ones_like(x), accumulate=True)
    for n in (1, 33, FEW, FEW + 1, MANY, MANY + 1, 38912, 38913, 50001):
        xn, bn = x[:, :n].contiguous(), b[:, :n].contiguous()
        assert torch.equal(fn(xn), y[:, :n]), n
        assert torch.equal(fn.adjoint(xn, bn), xb[:, :n]), n
        assert torch.equal(fn.adjoint(xn, bn, out=torch.ones_like(xn), accumulate=True), acc[:, :n]), n
