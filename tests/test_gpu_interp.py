"""The interpreter's two layouts (few and many instances) and its slot tiers:
every instance has the same bits whichever layout, shared-memory budget, batch
size or position it is evaluated in, and the results match the oracle within
the FP64 rule (FP32 rule for FP32)."""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

from oracle import Oracle, tolerance
from paper_2408_09662_gb300 import _lib as L, inputs, programs
from paper_2408_09662_gb300.api import Function
from paper_2408_09662_gb300.experiments import _spd

pytestmark = pytest.mark.gpu

FEW = 152 * 32      # instances up to which the wide layout runs


def program(name):
    if name == "cartpole":
        return programs.cartpole_rk4(), lambda n: inputs.cartpole(n, seed=3)
    if name == "jacobian":      # too short to share: one warp, four groups per CTA
        return programs.quadrotor_step_sparse_jacobian(), lambda n: inputs.uniform(8, n, 0.1, 1.0, seed=4)
    if name == "ldlt22":        # multiply-add bundles, slots in both tiers
        return programs.ldlt_spd_solve(22), lambda n: _spd(22, n, seed=5)
    return programs.random_program(3000, seed=12), lambda n: inputs.normal(64, n, seed=6)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("name", ["cartpole", "jacobian", "ldlt22", "random3k"])
def test_layouts_and_tiers_agree_bit_for_bit(name, dtype):
    ir, make = program(name)
    irb = ir.to_bytes()
    n = FEW + 33
    X = make(n).astype(np.float32).astype(np.float64)
    fn = Function(irb, dtype=dtype, path="interp")
    x = torch.tensor(X, dtype=fn.torch_dtype, device="cuda")
    many = fn(x)
    for k in (1, 31, 97, FEW):
        assert torch.equal(fn(x[:, :k].contiguous()), many[:, :k]), k
    for kb in (0, 3, 200):
        other = Function(irb, dtype=dtype, path="interp", interp_shared_kb=kb)
        assert torch.equal(other(x), many), kb
        assert torch.equal(other(x[:, :97].contiguous()), many[:, :97]), kb
    idx = np.arange(0, n, 97)
    orc = Oracle(irb)
    ref = orc.eval(X[:, idx])
    tol = tolerance(orc, X[:, idx], ref, 1e-12 if dtype == "f64" else 2e-4, kind=0 if dtype == "f64" else 1)
    assert np.all(np.abs(many[:, idx].double().cpu().numpy() - ref) <= tol)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_adjoint_layouts_agree(dtype):
    """Shared gain's gradient and the states' adjoints, few and many instances,
    against the oracle's reverse sweep."""
    irb = programs.srb_step().to_bytes()
    fn = Function(irb, dtype=dtype, path="interp")
    n = FEW + 5
    rng = np.random.default_rng(8)
    X = np.vstack([np.tile(rng.normal(0, 0.1, (144, 1)), (1, n)), rng.uniform(-0.1, 0.1, (12, n)), np.zeros((1, n))])
    X = X.astype(np.float32).astype(np.float64)
    B = rng.standard_normal((13, n)).astype(np.float32).astype(np.float64)
    x = torch.tensor(X, dtype=fn.torch_dtype, device="cuda")
    b = torch.tensor(B, dtype=fn.torch_dtype, device="cuda")
    many = fn.adjoint(x, b)
    few = fn.adjoint(x[:, :65].contiguous(), b[:, :65].contiguous())
    assert torch.equal(few[144:], many[144:, :65])
    ref = Oracle(irb).adjoint(X[:, :65], B[:, :65])
    tol = 1e-10 if dtype == "f64" else 2e-4
    s = np.max(np.abs(ref), axis=1, keepdims=True) + 1e-30
    assert np.all(np.abs(few.double().cpu().numpy() - ref) <= tol * s)
    for k in (65, n):
        g = torch.zeros(157, dtype=fn.torch_dtype, device="cuda")
        fn.adjoint(x[:, :k].contiguous(), b[:, :k].contiguous(), shared_out=g)
        want = many[:144, :k].double().sum(1)
        assert torch.all((g[:144].double() - want).abs() <= tol * many[:144, :k].double().abs().sum(1) + 1e-30)


HAMMER = r"""
#include <cstdint>
#include <thread>
typedef int (*eval_t)(void*, const void*, int64_t, void*, int64_t, int64_t, void*, void*);
extern "C" int hammer(eval_t eval, void** fn, const void* x, void** y, void** ws, void** stream, int64_t n) {
  int status[2] = {0, 0};
  std::thread t[2];
  for (int k = 0; k < 2; ++k)
    t[k] = std::thread([&, k] {
      for (int i = 0; i < 20000 && !status[k]; ++i) status[k] = eval(fn[k], x, n, y[k], n, n, ws[k], stream[k]);
    });
  for (auto& u : t) u.join();
  return status[0] ? status[0] : status[1];
}
"""


def test_two_threads_with_layouts_of_different_size(tmp_path):
    """Several host threads may evaluate at once: a launch that needs little shared memory
    does not lower the limit of the interpreter kernel under another thread's launch."""
    (tmp_path / "hammer.cpp").write_text(HAMMER)
    so = str(tmp_path / "hammer.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-pthread", "-o", so, str(tmp_path / "hammer.cpp")], check=True)
    ir, make = program("ldlt22")
    n = 64
    x = torch.tensor(make(n), device="cuda")
    fns = [Function(ir.to_bytes(), dtype="f64", path="interp", interp_shared_kb=kb) for kb in (12, 48)]
    want = fns[0](x)
    assert torch.equal(fns[1](x), want)
    ys, ws = [torch.empty_like(want) for _ in fns], [f.workspace(n, False, "cuda") for f in fns]
    streams = [torch.cuda.Stream() for _ in fns]
    torch.cuda.synchronize()
    two = ctypes.c_void_p * 2
    status = ctypes.CDLL(so).hammer(
        ctypes.cast(L.lib().cusadi_eval, ctypes.c_void_p), two(*[f.handle for f in fns]), ctypes.c_void_p(x.data_ptr()),
        two(*[y.data_ptr() for y in ys]), two(*[w.data_ptr() if w is not None else None for w in ws]),
        two(*[s.cuda_stream for s in streams]), ctypes.c_int64(n))
    torch.cuda.synchronize()
    assert status == 0
    assert all(torch.equal(y, want) for y in ys)


@pytest.mark.parametrize("rows", [1, 2, 4])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_chains_of_ops_leave_no_places_idle(dtype, rows):
    """Quotients that need one another, one to four rows of them side by side: the same
    bits at every batch size, and a batch that fits the GPU with one warp to each row
    takes about as long as a small one."""
    from paper_2408_09662_gb300 import tracer as T
    x = T.Graph().symbols(2 * rows)
    v = list(x[:rows])
    for _ in range(100):
        v = [x[rows + j] / (v[j] + 2.0) + 0.1 for j in range(rows)]
    fn = Function(T.Function([("x", x)], [("y", v)]).to_ir(), dtype=dtype, path="interp")
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.rand((2 * rows, 65536 // rows), generator=g, device="cuda", dtype=torch.float64).to(fn.torch_dtype) + 0.5
    y = fn(X)
    for n in (1, 33, FEW, FEW + 1, 9000):
        assert torch.equal(fn(X[:, :n].contiguous()), y[:, :n]), n

    def ms(x):
        times = []
        for _ in range(9):
            s, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            s.record()
            for _ in range(5):
                fn(x, out=out[:, :x.shape[1]])
            e.record()
            e.synchronize()
            times.append(s.elapsed_time(e))
        return sorted(times)[4]
    out = torch.empty_like(y)
    assert ms(X) < 1.6 * ms(X[:, :4000].contiguous())
