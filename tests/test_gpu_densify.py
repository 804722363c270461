"""Dense blocks of a sparse output at the edges of the copy's pieces: whole
16-byte pieces and single elements, ragged ends, strided results; a copy, so
bit for bit."""
import pytest
import torch

from paper_2408_09662_gb300 import _lib as L, programs
from paper_2408_09662_gb300.api import Function

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n,ld", [(1, 1), (3, 4), (8, 8), (2047, 2048), (4096, 4096), (4099, 4100), (10007, 10007)])
def test_densify_copies_every_entry(n, ld, dtype):
    ir = programs.quadrotor_step_sparse_jacobian()
    fn = Function(ir.to_bytes(), dtype=dtype)
    y = torch.randn((fn.nnz_out, ld), device="cuda", dtype=fn.torch_dtype)
    dense = torch.full((48, ld), float("nan"), device="cuda", dtype=fn.torch_dtype)
    fn(torch.rand((8, 32), device="cuda", dtype=fn.torch_dtype))
    L.cusadi_densify(fn.handle, 1, y.data_ptr(), ld, dense.data_ptr(), ld, n, torch.cuda.current_stream().cuda_stream)
    want = torch.zeros((48, n), device="cuda", dtype=fn.torch_dtype)
    for q, (r, c) in enumerate(ir.outputs[1].entries()):
        want[8 * r + c] = y[6 + q, :n]
    assert torch.equal(dense[:, :n], want)
    assert torch.all(torch.isnan(dense[:, n:]))
