"""Register caps of the one-thread kernels by the program's live values, read
off the generated source: none for small programs, 128 where 129 to 168 registers
would leave room for 12 warps only, 255 where the values exceed a thread's
registers; a caller's own cap stands."""
import re

import pytest

from paper_2408_09662_gb300 import programs
from paper_2408_09662_gb300.api import Function


def min_blocks(fn):
    m = re.search(r"__launch_bounds__\((\d+)(?:, (\d+))?\) cs_fwd", fn.source())
    return int(m.group(1)), int(m.group(2) or 0)


@pytest.mark.parametrize("make,dtype,opts,want", [
    (programs.cartpole_rk4, "f32", {}, (128, 0)),                      # 59 live values
    (programs.cartpole_rk4, "f64", {}, (128, 4)),                      # 118 registers of values
    (programs.cartpole_rk4, "f64", {"block": 64}, (64, 8)),
    (lambda: programs.ldlt_spd_solve(22), "f64", {}, (128, 2)),        # 554
    (programs.cartpole_rk4, "f64", {"maxrregcount": 64}, (128, 8)),
], ids=["none", "128", "128-block64", "255", "callers"])
def test_register_cap_rule(make, dtype, opts, want):
    assert min_blocks(Function(make(), dtype=dtype, cache_dir=None, **opts)) == want
