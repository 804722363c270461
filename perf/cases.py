"""Performance cases of the engine: what a program that uses it has it do.

Every case loads one program (or a batch of programs) once, as a user does, and
then evaluates it through the public API on device buffers of its own.  Sizes
are those of the repository's benchmark and tests (C1 cart-pole, C2 random
program, C3 MPC, C4 rollout, the LDL^T family, the sparse Jacobian), with odd
instance counts where a user's batch would have them.

The exact values come from a plain sequential evaluation of the program's
instruction list with torch in 64 bits on the CPU (torch.autograd for
gradients).
"""
import functools
import math

import torch

from paper_2408_09662_gb300 import programs
from paper_2408_09662_gb300.api import Batch, Function
from paper_2408_09662_gb300.ir import Op
from paper_2408_09662_gb300.rollout import GraphRollout, StepProgram

# Programs of the batched launch: (ops drawn, program seed, share of the instances)
BATCH = ((300, 100, 1.0), (1000, 101, 1.0), (2500, 102, 0.5), (5000, 103, 0.25))


def listed():
    return [
        # one control tick of a small simulation: latency and launches count
        {"name": "cartpole_f64_small", "kind": "cartpole", "dtype": "f64", "n": 1000},
        # the step with its Jacobian over the benchmark's batch
        {"name": "cartpole_f64", "kind": "cartpole", "dtype": "f64", "n": 65536},
        # a learning-sized batch in single precision, an odd instance count
        {"name": "cartpole_f32_large", "kind": "cartpole", "dtype": "f32", "n": 1000003},
        # the headline workload: a 20,000-op program, one thread per instance
        {"name": "random20k_f64", "kind": "random", "dtype": "f64", "n": 65536, "ops": 20000, "ways": 0},
        # the same long program on few instances, 8 warps per group of 32 instances
        {"name": "random20k_f64_few", "kind": "random", "dtype": "f64", "n": 4096, "ops": 20000, "ways": 8},
        # closed-form MPC as it is deployed: single precision with double pivots
        {"name": "mpc_mixed", "kind": "mpc", "dtype": "mixed", "n": 16384},
        # closed-loop LQR with the Riccati solve inside, the region-of-attraction batch
        {"name": "lqr_f64", "kind": "lqr", "dtype": "f64", "n": 10000},
        # gradient of one step for states and a shared gain
        {"name": "srb_adjoint_f64", "kind": "adjoint", "dtype": "f64", "n": 65536},
        # a training step: 50-step differentiable rollout and its reverse pass
        {"name": "srb_rollout_f32", "kind": "rollout", "dtype": "f32", "n": 4096, "steps": 50},
        # a program evaluated without compiling it: LDL^T solve of 47 unknowns
        {"name": "ldlt47_interp_f64", "kind": "ldlt", "dtype": "f64", "n": 16384, "order": 47},
        # several programs of uneven length in one launch
        {"name": "batch_f32", "kind": "batch", "dtype": "f32", "n": 65536},
        # a sparse Jacobian for a large batch, handed on as dense blocks
        {"name": "jacobian_dense_f64", "kind": "jacobian", "dtype": "f64", "n": 1000003},
    ]


def _size(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return n if rng.random() < 0.3 else n | 1


def draw(rng):
    kind = rng.choice(["cartpole", "cartpole", "random", "random", "mpc", "lqr", "adjoint", "rollout", "ldlt",
                       "batch", "jacobian"])
    both = rng.choice(["f64", "f32"])
    if kind == "cartpole":
        return {"kind": kind, "dtype": both, "n": _size(rng, 33, 1000003)}
    if kind == "random":
        ops = _size(rng, 300, 4000)
        ways = rng.choice([0, 0, 4, 8])
        return {"kind": kind, "dtype": "f64", "n": _size(rng, 33, 8192 if ways else 65536), "ops": ops, "ways": ways}
    if kind == "mpc":
        return {"kind": kind, "dtype": rng.choice(["mixed", "mixed", "f64"]), "n": _size(rng, 256, 16384)}
    if kind == "lqr":
        return {"kind": kind, "dtype": "f64", "n": _size(rng, 100, 16384)}
    if kind == "adjoint":
        return {"kind": kind, "dtype": both, "n": _size(rng, 500, 65536)}
    if kind == "rollout":
        return {"kind": kind, "dtype": both, "n": _size(rng, 64, 4096), "steps": rng.choice([10, 23, 50])}
    if kind == "ldlt":
        return {"kind": kind, "dtype": "f64", "n": _size(rng, 256, 16384), "order": rng.choice([10, 22, 47])}
    if kind == "batch":
        return {"kind": kind, "dtype": "f32", "n": _size(rng, 1000, 65536)}
    return {"kind": kind, "dtype": both, "n": _size(rng, 1000, 1000003)}


# ---------------------------------------------------------------------------
# programs and the functions loaded from them (kept, as a user keeps them)
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _program(kind, size=0, seed=0):
    if kind == "cartpole":
        return programs.cartpole_rk4()
    if kind == "random":
        return programs.random_program(size, seed=seed)
    if kind == "mpc":
        return programs.quadrotor_mpc()
    if kind == "lqr":
        return programs.quadrotor_lqr_step()
    if kind in ("adjoint", "rollout"):
        return programs.srb_step()
    if kind == "ldlt":
        return programs.ldlt_spd_solve(size)
    return programs.quadrotor_step_sparse_jacobian()


def _program_of(case):
    return _program(case["kind"], case.get("ops", case.get("order", 0)))


def _batch_of(case):
    """(program, instances) of each member of a batch case."""
    return [(_program("random", ops, seed), max(33, int(case["n"] * share))) for ops, seed, share in BATCH]


@functools.lru_cache(maxsize=None)
def _function(kind, size, dtype, ways, path, adjoint):
    return Function(_program(kind, size), dtype=dtype, path=path, ways=ways, adjoint=adjoint)


def _function_of(case):
    kind = case["kind"]
    return _function(kind, case.get("ops", case.get("order", 0)), case["dtype"], case.get("ways", 0),
                     "interp" if kind == "ldlt" else "auto", 1 if kind in ("adjoint", "rollout") else 0)


@functools.lru_cache(maxsize=None)
def _batch(sizes, dtype):
    return Batch([_program("random", ops, seed) for ops, seed, _ in BATCH], list(sizes), dtype=dtype)


@functools.lru_cache(maxsize=None)
def _rollout(dtype, n, steps):
    return GraphRollout(StepProgram(_function("rollout", 0, dtype, 0, "auto", 1), 144, 12), n, steps)


# ---------------------------------------------------------------------------
# inputs: drawn on the GPU from the seed, rounded to the buffers' type
# ---------------------------------------------------------------------------
def _inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, kind = case["n"], case["kind"]
    dt = torch.float64 if case["dtype"] == "f64" else torch.float32

    def uniform(rows, lo, hi, cols=n):
        return torch.rand((rows, cols), generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo

    def normal(rows, cols=n):
        return torch.randn((rows, cols), generator=g, device="cuda", dtype=torch.float64)

    if kind == "cartpole":
        x = [uniform(4, -1, 1), uniform(1, -10, 10)]
    elif kind == "random":
        x = [normal(64)]
    elif kind == "mpc":
        x = [uniform(6, -0.5, 0.5), uniform(2, -1, 1)]
    elif kind == "lqr":
        x = [uniform(6, -0.5, 0.5), uniform(1, 10, 20), uniform(1, 0.8, 1.2), uniform(1, 0.008, 0.012),
             uniform(6, 0.5, 10), uniform(1, 0.05, 0.5)]
    elif kind == "adjoint":
        gain = normal(144, 1) * 0.1
        return {"x": torch.cat([gain.expand(144, n), uniform(12, -0.1, 0.1), uniform(1, 0, 1)]).to(dt),
                "ybar": normal(13).to(dt)}
    elif kind == "rollout":
        return {"x0": uniform(12, -0.1, 0.1).to(dt), "K": (normal(1, 144)[0] * 0.1).to(dt)}
    elif kind == "ldlt":
        m = case["order"]
        a = torch.randn((n, m, m), generator=g, device="cuda", dtype=torch.float64)
        a = a @ a.transpose(1, 2) / m + torch.eye(m, device="cuda", dtype=torch.float64)
        i, j = torch.tril_indices(m, m, device="cuda")
        x = [a[:, i, j].T.contiguous(), normal(m)]
    elif kind == "batch":
        return {"xs": [normal(64, cols).to(dt) for _, cols in _batch_of(case)]}
    else:
        x = [uniform(6, -1, 1), uniform(2, 0, 10)]
    return {"x": torch.cat(x).to(dt)}


def prepare(case, seed):
    state = {"case": dict(case), **_inputs(case, seed)}
    if case["kind"] == "batch":
        state["f"] = _batch(tuple(cols for _, cols in _batch_of(case)), case["dtype"])
        state["outs"] = [torch.empty((p.nnz_out, cols), dtype=state["xs"][0].dtype, device="cuda")
                         for p, cols in _batch_of(case)]
    elif case["kind"] == "rollout":
        state["f"] = _rollout(case["dtype"], case["n"], case["steps"])
    else:
        state["f"] = _function_of(case)
        if case["kind"] == "adjoint":       # where the shared gain's gradient goes
            state["gain"] = torch.zeros(157, dtype=state["x"].dtype, device="cuda")
    return state


def run(state):
    f, kind = state["f"], state["case"]["kind"]
    if kind == "adjoint":
        return f.adjoint(state["x"], state["ybar"], shared_out=state["gain"])[144:], state["gain"][:144]
    if kind == "rollout":
        loss, last = f.forward(state["x0"], state["K"])
        gx, gk = f.backward()
        return {"loss": loss, "x": last, "gx": gx, "gK": gk}
    if kind == "batch":
        return f(state["xs"], state["outs"])
    y = f(state["x"])
    return (y, f.dense(y, 1)) if kind == "jacobian" else y


# ---------------------------------------------------------------------------
# what one pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    elt, n, kind = 8 if case["dtype"] == "f64" else 4, case["n"], case["kind"]
    if kind == "batch":
        members = _batch_of(case)
        return {"bytes": sum((p.nnz_in + p.nnz_out) * cols for p, cols in members) * elt,
                "flops": sum(p.count_ops() * cols for p, cols in members)}
    p = _program_of(case)
    ops = p.count_ops()
    if kind == "adjoint":      # states, seeds in; the states' adjoints and the gain's gradient out
        return {"bytes": (13 + 13 + 13) * n * elt + 2 * 144 * elt, "flops": 3 * ops * n}
    if kind == "rollout":      # the initial states in; last states, their gradient, loss, gain's gradient out
        return {"bytes": 3 * 12 * n * elt + 2 * 144 * elt, "flops": 4 * ops * n * case["steps"]}
    dense = 48 if kind == "jacobian" else 0
    return {"bytes": (p.nnz_in + p.nnz_out + dense) * n * elt, "flops": ops * n}


# ---------------------------------------------------------------------------
# the same outputs in 64 bits
# ---------------------------------------------------------------------------
_UNARY = {Op.NEG: torch.neg, Op.EXP: torch.exp, Op.SQ: torch.square, Op.SQRT: torch.sqrt, Op.SIN: torch.sin,
          Op.COS: torch.cos}
_BINARY = {Op.ADD: torch.add, Op.SUB: torch.sub, Op.MUL: torch.mul, Op.DIV: torch.div, Op.FMIN: torch.minimum,
           Op.FMAX: torch.maximum}


def _evaluate(p, rows):
    """The program's instructions in order on a list of float64 rows; the list of output rows."""
    w, out = [None] * p.n_work, [None] * p.nnz_out
    unary, binary = {int(k): f for k, f in _UNARY.items()}, {int(k): f for k, f in _BINARY.items()}
    zero = torch.zeros((), dtype=torch.float64)
    for i in p.instrs:
        if i.op in binary:
            w[i.out] = binary[i.op](w[i.a], w[i.b])
        elif i.op in unary:
            w[i.out] = unary[i.op](w[i.a])
        elif i.op == Op.INPUT:
            w[i.out] = rows[i.a]
        elif i.op == Op.OUTPUT:
            out[i.out] = w[i.a]
        elif i.op == Op.CONST:
            w[i.out] = zero + p.consts[i.a]
        elif i.op == Op.ASSIGN:
            w[i.out] = w[i.a]
        elif i.op == Op.FMA_CONST:
            w[i.out] = p.consts[i.c] * w[i.a] + w[i.b]
        else:
            raise ValueError(f"no 64-bit form of op {i.op}")
    return out


def _columns(out, n):
    return torch.stack([o.expand(n) for o in out])


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    s = {k: [t.double().cpu() for t in v] if isinstance(v, list) else v.double().cpu()
         for k, v in _inputs(case, seed).items()}
    if kind == "batch":
        return [_columns(_evaluate(p, list(x)), cols) for (p, cols), x in zip(_batch_of(case), s["xs"])]
    p = _program_of(case)
    if kind == "adjoint":
        gain, x = s["x"][:144, 0].clone().requires_grad_(), s["x"][144:].clone().requires_grad_()
        y = _columns(_evaluate(p, list(gain) + list(x)), n)
        y.backward(s["ybar"])
        return x.grad, gain.grad
    if kind == "rollout":
        gain, x0 = s["K"].requires_grad_(), s["x0"].requires_grad_()
        rows, k = list(x0) + [torch.zeros(n, dtype=torch.float64)], list(gain)
        for _ in range(case["steps"]):
            rows = _evaluate(p, k + rows)
        loss = rows[12].sum()
        loss.backward()
        return {"loss": loss.detach(), "x": torch.stack(rows[:12]).detach(), "gx": x0.grad, "gK": gain.grad}
    y = _columns(_evaluate(p, list(s["x"])), n)
    if kind != "jacobian":
        return y
    dense = torch.zeros((6, 8, n), dtype=torch.float64)
    for q, (r, c) in enumerate(p.outputs[1].entries()):
        dense[r, c] = y[6 + q]
    return y, dense
