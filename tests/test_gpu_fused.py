"""The two-pass V-cycle (csrc/mg_fused.cuh) against the FP64 oracle: one and
several strips, partial last strips and column chunks, the narrow and the wide
form on either side of the rule that picks them, a chunk of finished columns.
The cycle does the same steps as the kernel-per-sweep forms, so the bars are
theirs: 2e-5 of a column's largest entry for one cycle, 1e-4 for two
preconditioned CG steps."""
import numpy as np
import pytest

import sg_inputs as S
from oracle import gmg, krylov
from tests.gpu_common import problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import paper_1205_1864_gb300 as L
    return L


@pytest.mark.parametrize("ne,w", [(64, 1), (64, 24), (128, 3), (128, 25), (128, 290), (256, 9), (256, 71),
                                  (512, 33), (512, 41)])
def test_vcycle(lib, ne, w):
    import torch
    prob, A, _, _ = problem(ne, 1, 1)
    h = lib.SGProblem.from_inputs(prob, 1)
    B = S.random_block(prob.n, w, seed=ne + w).astype(np.float32)
    X = lib.sg_vcycle_apply(h, torch.tensor(B, device="cuda"), lib.prec_opts()).double().cpu().numpy()
    cols = sorted({0, w // 2, w - 1, min(32, w - 1)})
    ref = gmg.vcycle(gmg.hierarchy(A[0], ne), B[:, cols].astype(np.float64), nu=2, omega=0.8)
    assert np.all(np.abs(X[:, cols] - ref) <= 2e-5 * np.abs(ref).max(axis=0, keepdims=True))


@pytest.mark.parametrize("ne,w", [(256, 20), (256, 130)])
def test_inner_solve_with_finished_columns(lib, ne, w):
    import torch
    prob, A, _, _ = problem(ne, 1, 1)
    h = lib.SGProblem.from_inputs(prob, 1)
    lv = gmg.hierarchy(A[0], ne)
    B = S.random_block(prob.n, w, seed=w).astype(np.float32)
    B[:, w // 4: w // 4 + (32 if w > 64 else 8)] = 0.0
    B[:, 32:64] = 0.0
    X, it = lib.sg_inner_solve(h, torch.tensor(B, device="cuda"), lib.prec_opts(inner_fixed_iters=2))
    X = X.double().cpu().numpy()
    zero = ~B.any(axis=0)
    assert np.all(X[:, zero] == 0.0) and np.all(it[zero] == 0) and np.all(it[~zero] == 2)
    cols = np.flatnonzero(~zero)[[0, -1]]
    ref = krylov.pcg_columns(lambda v: A[0] @ v, B[:, cols].astype(np.float64), lambda r: gmg.vcycle(lv, r), tol=0.0,
                             maxit=2, fixed_iters=2)[0]
    assert np.all(np.abs(X[:, cols] - ref) <= 1e-4 * np.abs(ref).max(axis=0, keepdims=True))


@pytest.mark.parametrize("ne,w,prec", [(128, 1, "fp64"), (128, 20, "fp64"), (128, 131, "fp64"), (256, 3, "fp32"),
                                       (256, 230, "fp32"), (128, 701, "fp32")])
def test_direction_update_by_rows(lib, ne, w, prec):
    """The inner CG's p, q = A_0 p kernel walking down its strips (and node by
    node for FP64 shares of less than two rows: 127 x 127 nodes, 20 columns):
    shares that begin and end inside a strip, one block's and several strips'.
    Three steps against the oracle: 1e-10 in FP64, 1e-4 in FP32 (the bars of the
    solvers at these sizes)."""
    import torch
    prob, A, _, _ = problem(ne, 1, 1)
    h = lib.SGProblem.from_inputs(prob, 1)
    code, dt, tol = ((lib.SG_F64, torch.float64, 1e-10) if prec == "fp64" else (lib.SG_F32, torch.float32, 1e-4))
    B = S.random_block(prob.n, w, seed=w).astype(np.float64 if prec == "fp64" else np.float32)
    X, it = lib.sg_inner_solve(h, torch.tensor(B, dtype=dt, device="cuda"),
                               lib.prec_opts(precision=code, inner_fixed_iters=3))
    cols = sorted({0, w // 2, w - 1})
    lv = gmg.hierarchy(A[0], ne)
    ref = krylov.pcg_columns(lambda v: A[0] @ v, B[:, cols].astype(np.float64), lambda r: gmg.vcycle(lv, r), tol=0.0,
                             maxit=3, fixed_iters=3)[0]
    assert list(it) == [3] * w
    assert np.abs(X.double().cpu().numpy()[:, cols] - ref).max() <= tol * np.abs(ref).max()
