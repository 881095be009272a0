"""The block-per-column inner solver of small grids (csrc/inner_block.cu)
against the oracle's PCG and against the stand-alone kernels
(``SGHSC_NO_BLOCK=1`` at ``sg_setup``): the grid sizes where its split over
the blocks of a cluster, its nodes per thread or its number of grids change.

Tolerances. Both sides run the same steps; a step's rounding differs by the
order of sums. After k steps the iterates differ by about k u times the
condition of the preconditioned matrix (below 2 with the V-cycle, below the
number of nodes with the diagonal), relative to the largest entry: 1e-11 in
FP64 (u = 1.1e-16, 4 steps, up to 8281 nodes: 4e-12), 2e-3 in FP32 with the
diagonal and 2e-5 with the V-cycle (1e-4 on 63 x 63 nodes, the bar of the other
solvers there: A_0 itself is rounded, which its small eigenvalues feel)."""
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


def _handles(lib, monkeypatch, ne):
    prob, A, _, _ = problem(ne, 1, 1)
    h = lib.SGProblem.from_inputs(prob, 1)
    monkeypatch.setenv("SGHSC_NO_BLOCK", "1")
    h0 = lib.SGProblem.from_inputs(prob, 1)
    return prob, A, h, h0


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("m0,ne,w", [("diag", 2, 1), ("diag", 5, 3), ("diag", 10, 40), ("diag", 17, 7), ("diag", 30, 1),
                                     ("diag", 30, 35), ("diag", 33, 160), ("diag", 64, 2), ("diag", 91, 5),
                                     ("diag", 92, 3), ("vcycle", 2, 2), ("vcycle", 4, 3), ("vcycle", 8, 1),
                                     ("vcycle", 16, 20), ("vcycle", 32, 155), ("vcycle", 64, 3), ("vcycle", 64, 160)])
def test_block_solver_matches_oracle(lib, monkeypatch, m0, ne, w, prec):
    import torch
    dt, code = (torch.float64, lib.SG_F64) if prec == "fp64" else (torch.float32, lib.SG_F32)
    if prec == "fp32" and m0 == "vcycle":
        monkeypatch.setenv("SGHSC_NO_CLUSTER", "1")
    prob, A, h, h0 = _handles(lib, monkeypatch, ne)
    B = S.random_block(prob.n, w, seed=ne + w)
    if w > 2:
        B[:, 1] = 0.0   # a zero column is done at entry
    B = B.astype(np.float64 if prec == "fp64" else np.float32)
    Bt = torch.tensor(B, dtype=dt, device="cuda")
    if m0 == "diag":
        d = A[0].diagonal()
        pre = lambda r: r / d   # noqa: E731
        kind = lib.SG_M0_DIAG
    else:
        lv = gmg.hierarchy(A[0], ne)
        pre = lambda r: gmg.vcycle(lv, r)   # noqa: E731
        kind = lib.SG_M0_VCYCLE
    # no more steps than unknowns: past convergence the steps divide rounding errors by each other
    steps = {2: 1}.get(ne, 4)
    o = lib.prec_opts(precision=code, m0=kind, inner_fixed_iters=steps)
    X, it = lib.sg_inner_solve(h, Bt, o)
    ref = krylov.pcg_columns(lambda v: A[0] @ v, B.astype(np.float64), pre, tol=0.0, maxit=steps, fixed_iters=steps)[0]
    tol = 1e-11 if prec == "fp64" else (2e-3 if m0 == "diag" else 1e-4 if ne == 64 else 2e-5)
    assert np.abs(X.double().cpu().numpy() - ref).max() <= tol * np.abs(ref).max()
    assert all(it[c] == (0 if w > 2 and c == 1 else steps) for c in range(w))
    # to a tolerance: the same counts as the stand-alone kernels
    o = lib.prec_opts(precision=code, m0=kind, inner_tol=1e-3, inner_maxit=1000)
    X, it = lib.sg_inner_solve(h, Bt, o)
    X0, it0 = lib.sg_inner_solve(h0, Bt, o)
    if prec == "fp64":
        assert np.array_equal(it, it0)
        assert float((X - X0).abs().max()) <= 1e-9 * float(X0.abs().max())
    else:   # a residual at the threshold may stop one step apart
        assert int(np.abs(it - it0).max()) <= 1


@pytest.mark.parametrize("ne,prec,tol", [(16, "fp64", 1e-13), (32, "fp64", 1e-13), (16, "fp32", 1e-5), (32, "fp32", 1e-5),
                                         (64, "fp32", 1e-5)])
def test_coarse_matrix_equals_the_smoothed_cycle(lib, monkeypatch, ne, prec, tol):
    """The matrix of the grids from 7 x 7 down (the default smoothing) against
    the grid-by-grid cycle, which a damping one rounding away still takes, also
    after a change of scale. One step: the two differ by the rounding of some 60
    operations a node, 1e-14 in FP64 and 4e-6 in FP32."""
    import torch
    prob, A, h, _ = _handles(lib, monkeypatch, ne)
    dt, code = (torch.float64, lib.SG_F64) if prec == "fp64" else (torch.float32, lib.SG_F32)
    B = torch.tensor(S.random_block(prob.n, 5, seed=ne), dtype=dt, device="cuda")
    for scale in (1.0, 3.0):
        lib.sg_set_scales(h, np.full(2, scale))
        X = [lib.sg_inner_solve(h, B, lib.prec_opts(precision=code, inner_fixed_iters=1, omega=om))[0]
             for om in (0.8, float(np.nextafter(0.8, 1)))]
        assert float((X[0] - X[1]).abs().max()) <= tol * float(X[1].abs().max())
        ref = krylov.pcg_columns(lambda v: scale * (A[0] @ v), B.double().cpu().numpy(),
                                 lambda r: gmg.vcycle(gmg.hierarchy(scale * A[0], ne), r), tol=0.0, maxit=1,
                                 fixed_iters=1)[0]
        assert np.abs(X[0].double().cpu().numpy() - ref).max() <= (1e-12 if prec == "fp64" else 1e-4) * np.abs(ref).max()


@pytest.mark.parametrize("w", [5, 40, 100])
def test_coarse_matrix_on_clusters(lib, w):
    """The same in the cluster solvers (127 x 127 nodes; clusters of 16 and 8
    blocks, finest grid in global memory): one step, 1e-5."""
    import torch
    prob, A, _, _ = problem(128, 1, 1)
    h = lib.SGProblem.from_inputs(prob, 1)
    B = torch.tensor(S.random_block(prob.n, w, seed=w), dtype=torch.float32, device="cuda")
    X = [lib.sg_inner_solve(h, B, lib.prec_opts(precision=lib.SG_F32, inner_fixed_iters=1, omega=om))[0]
         for om in (0.8, float(np.nextafter(0.8, 1)))]
    assert float((X[0] - X[1]).abs().max()) <= 1e-5 * float(X[1].abs().max())
