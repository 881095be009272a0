"""The order in which the inner solvers of small grids are taken, and the
cluster solvers on the grids that the block-per-column solver holds too
(``SGHSC_NO_BLOCK=1`` at ``sg_setup`` leaves only them), against the oracle.

Tolerance of the solves: three FP32 steps, 1e-4 of a column's largest entry,
the bar of the cluster solvers' own tests (about 60 roundings a node and step,
u = 6e-8, 1e-5, times the spread of A_0's eigenvalues that the V-cycle leaves)."""
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


@pytest.mark.parametrize("ne", [16, 32, 64, 128])
def test_order_of_the_solvers(lib, monkeypatch, ne):
    """Where the block solver holds the grid (up to 63 x 63 nodes) it takes the
    preconditioners' own batches (degree levels of 1, 3 and 6 columns, 4 and
    10 in all)
    and those too wide for the on-chip clusters (path 0); any other batch takes
    the on-chip cluster solver that holds it."""
    prob, _, _, _ = problem(ne, 3, 2)
    h = lib.SGProblem.from_inputs(prob, 2)
    monkeypatch.setenv("SGHSC_NO_BLOCK", "1")
    c = lib.SGProblem.from_inputs(prob, 2)
    assert c.inner_path(1) in (1, 3) and c.inner_path(60) == 1
    for w in (1, 3, 4, 6, 10):
        assert h.inner_path(w) == (c.inner_path(w) if ne == 128 else 0), w
    for w in (2, 5, 7, 11, 20, 28, 32, 60):
        assert h.inner_path(w) == c.inner_path(w) != 0, w
    for w in (61, 100, 144):
        assert c.inner_path(w) == 2 and h.inner_path(w) == (2 if ne == 128 else 0), w
    assert h.inner_path(400) == 0 and h.inner_path(5, lib.SG_F64) == 0


def _cluster_and_plain(lib, monkeypatch, ne, M, p):
    """Handles whose inner solves run on the clusters, and on the stand-alone kernels."""
    prob, A, G, off = problem(ne, M, p)
    monkeypatch.setenv("SGHSC_NO_BLOCK", "1")
    c = lib.SGProblem.from_inputs(prob, p)
    monkeypatch.setenv("SGHSC_NO_CLUSTER", "1")
    return prob, A, G, off, c, lib.SGProblem.from_inputs(prob, p)


@pytest.mark.parametrize("ne,M,p", [(16, 3, 3), (32, 3, 3), (64, 2, 2)])
def test_algorithm_1_on_clusters(lib, monkeypatch, ne, M, p):
    """Algorithm 1 with FP32 inner solves of four steps on the clusters: the
    oracle, and the stand-alone kernels, within 2e-5 of the largest entry (1e-4
    on 63 x 63 nodes), the bars of these solvers at fixed step counts."""
    import torch
    from oracle import hsc
    prob, A, G, off, c, s = _cluster_and_plain(lib, monkeypatch, ne, M, p)
    widths = [off[l + 1] - off[l] for l in range(p + 1)]
    assert all(c.inner_path(w) in (1, 3) for w in widths) and all(s.inner_path(w) == 0 for w in widths)
    lv = gmg.hierarchy(A[0], ne)
    R = S.random_block(prob.n, c.P, seed=42)
    o = lib.prec_opts(precision=lib.SG_F32, inner_fixed_iters=4)
    Z, Z0 = (lib.hsc_precond_apply(h, torch.tensor(R, device="cuda"), o).cpu().numpy() for h in (c, s))

    def dsolve(l, X):
        return krylov.pcg_columns(lambda v: A[0] @ v, X, lambda r: gmg.vcycle(lv, r), tol=0.0, maxit=4,
                                  fixed_iters=4)[0]
    ref = hsc.hsc_apply(A, G, off, R, dsolve=dsolve)
    tol = (1e-4 if ne == 64 else 2e-5) * np.abs(ref).max()
    assert np.abs(Z - ref).max() <= tol and np.abs(Z - Z0).max() <= tol


def test_solve_on_clusters(lib, monkeypatch):
    """The mixed solve with its inner solves on the clusters reaches 1e-8 and
    the oracle's direct solution."""
    import torch
    from oracle import sg_operator as so
    prob, A, G, _, c, _ = _cluster_and_plain(lib, monkeypatch, 16, 3, 3)
    F = S.make_rhs(prob, 3)
    ref = so.direct_solve(A, G, F)
    U, st = lib.sg_solve(c, torch.tensor(F, device="cuda"),
                         lib.solve_opts(lib.prec_opts(precision=lib.SG_F32), precond=lib.SG_PREC_HSC, tol=1e-8))
    assert st.true_rel_res <= 1e-8 * 1.01
    assert np.abs(U.cpu().numpy() - ref).max() <= 1e-6 * np.abs(ref).max()


@pytest.mark.parametrize("nu,omega", [(2, 0.8), (1, 0.8), (3, 0.7)])
@pytest.mark.parametrize("ne,w,path", [(16, 7, 1), (16, 90, 2), (32, 13, 3), (32, 41, 1), (32, 90, 2), (64, 9, 3),
                                       (64, 41, 1), (64, 90, 2)])
def test_cluster_solvers_match_oracle(lib, monkeypatch, ne, w, path, nu, omega):
    import torch
    prob, A, _, _ = problem(ne, 1, 1)
    monkeypatch.setenv("SGHSC_NO_BLOCK", "1")
    h = lib.SGProblem.from_inputs(prob, 1)
    assert h.inner_path(w) == path
    lv = gmg.hierarchy(A[0], ne)
    B = S.random_block(prob.n, w, seed=21 + ne + w).astype(np.float32)
    B[:, 2] = 0.0
    X, it = lib.sg_inner_solve(h, torch.tensor(B, device="cuda"), lib.prec_opts(inner_fixed_iters=3, nu=nu, omega=omega))
    ref, it_ref = krylov.pcg_columns(lambda v: A[0] @ v, B.astype(np.float64),
                                     lambda r: gmg.vcycle(lv, r, nu=nu, omega=omega), tol=0.0, maxit=3, fixed_iters=3)
    assert list(it) == list(it_ref)
    X = X.double().cpu().numpy()
    assert np.all(np.abs(X - ref) <= 1e-4 * (np.abs(ref).max(axis=0, keepdims=True) + 1e-300))
    assert np.all(X[:, 2] == 0.0)


@pytest.mark.parametrize("ne", [16, 32, 64])
def test_coarse_matrix_in_the_fp32_block_solver(lib, monkeypatch, ne):
    """The block solver alone (SGHSC_NO_CLUSTER=1): the 7 x 7 grid and those
    below as one matrix (the default smoothing) against the grid-by-grid cycle
    of a damping one rounding away. One step, some 60 roundings a node: 1e-5."""
    import torch
    prob, _, _, _ = problem(ne, 1, 1)
    monkeypatch.setenv("SGHSC_NO_CLUSTER", "1")
    h = lib.SGProblem.from_inputs(prob, 1)
    B = torch.tensor(S.random_block(prob.n, 5, seed=ne), dtype=torch.float32, device="cuda")
    X = [lib.sg_inner_solve(h, B, lib.prec_opts(precision=lib.SG_F32, inner_fixed_iters=1, omega=om))[0]
         for om in (0.8, float(np.nextafter(0.8, 1)))]
    assert float((X[0] - X[1]).abs().max()) <= 1e-5 * float(X[1].abs().max())


@pytest.mark.parametrize("ne,w,prec", [(16, 6, "fp64"), (32, 5, "fp64"), (16, 6, "fp32"), (32, 5, "fp32"), (64, 7, "fp32")])
@pytest.mark.parametrize("nu,omega", [(1, 0.8), (3, 0.7), (2, 0.6)])
def test_block_solver_with_other_smoothing(lib, monkeypatch, ne, w, prec, nu, omega):
    """The block solver alone, grid by grid (no coarse matrix), odd and even
    numbers of sweeps: three steps against the oracle, 1e-11 of the largest entry
    in FP64, 1e-4 in FP32."""
    import torch
    prob, A, _, _ = problem(ne, 1, 1)
    monkeypatch.setenv("SGHSC_NO_CLUSTER", "1")
    h = lib.SGProblem.from_inputs(prob, 1)
    code, dt, tol = (lib.SG_F64, np.float64, 1e-11) if prec == "fp64" else (lib.SG_F32, np.float32, 1e-4)
    lv = gmg.hierarchy(A[0], ne)
    B = S.random_block(prob.n, w, seed=ne + nu).astype(dt)
    n0 = lib._lib.LIB.sg_kernel_launches()
    X, it = lib.sg_inner_solve(h, torch.tensor(B, device="cuda"),
                               lib.prec_opts(precision=code, inner_fixed_iters=3, nu=nu, omega=omega))
    assert lib._lib.LIB.sg_kernel_launches() - n0 == 1
    ref = krylov.pcg_columns(lambda v: A[0] @ v, B.astype(np.float64), lambda r: gmg.vcycle(lv, r, nu=nu, omega=omega),
                             tol=0.0, maxit=3, fixed_iters=3)[0]
    assert list(it) == [3] * w
    assert np.abs(X.double().cpu().numpy() - ref).max() <= tol * np.abs(ref).max()
