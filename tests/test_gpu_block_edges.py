"""The diagonal block solver (csrc/inner_block.cu) where its split changes: the
largest square grid that a cluster of eight blocks holds (88 x 88 nodes: 256
threads a block, 64 partial sums a slot), one whose last block has fewer rows
(74 x 74: 10 rows, then 4), the wide batch that takes four blocks a column
because one does not hold it (63 x 63, 160 columns), and the first grid refused.
One launch per solve says that it ran.

Tolerances: four steps, k u times the condition (below the number of nodes):
1e-11 in FP64 (4 * 7921 * 1.1e-16 = 3.5e-12), 2e-3 in FP32."""
import numpy as np
import pytest

import sg_inputs as S
from oracle import krylov
from tests.gpu_common import problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("ne,w,taken", [(89, 3, True), (75, 2, True), (64, 160, True), (90, 3, False)])
def test_diagonal_block_solver(monkeypatch, ne, w, taken, prec):
    import torch

    import paper_1205_1864_gb300 as L
    prob, A, _, _ = problem(ne, 1, 1)
    h = L.SGProblem.from_inputs(prob, 1)
    monkeypatch.setenv("SGHSC_NO_BLOCK", "1")
    h0 = L.SGProblem.from_inputs(prob, 1)
    dt, code = (torch.float64, L.SG_F64) if prec == "fp64" else (torch.float32, L.SG_F32)
    B = S.random_block(prob.n, w, seed=ne + w).astype(np.float64 if prec == "fp64" else np.float32)
    B[:, 1] = 0.0
    Bt = torch.tensor(B, dtype=dt, device="cuda")
    n0 = L._lib.LIB.sg_kernel_launches()
    X, it = L.sg_inner_solve(h, Bt, L.prec_opts(precision=code, m0=L.SG_M0_DIAG, inner_fixed_iters=4))
    assert (L._lib.LIB.sg_kernel_launches() - n0 == 1) == taken
    d = A[0].diagonal()
    cols = sorted({0, 1, w - 1})
    ref = krylov.pcg_columns(lambda v: A[0] @ v, B[:, cols].astype(np.float64), lambda r: r / d, tol=0.0, maxit=4,
                             fixed_iters=4)[0]
    tol = 1e-11 if prec == "fp64" else 2e-3
    assert np.abs(X.double().cpu().numpy()[:, cols] - ref).max() <= tol * np.abs(ref).max()
    assert list(it) == [0 if c == 1 else 4 for c in range(w)]
    if prec == "fp64":   # to a tolerance: the counts of the stand-alone kernels
        o = L.prec_opts(precision=code, m0=L.SG_M0_DIAG, inner_tol=1e-3, inner_maxit=1000)
        assert np.array_equal(L.sg_inner_solve(h, Bt, o)[1], L.sg_inner_solve(h0, Bt, o)[1])
