"""sg_set_scales: one launch for the values and one per grid, and everything the
inner solvers read rescaled with them. A power of two scales every rounding
alike, so the solves of 4 A_0 are the solves of A_0 divided by 4, bit for bit:
the FP64 and FP32 block solvers (stencils, planes, coarse matrix), the clusters
and the stand-alone kernels (48-byte stencil records)."""
import numpy as np
import pytest

import sg_inputs as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("ne,clusters", [(2, True), (8, True), (16, False), (16, True), (64, False), (64, True), (128, False),
                                         (128, True)])
def test_scales(monkeypatch, ne, clusters, prec):
    import torch

    import paper_1205_1864_gb300 as L
    if not clusters:
        monkeypatch.setenv("SGHSC_NO_CLUSTER", "1")
    h = L.SGProblem.from_inputs(S.make_problem(ne, 1, 0.3, 0.5), 1)
    dt, code = (torch.float64, L.SG_F64) if prec == "fp64" else (torch.float32, L.SG_F32)
    B = torch.tensor(S.random_block(h.n, 5, seed=ne), dtype=dt, device="cuda")
    steps = 1 if ne == 2 else 3
    for nu in (1, 2):
        o = L.prec_opts(precision=code, inner_fixed_iters=steps, nu=nu)
        X = []
        for s in (1.0, 4.0):
            n0 = L._lib.LIB.sg_kernel_launches()
            L.sg_set_scales(h, np.array([s, s]))
            assert L._lib.LIB.sg_kernel_launches() - n0 == 1 + int(np.log2(ne))
            X.append(L.sg_inner_solve(h, B, o)[0])
        assert bool(torch.isfinite(X[0]).all()) and torch.equal(X[0], 4.0 * X[1])
