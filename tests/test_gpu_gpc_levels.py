"""sg_level_apply on a gPC coefficient: its level products reach every lower
level, more columns than the two blocks of the call hold. Levels 0 and 1 are the
adjacent pair that has no other; any other pair is refused."""
import numpy as np
import pytest

import sg_inputs as S
from oracle import chaos, sg_operator as so
from tests.gpu_common import TOL32, TOL64

pytestmark = pytest.mark.gpu


def test_level_products():
    import torch

    import paper_1205_1864_gb300 as L
    M, p = 2, 3
    prob = S.make_lognormal_problem(8, M, 1.0, 0.5, 2 * p)
    h = L.SGProblem.from_inputs(prob, p)
    A, G = so.kl_matrices(prob.rowptr, prob.colidx, prob.vals), chaos.gpc_g_matrices(M, p, 2 * p)
    off = h.off
    for dt, tol in ((torch.float64, TOL64), (torch.float32, TOL32)):
        for lo in range(p + 1):
            for li in (lo - 1, lo + 1):
                if not 0 <= li <= p:
                    continue
                X = S.random_block(prob.n, off[li + 1] - off[li], seed=li)
                B = S.random_block(prob.n, off[lo + 1] - off[lo], seed=9 + lo)
                Xt, Bt = torch.tensor(X, dtype=dt, device="cuda"), torch.tensor(B, dtype=dt, device="cuda")
                if max(lo, li) > 1:
                    with pytest.raises(RuntimeError, match="lower levels"):
                        L.sg_level_apply(h, lo, li, Xt, Bt)
                    continue
                Y = L.sg_level_apply(h, lo, li, Xt, Bt).double().cpu().numpy()
                X, B = Xt.double().cpu().numpy(), Bt.double().cpu().numpy()
                ref = B - so.level_apply(A, G, off, lo, li, X)
                bound = np.abs(B) + so.level_apply([abs(a) for a in A], [abs(g) for g in G], off, lo, li, np.abs(X))
                assert np.all(np.abs(Y - ref) <= tol * bound)
