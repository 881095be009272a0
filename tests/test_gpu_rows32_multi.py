"""The FP32 row kernel with several rows per block (eight, four and two, full
and level products; the counts rows32_pick gives) on ragged CSR rows and a row
count that leaves the last block partly empty, against the oracle: within m u
sum|terms|, m the longest chain of roundings (23 nonzeros of the longest row
plus the 2M + 1 couplings of an output, the difference and the store)."""
import numpy as np
import pytest

import sg_inputs as S
from oracle import chaos, sg_operator as so
from tests.gpu_common import abs_bound, random_csr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,p", [(2, 4), (5, 4), (6, 4), (10, 3), (7, 4)])   # P = 15, 126, 210, 286, 330
def test_products(M, p):
    import torch

    import paper_1205_1864_gb300 as L
    n = 205
    rowptr, colidx = random_csr(n, seed=M, max_row=23)
    vals = np.random.default_rng(p).uniform(-1, 1, size=(len(colidx), M + 1))
    h = L.SGProblem(0, 0, M, p, rowptr, colidx, vals)
    A, G = so.kl_matrices(rowptr, colidx, vals), chaos.g_matrices(M, p)
    _, off = chaos.multi_indices(M, p)
    aA, aG = [abs(a) for a in A], [abs(g) for g in G]
    u = (23 + 2 * M + 3) * 2.0 ** -24
    U = S.random_block(n, h.P, seed=3).astype(np.float32)
    Y = L.sg_apply(h, torch.tensor(U, device="cuda")).double().cpu().numpy()
    U = U.astype(np.float64)
    assert np.all(np.abs(Y - so.sg_apply(A, G, U)) <= u * abs_bound(A, G, U) + 1e-300)
    for l in range(1, p + 1):
        for lo, li in ((l - 1, l), (l, l - 1)):
            X = S.random_block(n, off[li + 1] - off[li], seed=lo + 10 * li).astype(np.float32)
            B = S.random_block(n, off[lo + 1] - off[lo], seed=5 + lo).astype(np.float32)
            Y = L.sg_level_apply(h, lo, li, torch.tensor(X, device="cuda"), torch.tensor(B, device="cuda"))
            X, B = X.astype(np.float64), B.astype(np.float64)
            bound = np.abs(B) + so.level_apply(aA, aG, off, lo, li, np.abs(X))
            err = np.abs(Y.double().cpu().numpy() - (B - so.level_apply(A, G, off, lo, li, X)))
            assert np.all(err <= u * bound + 1e-300), (lo, li)
