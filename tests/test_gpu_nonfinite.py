"""An infinity or a NaN in one entry of the input reaches the outputs that couple
to it and no other, in every form of the SG and level products: FP64, FP32 (the
row kernel with one to eight rows a block and the narrower general one) and
double-float. The couplings of a warp's outputs are padded to the longest list;
the padding must not read a sum that the entry is part of."""
import numpy as np
import pytest
import scipy.sparse as sp

import sg_inputs as S
from oracle import chaos, sg_operator as so

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,p", [(2, 2), (3, 3), (5, 4), (6, 4), (8, 4), (10, 4)])   # P = 6, 20, 126, 210, 495, 1001
def test_products(M, p):
    import torch

    import paper_1205_1864_gb300 as L
    prob = S.make_problem(16, M, 0.3, 0.5)
    h = L.SGProblem.from_inputs(prob, p)
    n, off = h.n, h.off
    pattern = sp.csr_matrix((np.ones(len(prob.colidx)), prob.colidx, prob.rowptr), shape=(n, n))
    A, G = [pattern] * (M + 1), [abs(g) for g in chaos.g_matrices(M, p)]
    row, f32, f64 = 100, torch.float32, torch.float64

    def block(w, dtype, col, value):
        X = torch.tensor(S.random_block(n, w, seed=w), dtype=dtype, device="cuda")
        X[row, col] = value
        hit = np.zeros((n, w))
        hit[row, col] = 1.0
        return X, hit

    def same(Y, hit):
        return np.array_equal(~torch.isfinite(Y).cpu().numpy(), hit > 0)

    for value in (float("inf"), float("nan")):
        for col in (0, 1, h.P - 1):
            for dtype, df in ((f64, False), (f32, False), (f32, True)):
                U, hit = block(h.P, dtype, col, value)
                assert same(L.sg_apply(h, U, df64=df), so.sg_apply(A, G, hit)), (col, dtype, df)
        for lo, li in [(l - 1, l) for l in range(1, p + 1)] + [(l, l - 1) for l in range(1, p + 1)]:
            wi, wo = off[li + 1] - off[li], off[lo + 1] - off[lo]
            for col in {0, wi - 1}:
                for dtype, ydtype in ((f64, f64), (f32, f32), (f32, f64)):
                    X, hit = block(wi, dtype, col, value)
                    Y = L.sg_level_apply(h, lo, li, X, torch.ones(n, wo, dtype=ydtype, device="cuda"), df64=ydtype != dtype)
                    assert same(Y, so.level_apply(A, G, off, lo, li, hit)), (lo, li, col, dtype, ydtype)
