"""The inner solver's workspace grows with the batch: one more group of four
columns takes no more than its share (28 vectors' worth of pieces of 16 bytes a
node; a tenth allows for the allocator's granularity)."""
import pytest

import sg_inputs as S

pytestmark = pytest.mark.gpu


def test_workspace_follows_the_width(monkeypatch):
    import torch

    import paper_1205_1864_gb300 as L
    prob = S.make_problem(256, 1, 0.3, 0.5)

    def taken(w):
        h = L.SGProblem.from_inputs(prob, 1)
        B = torch.ones(h.n, w, dtype=torch.float32, device="cuda")
        torch.empty_like(B)   # (the output's block, kept by the caching allocator)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        L.sg_inner_solve(h, B, L.prec_opts(inner_fixed_iters=1))
        torch.cuda.synchronize()
        return free - torch.cuda.mem_get_info()[0]

    taken(96)   # what the first call of the process loads
    a, b = taken(96), taken(97)
    assert a > 0 and b <= 1.1 * a
