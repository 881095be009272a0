"""Two host threads on handles of their own whose calls launch the same kernels
with different amounts of dynamic shared memory. The limit on it belongs to the
kernel, so one thread's call must not change what the other's launch may take:
every call succeeds and repeats the bits of the same call made alone."""
import threading

import numpy as np
import pytest

import sg_inputs as S
from tests.gpu_common import random_csr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import paper_1205_1864_gb300 as L
    return L


def _csr(lib, M, p, max_row, n=200):
    rowptr, colidx = random_csr(n, seed=M + max_row, max_row=max_row)
    vals = np.random.default_rng(p).uniform(-1, 1, size=(len(colidx), M + 1))
    return lib.SGProblem(0, 0, M, p, rowptr, colidx, vals)


def _block(n, w, dtype):
    import torch
    return torch.tensor(S.random_block(n, w, seed=w), dtype=dtype, device="cuda")


def _args(lib, kind):
    """The entry point and, for a call with little shared memory and one with
    much (above the 48 KB that every kernel may have), its arguments before the
    stream, its output and what must stay alive."""
    import torch
    from ctypes import POINTER, byref, c_double
    ptr = lib._ptr
    if kind == "vcycle":        # the restriction's residuals: 1024 doubles wide, 9 * 512 * 16 bytes
        o, got = lib.prec_opts(), []
        for w in (2, 1024):
            h = lib.SGProblem.from_inputs(S.make_problem(64, 1, 0.3, 0.5), 1)
            B = _block(h.n, w, torch.float64)
            X = torch.zeros_like(B)
            got.append(((h.h, ptr(B), ptr(X), w, lib.SG_F64, byref(o)), X, (h, B, o)))
        return lib._lib.LIB.sg_vcycle_apply, got
    # up to 60 nonzeros of 217 doubles a row, 96 KB; pair sums and inputs of P = 715 and 1001, 72 and 98 KB
    hs = [_csr(lib, 9, 4, 4), _csr(lib, 10, 4, 4)] if kind == "apply_df64" else [_csr(lib, 2, 1, 4), _csr(lib, 6, 4, 60)]
    got = []
    for h in hs:
        U = _block(h.n, h.P, torch.float32 if kind == "apply_df64" else torch.float64)
        if kind == "gradient":
            W, g, hk = np.ones((1, h.M + 1)), torch.zeros(1, dtype=torch.float64, device="cuda"), None
            got.append(((h.h, ptr(U), ptr(U), 1, W.ctypes.data_as(POINTER(c_double)), ptr(g), hk), g, (h, U, W)))
        else:
            Y = torch.zeros(h.n, h.P, dtype=torch.float64, device="cuda")
            got.append(((h.h, ptr(U), ptr(Y), lib._lib.SG_F32_ACCDF64 if kind == "apply_df64" else lib.SG_F64), Y, (h, U)))
    return (lib._lib.LIB.sg_qoi_grad if kind == "gradient" else lib._lib.LIB.sg_apply), got


@pytest.mark.parametrize("kind,n", [("apply", 20000), ("apply_df64", 20000), ("gradient", 20000), ("vcycle", 2000)])
def test_launches_do_not_meet(lib, kind, n):
    """The calls go to the library with prepared arguments: nothing but the
    call itself, which runs outside the interpreter lock, between two of them."""
    import torch
    call, both = _args(lib, kind)
    streams = [torch.cuda.Stream() for _ in both]
    alone = []
    torch.cuda.synchronize()
    for (args, out, _), st in zip(both, streams):
        assert call(*args, st.cuda_stream) == 0
        torch.cuda.synchronize()
        alone.append(out.clone())
    torch.cuda.synchronize()
    refused = [0, 0]
    gate = threading.Barrier(2)

    def work(i):
        args, st = both[i][0], streams[i].cuda_stream
        gate.wait()
        for _ in range(n):
            refused[i] += call(*args, st) != 0

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert refused == [0, 0]
    assert all(torch.equal(out, a) for (_, out, _), a in zip(both, alone))
