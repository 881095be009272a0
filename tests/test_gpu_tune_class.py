"""sg_autotune keeps what it timed per class of problem in the process: a handle
that may not take the same inner solvers is another class and is timed itself."""
import pytest

import sg_inputs as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("switch", ["SGHSC_NO_BLOCK", "SGHSC_NO_CLUSTER", "SGHSC_NO_CLUSTER16", "SGHSC_NO_PIPE"])
def test_switches_are_another_class(monkeypatch, switch):
    import paper_1205_1864_gb300 as L
    prob = S.make_problem(64, 3, 0.3, 0.5)

    def launches():
        h = L.SGProblem.from_inputs(prob, 2)
        n0 = L._lib.LIB.sg_kernel_launches()
        L.sg_autotune(h)
        return L._lib.LIB.sg_kernel_launches() - n0

    launches()
    assert launches() == 0
    monkeypatch.setenv(switch, "1")
    assert launches() > 0 and launches() == 0
