"""What shares a piece of the workspace does not meet: a state read between the
stages of a step (in the double form beside the sides' values of the edge pass),
a harvest there, statistics, states set and read in turn change nothing of a run,
at sizes from a mesh whose padding is larger than itself on."""
import numpy as np
import pytest

from paper_2306_04467_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2306_04467_gb300 import gks2l as g  # noqa: E402

GATED = dict(indicator=g.GKS2L_INDICATOR_MLP)
FORMS = {"fp64": dict(precision=g.GKS2L_FP64), "fp32": dict(precision=g.GKS2L_FP32),
         "fp64_positivity": dict(precision=g.GKS2L_FP64, positivity_floor=1e-3),
         "fp64_gate": dict(precision=g.GKS2L_FP64, **GATED), "fp32_gate": dict(precision=g.GKS2L_FP32, **GATED)}


@pytest.mark.parametrize("squares", [2, 3, 20])
@pytest.mark.parametrize("form", list(FORMS))
def test_reads_and_harvests_between_stages_change_nothing(form, squares):
    prob = inputs.interface_dambreak(squares)

    def solver():
        s = g.problem_solver(prob, **FORMS[form])
        if "gate" in form:
            s.set_mlp(inputs.gate_init(9))
            s.set_state(prob.avg, prob.grad)
        return s

    plain, other = solver(), solver()
    for k in range(4):
        plain.advance(1)
        other.advance(1)
        mid = other.get_state()
        X, y, _ = other.harvest(1e-2)
        other.stats()
        X1, y1, _ = other.harvest(1e-2)
        assert torch.equal(X, X1) and torch.equal(y, y1)
        for a, b, c in zip(plain.get_state(), other.get_state(), mid):
            assert np.array_equal(a, b) and np.array_equal(b, c), k
        assert np.isfinite(mid[0]).all()
    again = solver()
    again.set_state(*mid)
    for a, b in zip(again.get_state(), mid):
        assert np.array_equal(a, b)
