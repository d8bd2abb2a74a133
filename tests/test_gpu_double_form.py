"""The double form's branches of argument range against the FP64 oracle: the
error function's series and the library's beyond it (Froude numbers on both
sides of the switch and across it), and the nonlinear weights where the
product of two regularised indicators leaves the normal range.

Tolerance: the form's own bound after 100 stages, 1e-11 relative (each stage
adds a few roundings of 1e-16, and fewer stages are run here).
"""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2306_04467_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2306_04467_gb300 import gks2l as g  # noqa: E402

from test_gpu_parity import max_rel  # noqa: E402


def against_oracle(prob, stages, **kw):
    s = g.problem_solver(prob, precision=g.GKS2L_FP64, **kw)
    s.advance(stages)
    o = Oracle.from_problem(prob, **kw)
    o.advance(stages)
    return max_rel(prob, *s.get_state(), *o.get_state())


@pytest.mark.parametrize("speed", [0.0, 1.4, 1.57, 1.7, 3.0, 9.0])
def test_froude_numbers_on_both_sides_of_the_series(speed):
    prob = inputs.smooth_periodic(9)
    for base in (0, 3):
        prob.avg[base + 1] = speed * prob.avg[base]
        prob.avg[base + 2] = -0.5 * speed * prob.avg[base]
        prob.grad[base + 1] = speed * prob.grad[base]
        prob.grad[base + 2] = -0.5 * speed * prob.grad[base]
    ra, rg = against_oracle(prob, 6)
    assert ra <= 1e-11 and rg <= 1e-11, (ra, rg)


@pytest.mark.parametrize("scale", [1.0, 1e-60, 1e-85])
def test_weights_of_tiny_discharges_without_the_regulariser(scale):
    prob = inputs.smooth_periodic(9)
    x = np.arange(prob.mesh.n_tri)
    for v in (1, 2, 4, 5):
        prob.avg[v] = scale * (1.0 + 0.3 * np.sin(0.7 * x + v))
        prob.grad[v] = scale * np.cos(0.3 * x + v)
    ra, rg = against_oracle(prob, 1, weno_eps=0.0)
    assert ra <= 1e-11 and rg <= 1e-11, (ra, rg)
