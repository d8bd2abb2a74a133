"""Runs to one end time after another: an instance that stood at an end time
while more stages were asked for goes on with the CFL step of its state, as
the FP64 oracle does, and so do the instances of an ensemble that arrived
before the others.

Tolerances: the FP64 form's own bound against the oracle after 100 stages, 1e-11
relative; an ensemble's instances equal the same meshes run alone bit for bit."""
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


def test_end_times_one_after_another_match_the_oracle():
    prob = inputs.interface_dambreak(12)
    s, o = g.problem_solver(prob), Oracle.from_problem(prob)
    dt = s.advance(2)
    o.advance(2)
    for end in (3.4 * dt, 3.4 * dt, 7.7 * dt):
        assert abs(s.advance(40, t_end=end) - end) < 1e-12
        o.advance(40, t_end=end)
    s.advance(2)
    o.advance(2)
    assert s.stats()["status"] == 0 and abs(s.stats()["t"] - o.t) < 1e-12
    ra, rg = max_rel(prob, *s.get_state(), *o.get_state())
    assert ra <= 1e-11 and rg <= 1e-11, (ra, rg)


@pytest.mark.parametrize("precision", [g.GKS2L_FP64, g.GKS2L_FP32])
def test_instances_that_arrived_first_go_on_like_alone(precision):
    probs = [inputs.ensemble_member(n, 11 + n) for n in (6, 24)]
    par = g.default_params(g=probs[0].g, chi=probs[0].chi, cfl=probs[0].cfl, precision=precision)
    ens = g.Solver([p.mesh for p in probs], par, np.concatenate([p.b_vert for p in probs]))
    ens.set_state(np.concatenate([p.avg for p in probs], axis=1), np.concatenate([p.grad for p in probs], axis=2))
    for end in (0.01, 0.02):
        ens.advance(400, t_end=end)
    a, gr = ens.get_state()
    first = 0
    for p in probs:
        alone = g.problem_solver(p, precision=precision)
        for end in (0.01, 0.02):
            while alone.advance(2, t_end=end) < end * (1 - 1e-12):     # it never stands
                pass
        n = p.mesh.n_tri
        b, h = alone.get_state()
        assert np.array_equal(a[:, first:first + n], b) and np.array_equal(gr[:, :, first:first + n], h)
        first += n
