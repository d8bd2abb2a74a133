"""States and statistics read between the two stages of a step: the state a
run shows there continues like the uninterrupted run, and an instance that has
reached the end time shows its final state and mass, in both forms."""
import numpy as np
import pytest

from paper_2306_04467_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2306_04467_gb300 import gks2l as g  # noqa: E402

from test_gpu_parity import areas  # noqa: E402


@pytest.mark.parametrize("precision", [g.GKS2L_FP64, g.GKS2L_FP32])
def test_a_stopped_instance_shows_its_final_state(precision):
    # the coarse instance takes larger steps and arrives first
    probs = [inputs.ensemble_member(6, 11), inputs.ensemble_member(24, 12)]
    n0 = probs[0].mesh.n_tri
    par = g.default_params(g=probs[0].g, chi=probs[0].chi, cfl=probs[0].cfl, precision=precision)
    s = g.Solver([p.mesh for p in probs], par, np.concatenate([p.b_vert for p in probs]))
    s.set_state(np.concatenate([p.avg for p in probs], axis=1), np.concatenate([p.grad for p in probs], axis=2))
    alone = g.problem_solver(probs[0], precision=precision)
    t_end = 0.02
    while alone.advance(2, t_end=t_end) < t_end * (1 - 1e-12):
        pass
    final, fgrad = alone.get_state()
    steps = alone.stats()["stages"]
    s.advance(steps + 4, t_end=t_end)          # the first instance has arrived, the second has not
    before, _ = s.get_state()
    s.advance(1, t_end=t_end)
    a, gr = s.get_state()
    assert np.array_equal(a[:, :n0], final) and np.array_equal(gr[:, :, :n0], fgrad)
    assert not np.array_equal(a[:, n0:], before[:, n0:])
    area = np.concatenate([areas(p.mesh) for p in probs])
    mass = (area * a[3]).sum(), (area * a[0]).sum()
    got = s.stats()["mass"]
    # FP64 sums of a few thousand terms in another order
    assert abs(got[0] - mass[0]) < 1e-12 * mass[0] and abs(got[1] - mass[1]) < 1e-12 * mass[1]


@pytest.mark.parametrize("precision", [g.GKS2L_FP64, g.GKS2L_FP32])
def test_reading_between_stages_changes_nothing(precision):
    prob = inputs.interface_dambreak(12)
    whole = g.problem_solver(prob, precision=precision)
    whole.advance(6)
    s = g.problem_solver(prob, precision=precision)
    states = []
    for _ in range(6):
        s.advance(1)
        states.append(s.get_state()[0])
        s.stats()
    assert all(not np.array_equal(x, y) for x, y in zip(states, states[1:]))
    for x, y in zip(s.get_state(), whole.get_state()):
        assert np.array_equal(x, y)
