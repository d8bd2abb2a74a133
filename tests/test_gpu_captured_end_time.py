"""A step captured in a caller's graph keeps the end time of the call that was
captured, whatever end times calls before and between its replays have, and
calls after a replay keep theirs: the run equals the same calls without a
capture bit for bit."""
import numpy as np
import pytest

from paper_2306_04467_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2306_04467_gb300 import gks2l as g  # noqa: E402


@pytest.mark.parametrize("precision", [g.GKS2L_FP64, g.GKS2L_FP32])
@pytest.mark.parametrize("captured", [0.0, 1.4], ids=["none", "within_the_next_step"])
def test_a_captured_step_keeps_its_end_time(captured, precision):
    prob = inputs.interface_dambreak(17)
    st = torch.cuda.Stream()
    par = g.default_params(g=prob.g, chi=prob.chi, cfl=prob.cfl, precision=precision)
    out = []
    for graphed in (True, False):
        with torch.cuda.stream(st):
            s = g.Solver(prob.mesh, par, prob.b_vert)
            s.set_state(prob.avg, prob.grad)
            dt = s.advance(2)
            end = captured * dt

            def step():                                # by its stages: a whole step's graph cannot be captured
                s.advance(1, t_end=end, sync=False)
                s.advance(1, t_end=end, sync=False)
        if graphed:
            st.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=st, capture_error_mode="thread_local"):
                step()
            step = graph.replay
        times = []
        with torch.cuda.stream(st):
            step()                                     # to the captured end, or a whole step
            times.append(s.advance(0, t_end=1e-3 * dt))
            # past the captured end, or (with none captured) to an end of its own
            times.append(s.advance(2, t_end=0.0 if end else times[0] + 0.3 * dt))
            step()                                     # stands (its end is behind), or a whole step again
            times.append(s.advance(0))
        out.append((times, s.get_state()))
        if end:
            assert abs(times[0] - end) < 1e-12 and times[1] > end and times[2] == times[1]
        else:
            assert abs(times[1] - times[0] - 0.3 * dt) < 1e-12 and times[2] > times[1]
    assert out[0][0] == out[1][0]
    for x, y in zip(out[0][1], out[1][1]):
        assert np.array_equal(x, y)
