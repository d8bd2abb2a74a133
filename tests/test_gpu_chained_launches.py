"""Kernels launched behind one another (a step's graph, a new state's set-up, a
gradient's reduction) read what the one before has written: runs by whole
steps, whose kernels are chained, by single stages, whose first kernel is not,
and with a stage inside a caller's captured graph agree bit for bit at sizes from one tile
on, for the kernels of every form; gradients queued without a synchronisation
equal those taken one at a time."""
import numpy as np
import pytest

from paper_2306_04467_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2306_04467_gb300 import gks2l as g  # noqa: E402

DEV = torch.device("cuda", 0)
FORMS = {
    "fp64": dict(precision=g.GKS2L_FP64),
    "fp32": dict(precision=g.GKS2L_FP32),
    "positivity": dict(precision=g.GKS2L_FP32, positivity_floor=1e-3),
}


def solver(prob, form, stream):
    kw = dict(FORMS[form])
    par = g.default_params(g=prob.g, chi=prob.chi, cfl=prob.cfl, **kw)
    with torch.cuda.stream(stream):
        s = g.Solver(prob.mesh, par, prob.b_vert)
        s.set_state(prob.avg, prob.grad)
    return s


@pytest.mark.parametrize("squares", [3, 17, 90])
@pytest.mark.parametrize("form", list(FORMS))
def test_steps_stages_and_a_callers_graph_agree(form, squares):
    prob = inputs.interface_dambreak(squares)
    st = torch.cuda.Stream()
    whole, single, graphed = (solver(prob, form, st) for _ in range(3))
    with torch.cuda.stream(st):
        whole.advance(4)
        for _ in range(4):
            single.advance(1)
        graphed.advance(2)
    st.synchronize()
    cg = torch.cuda.CUDAGraph()
    with torch.cuda.graph(cg, stream=st, capture_error_mode="thread_local"):
        graphed.advance(1, sync=False)         # a step's first stage
    with torch.cuda.stream(st):
        cg.replay()
        graphed.advance(1)
    ref = whole.get_state()
    for other in (single, graphed):
        for x, y in zip(ref, other.get_state()):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("variant", [0, 2, 4, 8, 12])
def test_gate_placements_agree_over_steps_and_stages(variant):
    prob = inputs.interface_dambreak(40)
    P = inputs.gate_init(9)
    out = []
    for by in (8, 1):
        s = g.problem_solver(prob, precision=g.GKS2L_FP32)
        s.set_mlp(P)
        s.set_state(prob.avg, prob.grad)
        s.set_launch_shapes([0, 0, 0, variant])
        for _ in range(8 // by):
            s.advance(by)
        out.append(s.get_state())
    for x, y in zip(*out):
        assert np.array_equal(x, y)


def test_queued_gradients_equal_single_ones():
    X, y = inputs.gate_samples(8192, seed=3)
    X, y = torch.from_numpy(X).to(DEV), torch.from_numpy(y).to(DEV)
    P = [torch.from_numpy(inputs.gate_init(k)).to(DEV) for k in range(4)]
    L = torch.empty(1, dtype=torch.float32, device=DEV)

    def run(sync):
        out = [torch.empty(g.GKS2L_MLP_NTRAIN, dtype=torch.float32, device=DEV) for _ in range(40)]
        for i, G in enumerate(out):
            g.mlp_grad(X, y, P[i % 4], 2.0, G, L)
            if sync:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return out

    for a, b in zip(run(False), run(True)):
        assert torch.equal(a, b)
