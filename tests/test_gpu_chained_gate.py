"""Chained launches with the learned gate on: the reconstruction with the
decisions inside, the fused edge pass, its deferred units and the update read what
the one before has written. Runs by whole steps, by single stages and with a step
captured in a caller's graph agree bit for bit, for a network that calls about
half of the cells smooth, with walls and ragged last tiles; the decisions taken
inside the reconstruction and those of the gate's own mma.sync kernel are the
same, and the forms with the gate agree with each other."""
import numpy as np
import pytest

from oracle import mlp
from oracle.oracle import Oracle
from paper_2306_04467_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2306_04467_gb300 import gks2l as g  # noqa: E402

STAGES = 8


def case(squares):
    """Walls, features in every cell; a network whose median logit on the
    initial state is at the threshold."""
    prob = inputs.internal_wave_ridge(8 * squares, squares, seed=5)
    rng = np.random.default_rng(squares)
    prob.avg[0] += 1e-3 * rng.standard_normal(prob.mesh.n_tri)
    prob.avg[3] += 1e-3 * rng.standard_normal(prob.mesh.n_tri)
    P = inputs.gate_init(9).astype(np.float32)
    P[mlp.B3] -= np.float32(np.median(mlp.forward(P, Oracle.from_problem(prob).gate_features(), use_bf16=True)))
    return prob, P


def solver(prob, P, precision, variant, stream):
    par = g.default_params(g=prob.g, chi=prob.chi, cfl=prob.cfl, precision=precision,
                           indicator=g.GKS2L_INDICATOR_MLP, indicator_threshold=0.5)
    with torch.cuda.stream(stream):
        s = g.Solver(prob.mesh, par, prob.b_vert)
        if variant is not None:
            s.set_launch_shapes([0, 0, 0, variant])
        s.set_mlp(P)
        s.set_state(prob.avg, prob.grad)
    return s


def finish(s):
    st = s.stats()
    assert st["status"] == 0 and 0.0 < st["smooth_fraction"] < 1.0
    return (st["smooth_fraction"],) + s.get_state()


def same(a, b):
    return a[0] == b[0] and np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])


@pytest.mark.parametrize("squares", [3, 9, 29])      # 144, 1,296 and 13,456 triangles: each ends in half a tile
@pytest.mark.parametrize("precision", [g.GKS2L_FP32, g.GKS2L_FP64])
def test_gated_steps_stages_and_a_callers_graph_agree(precision, squares):
    prob, P = case(squares)
    st = torch.cuda.Stream()
    ref = {}
    for variant in (None, 0, 2, 4, 8, 12):
        whole, single, graphed = (solver(prob, P, precision, variant, st) for _ in range(3))
        with torch.cuda.stream(st):
            whole.advance(STAGES)
            for _ in range(STAGES):
                single.advance(1)
            graphed.advance(2)
        st.synchronize()
        cg = torch.cuda.CUDAGraph()
        with torch.cuda.graph(cg, stream=st, capture_error_mode="thread_local"):
            graphed.advance(1, sync=False)
            graphed.advance(1, sync=False)
        with torch.cuda.stream(st):
            for _ in range(STAGES // 2 - 1):
                cg.replay()
        st.synchronize()
        out = finish(whole)
        for other in (single, graphed):
            assert same(out, finish(other)), variant
        ref[variant] = out
        del whole, single, graphed
    # the mma.sync kernel's placements, the edge path and the decisions inside
    # the reconstruction change nothing (the tcgen05 kernel's logits may differ
    # in their last bit)
    for variant in (None, 4, 8, 12):
        assert same(ref[0], ref[variant]), variant
