"""The launch shapes of the interface, edge and update kernels are chosen without
touching the gate's variant: where none has been chosen the single form goes on
taking the decisions inside its reconstruction, and a chosen variant stays."""
import pytest

from paper_2306_04467_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2306_04467_gb300 import gks2l as g  # noqa: E402


@pytest.mark.parametrize("chosen", [None, 0, 4])
def test_three_shapes_leave_the_gate_where_it_is(chosen):
    # 180,000 triangles: the gate's own kernel takes some 20 us, the time between
    # two events some 2 us where its decisions are taken inside
    prob = inputs.interface_dambreak(300)
    s = g.problem_solver(prob, precision=g.GKS2L_FP32, indicator=g.GKS2L_INDICATOR_MLP)
    if chosen is not None:
        s.set_launch_shapes([0, 0, 1, chosen])
    else:
        s.set_launch_shapes(s.autotune(1)[:3])      # before a network is loaded: no variant
    s.set_mlp(inputs.gate_init(9))
    s.set_launch_shapes([1, 1, 1])
    s.advance(4)
    s.profile_kernels(3)
    us = 1e3 * s.profile_kernels(10)["gate"]
    assert us > 8 if chosen == 0 else us < 6, us
    for bad in ([1, 1, 1, 1, 1], [1, 5, 1], [1, 1, 1, -1], [1, 1, 1, g.GKS2L_GATE_VARIANTS]):
        with pytest.raises((g.GKSError, IndexError, ValueError)):
            s.set_launch_shapes(bad)
