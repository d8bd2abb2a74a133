"""The stage kernels at the edges of their tiles and launch rules: meshes of
fewer cells than a tile, one tile, a few cells more, and more tiles than SMs,
periodic and walled (mirrored stencils), in both forms against the oracle.

Tolerances. Double form: its bound after 100 stages, 1e-11. Single form: a
stage's averages carry some tens of roundings of 6e-8, so four stages stay
below 1e-5 of a variable's largest value; gradients divide interface values'
roundings by the cell size, which the scale of max_rel does too, and add the
fit's amplification of about ten: 1e-3.
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


def problem(kind, nx, ny):
    mesh = inputs.jittered_mesh(nx, ny, domain=(0.0, nx / ny, 0.0, 1.0), seed=3, bc=kind)
    b = inputs.vertex_samples(lambda x, y: 0.05 * np.sin(2 * np.pi * x * ny / nx) * np.cos(2 * np.pi * y), mesh)
    bm, bg = inputs.p1_average_and_gradient(b, mesh)
    x = np.arange(mesh.n_tri)
    avg = np.zeros((6, mesh.n_tri))
    grad = np.zeros((6, 2, mesh.n_tri))
    avg[3], grad[3] = 0.9 - bm + 0.004 * np.sin(x), -bg
    avg[0] = 0.6 + 0.004 * np.cos(0.7 * x)
    for v in (1, 2, 4, 5):
        avg[v] = 0.02 * np.sin(0.3 * x + v)
    return inputs.Problem("tiles", mesh, b, avg, grad, g=9.81, chi=0.97, cfl=0.4)


@pytest.mark.parametrize("precision,ta,tg", [(g.GKS2L_FP64, 1e-11, 1e-11), (g.GKS2L_FP32, 1e-5, 1e-3)])
@pytest.mark.parametrize("kind,nx,ny", [("periodic", 3, 3), ("periodic", 4, 4), ("periodic", 17, 1 + 2), ("wall", 1, 2),
                                        ("wall", 5, 3), ("wall", 11, 3), ("wall", 51, 50), ("periodic", 49, 50)])
def test_tile_edges(kind, nx, ny, precision, ta, tg):
    prob = problem(kind, nx, ny)
    s = g.problem_solver(prob, precision=precision)
    s.advance(4)
    o = Oracle.from_problem(prob)
    o.advance(4)
    ra, rg = max_rel(prob, *s.get_state(), *o.get_state())
    assert ra <= ta and rg <= tg, (ra, rg)
