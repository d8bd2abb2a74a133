"""A workspace sized for the library before its double form kept the sides'
values of the interface pass still suffices: those values, the staging area,
the between-stage state and the other arrays that are never alive together
share memory, and no row is kept that no kernel reads."""
import ctypes

import pytest

from paper_2306_04467_gb300 import build, gks2l, inputs

# bytes that gks2l_workspace_bytes gave then, in the double and the single form
SIZES = [("smooth_periodic", 4, 237616, 142384), ("interface_dambreak", 4, 241712, 144688),
         ("smooth_periodic", 16, 2124592, 1239088), ("interface_dambreak", 16, 2137904, 1247024),
         ("smooth_periodic", 33, 8775472, 5110064), ("interface_dambreak", 33, 8801328, 5125168),
         ("smooth_periodic", 96, 72599696, 42253712), ("interface_dambreak", 96, 72676752, 42298512)]


@pytest.mark.parametrize("problem,squares,fp64,fp32", SIZES)
def test_workspace_is_no_larger_than_before(problem, squares, fp64, fp32):
    build.build()
    lib = gks2l.load()
    mesh = gks2l._MeshArrays(getattr(inputs, problem)(squares).mesh)
    for precision, size in ((gks2l.GKS2L_FP64, fp64), (gks2l.GKS2L_FP32, fp32)):
        h, n = gks2l._P(), ctypes.c_size_t(0)
        par = gks2l.default_params(precision=precision)
        assert lib.gks2l_create((gks2l.gks2l_mesh * 1)(mesh.s), ctypes.byref(par), ctypes.byref(h)) == 0
        assert lib.gks2l_workspace_bytes(h, ctypes.byref(n)) == 0
        lib.gks2l_destroy(h)
        assert n.value <= size, (precision, n.value, size)
