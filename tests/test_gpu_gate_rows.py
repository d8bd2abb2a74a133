"""The gate network's kernels on samples that do not lie on 16-byte boundaries
and in numbers beyond one tile per warp: the logits are a function of a
sample's row alone, so they are equal bit for bit however the rows lie in
memory and in whichever call they come; a gradient is the sum over its
samples, so a large batch's equals the sum of its pieces' to FP32 summation
(tiles of 16 samples added one after the other: relative error below the
number of additions, some hundreds, times 6e-8, of the summed magnitudes).
"""
import numpy as np
import pytest

from paper_2306_04467_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2306_04467_gb300 import gks2l as g  # noqa: E402

DEV = torch.device("cuda", 0)


def placed(X, offset):
    """X at `offset` floats from a 16-byte boundary."""
    buf = torch.empty(X.size + offset, dtype=torch.float32, device=DEV)
    view = buf[offset:].view(X.shape)
    view.copy_(torch.from_numpy(X))
    return view


def logits(X, P):
    s = torch.empty(X.shape[0], dtype=torch.float32, device=DEV)
    g.mlp_forward(X, P, s)
    return s


@pytest.mark.parametrize("n", [1, 33, 4097, 100003])
def test_logits_do_not_depend_on_placement_or_call(n):
    X, _ = inputs.gate_samples(n, seed=5)
    P = torch.from_numpy(inputs.gate_init(9)).to(DEV)
    ref = logits(placed(X, 0), P)
    for offset in (1, 2, 3):
        assert torch.equal(logits(placed(X, offset), P), ref)
    whole = placed(X, 0)
    pieces = torch.cat([logits(whole[i:i + 999], P) for i in range(0, n, 999)])
    assert torch.equal(pieces, ref)


@pytest.mark.parametrize("n,offset", [(15, 1), (3001, 3), (40007, 0), (40007, 1)])
def test_gradient_is_the_sum_over_pieces(n, offset):
    X, y = inputs.gate_samples(n, seed=6)
    P = torch.from_numpy(inputs.gate_init(9)).to(DEV)
    X, y = placed(X, offset), torch.from_numpy(y).to(DEV)

    def grad(a, b):
        G = torch.empty(g.GKS2L_MLP_NTRAIN, dtype=torch.float32, device=DEV)
        L = torch.empty(1, dtype=torch.float32, device=DEV)
        g.mlp_grad(X[a:b], y[a:b], P, 2.0, G, L)
        return torch.cat([G, L]).double()

    whole = grad(0, n)
    pieces = [grad(a, min(a + 16, n)) for a in range(0, n, 16)] if n < 4000 else \
        [grad(a, min(a + 992, n)) for a in range(0, n, 992)]
    total, size = sum(pieces), sum(p.abs() for p in pieces)
    assert float(((whole - total).abs() / (size + 1e-30)).max()) < 300 * 6e-8
