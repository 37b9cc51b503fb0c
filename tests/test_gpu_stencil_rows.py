"""The TMA-fed FP32 stencil with one row of nodes per thread (launches of one wave) and with two:
the same bits, at row counts that leave half a pair, a single row or a whole tile over, and the
oracle's values (1e-5 of the largest for the filter, as in the other FP32 tests).
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from paper_1603_04334_gb300 import sparc  # noqa: E402


@pytest.mark.parametrize("n3", [(32, 16, 20), (36, 33, 25), (4, 1, 40), (64, 47, 9), (8, 2, 3)])
@pytest.mark.parametrize("degree", [1, 4])
def test_rows(n3, degree):
    nd = n3[0] * n3[1] * n3[2]
    g = np.random.default_rng(nd)
    V = g.uniform(-3.0, 1.0, nd)
    ctx = sparc.Context(n3, 0.4, veff=V)
    X = torch.from_numpy(g.uniform(-0.5, 0.5, (700, nd))).to("cuda:0", torch.float32)
    x64 = X[:2].double().cpu().numpy()
    few, many = X[:2].contiguous(), X.clone()
    ctx.cheb_filter(many, torch.empty_like(many), degree, 5.0, 75.0, -4.0)
    ctx.cheb_filter(few, torch.empty_like(few), degree, 5.0, 75.0, -4.0)
    ctx.close()
    assert torch.equal(many[:2], few)
    ref = oracle.Hamiltonian(n3, 0.4, V).cheb_filter(x64, degree, 5.0, 75.0, -4.0)
    assert np.abs(few.double().cpu().numpy() - ref).max() <= 1e-5 * np.abs(ref).max()
