"""H X and the Chebyshev filter in FP64 at every stencil radius, against the oracle: the integer
weights, and with them the units in which the stencil rounds, depend on the radius. Potentials
inside the integer form's range, at its edge and beyond it. Tolerances as in
test_gpu_parity.py: 1e-12 normwise for H X, degree * 1e-12 for the filter."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from paper_1603_04334_gb300 import sparc  # noqa: E402


@pytest.mark.parametrize("radius", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("depth", [4.0, 60.0, 1000.0])
def test_apply_and_filter(radius, depth):
    n3, h, ncols, degree = (37, 18, 21), 0.3, 3, 6
    nd = n3[0] * n3[1] * n3[2]
    g = np.random.default_rng(radius)
    V = g.uniform(-depth, 1.0, nd)
    H = oracle.Hamiltonian(n3, h, V, no=radius)
    ctx = sparc.Context(n3, h, veff=V, radius=radius)
    X = g.uniform(-0.5, 0.5, (ncols, nd))
    Xd = torch.from_numpy(X.copy()).to("cuda:0")
    HX = torch.empty_like(Xd)
    ctx.apply_H(Xd, HX)
    ref = H.apply(X)
    assert np.abs(HX.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
    a, b, a0 = -0.5 * depth, 6.0 * np.pi ** 2 / h ** 2, -depth
    ctx.cheb_filter(Xd, torch.empty_like(Xd), degree, a, b, a0)
    ref = H.cheb_filter(X, degree, a, b, a0)
    assert np.abs(Xd.cpu().numpy() - ref).max() <= degree * 1e-12 * np.abs(ref).max()
    ctx.close()
