"""The FP64 stencil's forms against the oracle: paired and single loads (odd rows, odd leading
dimensions, blocks that start off a pair boundary), the integer potential and the general form
(kinetic scale, potentials too large for the integer weights), short z ranges and grids smaller
than a tile. Tolerance: the contract's 1e-12 of the largest |H X|, degree * 1e-12 for the filter.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from paper_1603_04334_gb300 import sparc  # noqa: E402


def block(ncols, ld, shift, dtype=torch.float64):
    """A contiguous (ncols, ld) block that starts `shift` elements into its allocation."""
    flat = torch.zeros(ncols * ld + shift, dtype=dtype, device="cuda:0")
    return flat[shift:].view(ncols, ld)


@pytest.mark.parametrize("n3,pad,shift,ncols", [
    ((34, 18, 23), 0, 0, 3),    # pairs, ragged tiles
    ((34, 18, 23), 1, 0, 3),    # odd leading dimension
    ((34, 18, 23), 0, 1, 2),    # off the pair boundary
    ((33, 17, 5), 0, 0, 4),     # odd rows, one z range
    ((1, 1, 1), 0, 0, 1),
    ((2, 40, 3), 0, 0, 1),
    ((65, 3, 64), 2, 0, 40),
])
@pytest.mark.parametrize("vmax,kscale", [(3.0, 1.0), (3.0, 0.7), (2e3, 1.0)])
def test_apply_and_filter(n3, pad, shift, ncols, vmax, kscale):
    h = 0.4
    nd = n3[0] * n3[1] * n3[2]
    ld = nd + pad
    g = np.random.default_rng(nd + pad + shift)
    V = g.uniform(-vmax, 0.2 * vmax, nd)
    H = oracle.Hamiltonian(n3, h, V, kscale=kscale)
    ctx = sparc.Context(n3, h, veff=V)
    ctx.set_kinetic_scale(kscale)
    X = np.zeros((ncols, ld))
    X[:, :nd] = g.uniform(-0.5, 0.5, (ncols, nd))
    Xd, Yd = block(ncols, ld, shift), block(ncols, ld, shift)
    Xd.copy_(torch.from_numpy(X))
    Yd.fill_(7.0)
    ctx.apply_H(Xd, Yd)
    ref = H.apply(X[:, :nd].copy())
    got = Yd.cpu().numpy()
    assert np.abs(got[:, :nd] - ref).max() <= 1e-12 * np.abs(ref).max()
    assert np.all(got[:, nd:] == 7.0)
    a0, a, b = -1.1 * vmax, 0.0, 0.3 * vmax + 70.0
    ref = H.cheb_filter(X[:, :nd].copy(), 5, a, b, a0)
    ctx.cheb_filter(Xd, Yd, 5, a, b, a0)
    got = Xd.cpu().numpy()
    assert np.abs(got[:, :nd] - ref).max() <= 5e-12 * np.abs(ref).max()
    ctx.close()
