"""The FP32 stencil fed by 4-byte copies (rows or blocks that TMA cannot address) against the
oracle and against the TMA-fed form, whose arithmetic it shares: grids around the 32 x 16 tile,
thinner than the halo, one and several z ranges. Tolerances: 2e-6 of the largest |H X|, 1e-5 for
the filter (as in the other FP32 tests); equality with the TMA form.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from paper_1603_04334_gb300 import sparc  # noqa: E402


def block(ncols, ld, shift):
    flat = torch.zeros(ncols * ld + shift, dtype=torch.float32, device="cuda:0")
    return flat[shift:].view(ncols, ld)


@pytest.mark.parametrize("n3,pad,ncols", [((33, 17, 70), 0, 2), ((5, 7, 9), 0, 3), ((1, 1, 1), 0, 1),
                                          ((31, 15, 8), 3, 1), ((65, 33, 1), 0, 40),
                                          ((2, 50, 200), 1, 1)])
def test_copy_form_matches_oracle(n3, pad, ncols):
    h = 0.4
    nd = n3[0] * n3[1] * n3[2]
    ld = nd + pad
    g = np.random.default_rng(nd)
    V = g.uniform(-3.0, 1.0, nd)
    H = oracle.Hamiltonian(n3, h, V)
    ctx = sparc.Context(n3, h, veff=V)
    X, Y = block(ncols, ld, 1), block(ncols, ld, 1)
    X.copy_(torch.from_numpy(g.uniform(-0.5, 0.5, (ncols, ld))))
    Y.fill_(7.0)
    x64 = X.double().cpu().numpy()[:, :nd].copy()
    ctx.apply_H(X, Y)
    got = Y.double().cpu().numpy()
    ref = H.apply(x64)
    assert np.abs(got[:, :nd] - ref).max() <= 2e-6 * np.abs(ref).max()
    assert np.all(got[:, nd:] == 7.0)
    a0, a, b = -4.0, 5.0, 75.0
    ref = H.cheb_filter(x64, 7, a, b, a0)
    ctx.cheb_filter(X, Y, 7, a, b, a0)
    got = X.double().cpu().numpy()[:, :nd]
    assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max()
    ctx.close()


@pytest.mark.parametrize("n3,ncols", [((64, 48, 40), 5), ((36, 20, 90), 1)])
def test_copy_form_equals_the_tma_form(n3, ncols):
    nd = n3[0] * n3[1] * n3[2]
    g = np.random.default_rng(nd)
    ctx = sparc.Context(n3, 0.4, veff=g.uniform(-3.0, 1.0, nd))
    out = []
    for shift in (0, 1):               # on and off the 16-byte boundary
        X, Y = block(ncols, nd, shift), block(ncols, nd, shift)
        X.copy_(torch.from_numpy(np.random.default_rng(3).uniform(-0.5, 0.5, (ncols, nd))))
        ctx.cheb_filter(X, Y, 6, 5.0, 75.0, -4.0)
        out.append(X.clone())
    assert torch.equal(out[0], out[1])
    ctx.close()
