"""The FP64 nonlocal term and the Lanczos bounds at the column counts and sizes where their launch
shapes change: one vector, one and several column groups per thread, columns that do not start
on 16 bytes (single loads in the bound pass), grids smaller than a CTA and a Krylov space of one
vector. H X against the oracle to the contract's 1e-12 of the largest |H X|, the bounds to 1e-10
of the spectrum's size, as in the other tests of both.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from paper_1603_04334_gb300 import sparc  # noqa: E402


@pytest.mark.parametrize("ncols", [1, 2, 5, 33, 260])
@pytest.mark.parametrize("pad", [0, 1])
def test_nonlocal_columns(ncols, pad):
    n3, h = (37, 29, 23), 0.45
    nd = n3[0] * n3[1] * n3[2]
    g = np.random.default_rng(ncols + pad)
    R = np.array([n * h for n in n3]) * g.uniform(0.1, 0.9, (14, 3))
    gamma = g.uniform(-2, 2, (14, 4))
    V = g.uniform(-3.0, 0.5, nd)
    H = oracle.Hamiltonian(n3, h, V, R, gamma)
    ctx = sparc.Context(n3, h, R, None, gamma, veff=V)
    X = np.zeros((ncols, nd + pad))
    X[:, :nd] = g.uniform(-0.5, 0.5, (ncols, nd)) * 2.0 ** g.integers(-20, 20, (ncols, 1))
    Xd = torch.from_numpy(X).to("cuda:0")
    Yd = torch.empty_like(Xd)
    ctx.apply_H(Xd, Yd)
    ctx.close()
    got = Yd.cpu().numpy()[:, :nd]
    ref = H.apply(X[:, :nd].copy())
    assert np.all(np.abs(got - ref).max(axis=1) <= 1e-12 * np.abs(ref).max(axis=1))


@pytest.mark.parametrize("ncols", [1, 5, 33, 100])
def test_nonlocal_columns_f32(ncols):
    # a column's FP32 sums are the same bits in every launch shape
    n3, h = (37, 29, 23), 0.45
    nd = n3[0] * n3[1] * n3[2]
    g = np.random.default_rng(3)
    R = np.array([n * h for n in n3]) * g.uniform(0.1, 0.9, (14, 3))
    gamma = g.uniform(-2, 2, (14, 4))
    V = g.uniform(-3.0, 0.5, nd)
    ctx = sparc.Context(n3, h, R, None, gamma, veff=V)
    X = torch.from_numpy(g.uniform(-0.5, 0.5, (480, nd))).to("cuda:0", torch.float32)
    Y, Z = torch.empty_like(X), torch.empty_like(X[:ncols])
    ctx.apply_H(X, Y)
    ctx.apply_H(X[:ncols].contiguous(), Z)
    ctx.close()
    assert torch.equal(Y[:ncols], Z)
    H = oracle.Hamiltonian(n3, h, V, R, gamma)
    ref = H.apply(X[:ncols].double().cpu().numpy())
    assert np.abs(Z.double().cpu().numpy() - ref).max() <= 2e-6 * np.abs(ref).max()


@pytest.mark.parametrize("n3", [(1, 1, 1), (7, 5, 3), (33, 17, 5), (40, 41, 43)])
@pytest.mark.parametrize("k", [1, 3, 10])
def test_lanczos_sizes(n3, k):
    h = 0.4
    nd = n3[0] * n3[1] * n3[2]
    V = np.random.default_rng(nd).uniform(-3.0, 0.5, nd)
    H = oracle.Hamiltonian(n3, h, V)
    ctx = sparc.Context(n3, h, veff=V)
    lo, hi = ctx.lanczos_bounds(k, 5)
    ctx.close()
    rlo, rhi, _ = H.lanczos_bounds(k, 5)
    s = max(abs(rlo), abs(rhi))
    assert abs(lo - rlo) <= 1e-10 * s and abs(hi - rhi) <= 1e-10 * s
