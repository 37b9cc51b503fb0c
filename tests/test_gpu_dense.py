"""The Ns x Ns eigensolve at the sizes where its path changes: one CTA (up to 32 states), FP32
block Jacobi with one pair of blocks (up to 64), several blocks with a short or odd last one,
larger product tiles (above 256), and spectra that the refinement cannot separate (exactly
equal and nearly equal eigenvalues). Ritz values against a 64-bit eigensolve of the same
problem to 1e-10 Ha (the FP64 contract), orthonormality to 1e-12, residuals to 1e-9, as in the
other Rayleigh-Ritz tests.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from paper_1603_04334_gb300 import sparc  # noqa: E402


def solve(n3, V, Y):
    H = oracle.Hamiltonian(n3, 0.5, V)
    ctx = sparc.Context(n3, 0.5, veff=V)
    Yd = torch.from_numpy(Y.copy()).to("cuda:0")
    ritz, resid = ctx.orth_rr(Yd)
    X = Yd.cpu().numpy()
    ctx.close()
    Xo, HXo, lam, res, _ = oracle.orth_rr(Y, H.apply(Y))
    assert np.abs(ritz - lam).max() <= 1e-10
    assert np.abs(resid - res).max() <= 1e-9
    assert np.abs(X @ X.T - np.eye(Y.shape[0])).max() <= 1e-12
    HX = H.apply(X)
    A = X @ HX.T                                  # the rotated problem is diagonal
    assert np.abs(A - np.diag(ritz)).max() <= 1e-10
    return X, Xo


@pytest.mark.parametrize("ns", [1, 2, 3, 31, 32, 33, 46, 63, 64, 65, 97, 128, 255, 257])
def test_sizes(ns):
    n3 = (16, 15, 14)
    g = np.random.default_rng(ns)
    nd = n3[0] * n3[1] * n3[2]
    solve(n3, g.uniform(-4.0, 1.0, nd), g.uniform(-0.5, 0.5, (ns, nd)))


@pytest.mark.parametrize("ns,spread", [(24, 0.0), (60, 0.0), (100, 0.0), (60, 1e-9), (100, 1e-6)])
def test_close_eigenvalues(ns, spread):
    # kinetic eigenvectors of a cube (multiplets of up to six equal eigenvalues) and copies of
    # their space lifted apart by `spread`, mixed by a random rotation
    n = 14
    k = np.arange(n)
    T = np.zeros((n, n))
    w = [-2.0 * sum(1.0 / q ** 2 for q in range(1, 7))]
    for p in range(1, 7):
        r = 1.0
        for q in range(1, p + 1):
            r *= (6 - q + 1) / (6 + q)
        w.append(2.0 * (-1.0) ** (p + 1) / p ** 2 * r)
    for p in range(7):
        T[np.abs(k[:, None] - k[None, :]) == p] = w[p] / 0.25
    ev, Q = np.linalg.eigh(-0.5 * T)
    e3 = ev[:, None, None] + ev[None, :, None] + ev[None, None, :]
    low = np.argsort(e3.reshape(-1), kind="stable")[:ns]
    B = np.stack([np.einsum("i,j,k->ijk", Q[:, a], Q[:, b], Q[:, c]).reshape(-1)
                  for a, b, c in (np.unravel_index(t, e3.shape) for t in low)])
    g = np.random.default_rng(ns)
    R, _ = np.linalg.qr(g.standard_normal((ns, ns)))
    V = spread * g.uniform(-1.0, 1.0, n ** 3)
    solve((n, n, n), V, R @ B)
