"""The contraction kernels on blocks whose columns live in part of the grid: row chunks that are
zero in some columns or all, magnitudes that fall from chunk to chunk far below FP64's
resolution of the largest, odd column strides (scalar loads), one to several column blocks and
one to several chunks along the states (the rotation). sparc_gram_tc within its stated bound;
the projection pair and the rotation through sparc_orth_rr to the FP64 contract (Ritz values
1e-10 Ha, orthonormality 1e-12, residuals 1e-9), as in the other Rayleigh-Ritz tests.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from paper_1603_04334_gb300 import sparc  # noqa: E402

N3 = (17, 15, 27)


def local_block(seed, ns, nd):
    """Column j: noise over two thirds of the rows from a start of its own, falling to 1e-40 at
    both ends of that range, zero outside."""
    g = np.random.default_rng(seed)
    Y = np.zeros((ns, nd))
    m = 2 * nd // 3
    t = np.linspace(-1.0, 1.0, m)
    env = 10.0 ** (-40.0 * np.clip(np.abs(t) - 0.6, 0.0, None) / 0.4)
    for j in range(ns):
        a = int(g.integers(0, nd - m + 1))
        Y[j, a:a + m] = env * g.uniform(-0.5, 0.5, m)
    return Y


@pytest.mark.parametrize("ns", [1, 40, 130, 260])
@pytest.mark.parametrize("types", [("f32", "f64"), ("f64", "f64")])
def test_gram_tc_local(ns, types):
    nd = int(np.prod(N3))
    ctx = sparc.Context(N3, 0.5)
    tt = {"f32": torch.float32, "f64": torch.float64}
    A = torch.from_numpy(local_block(1, ns, nd)).to("cuda:0", tt[types[0]])
    B = torch.from_numpy(local_block(2, ns, nd)).to("cuda:0", tt[types[1]])
    G = ctx.gram_tc(A, B).cpu().numpy().T
    ctx.close()
    A, B = A.double().cpu().numpy(), B.double().cpu().numpy()

    def chunk_max(X):
        n = -(-nd // 256)
        P = np.zeros((ns, n * 256))
        P[:, :nd] = np.abs(X)
        return np.repeat(P.reshape(ns, n, 256).max(axis=2), 256, axis=1)[:, :nd]

    mA, mB = chunk_max(A), chunk_max(B)
    bound = 2.0 ** -21 * (mA @ mB.T + mA @ np.abs(B).T + np.abs(A) @ mB.T)
    assert np.all(np.abs(G - A @ B.T) <= bound + 1e-300)


@pytest.mark.parametrize("ns", [33, 64, 129, 260])
def test_projection_and_rotation_local(ns):
    nd = int(np.prod(N3))
    V = np.random.default_rng(ns).uniform(-4.0, 1.0, nd)
    Y = local_block(ns, ns, nd)
    H = oracle.Hamiltonian(N3, 0.5, V)
    ctx = sparc.Context(N3, 0.5, veff=V)
    Yd = torch.from_numpy(Y.copy()).to("cuda:0")
    ritz, resid = ctx.orth_rr(Yd)
    X = Yd.cpu().numpy()
    ctx.close()
    _, _, lam, res, _ = oracle.orth_rr(Y, H.apply(Y))
    assert np.abs(ritz - lam).max() <= 1e-10
    assert np.abs(resid - res).max() <= 1e-9
    assert np.abs(X @ X.T - np.eye(ns)).max() <= 1e-12
    assert np.abs(X @ H.apply(X).T - np.diag(ritz)).max() <= 1e-10
