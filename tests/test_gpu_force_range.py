"""The non-local force where the gradient's integer form changes: values of very different size
side by side, zero stretches, whole blocks scaled by powers of two up to the exponents that take
the plain FP64 sums, supports at the grid's faces. Against the FP64 oracle on the unscaled block
(scaling by a power of two is exact), to 1e-12 of the sum of the magnitudes that cancel, as in
the other force tests.
"""
import numpy as np
import pytest

import oracle
from oracle import observables as OB

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from paper_1603_04334_gb300 import sparc  # noqa: E402

N3, HH = (37, 29, 23), 0.45
R = np.array([[0.3, 5.0, 4.4], [15.9, 12.4, 0.2], [8.0, 6.1, 5.0]])


def block(kind):
    g = np.random.default_rng(8)
    nd = int(np.prod(N3))
    X = g.uniform(-0.5, 0.5, (4, nd))
    if kind == "mixed":
        X *= 2.0 ** g.integers(-60, 1, X.shape)
    elif kind == "gaps":
        X[g.uniform(size=X.shape) < 0.7] = 0.0
        X[1] = 0.0
    return X


@pytest.mark.parametrize("kind", ["plain", "mixed", "gaps"])
@pytest.mark.parametrize("dtype,power,radius", [("f64", 0, 6), ("f64", -420, 6), ("f64", 420, 6),
                                                ("f32", 0, 6), ("f32", -56, 6), ("f32", 40, 6),
                                                ("f64", 0, 1), ("f64", 0, 5)])
def test_force_range(kind, dtype, power, radius):
    gamma = np.random.default_rng(4).uniform(-2, 2, (3, 4))
    nd = int(np.prod(N3))
    tt = torch.float64 if dtype == "f64" else torch.float32
    Xd = torch.from_numpy(block(kind)).to("cuda:0", tt)
    Xo = Xd.double().cpu().numpy()
    g = np.array([1.0, 0.7, 0.2, 0.9])
    H = oracle.Hamiltonian(N3, HH, np.zeros(nd), R, gamma, no=radius)
    ctx = sparc.Context(N3, HH, R, None, gamma, veff=np.zeros(nd), radius=radius)
    f = ctx.nonlocal_force(Xd * 2.0 ** power, g) * 2.0 ** (-2 * power)
    ctx.close()
    Y, W = OB.nonlocal_projections(H, Xo)
    S = 4.0 / HH ** 3 * np.einsum("n,Jl,Jnl,Jndl->Jd", g, np.abs(gamma), np.abs(Y), np.abs(W))
    assert np.all(np.abs(f - OB.nonlocal_force(H, Xo, g)) <= 1e-12 * S)
