"""Rayleigh-Ritz of blocks far from normalised: right within the range of FP32 products (column
norms of about 2^-68 to 2^68), refused beyond it, with the same errors at every size of the dense
step. Tolerances as in test_gpu_dense.py (FP64) and the mixed form's 1e-5 for FP32 blocks."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from paper_1603_04334_gb300 import sparc  # noqa: E402

NOT_SPD, NONFINITE = -4, -5


@pytest.mark.parametrize("ns", [1, 5, 40])
@pytest.mark.parametrize("dtype,scale,status", [
    ("f64", 1e-310, NOT_SPD), ("f64", 1e-140, NOT_SPD), ("f64", 1e-60, NOT_SPD),
    ("f64", 1e-30, NOT_SPD), ("f64", 1e-15, 0), ("f64", 1e10, 0), ("f64", 1e60, NONFINITE),
    ("f64", 1e140, NONFINITE), ("f32", 1e-40, NOT_SPD), ("f32", 1e-30, NOT_SPD),
    ("f32", 1e-15, 0), ("f32", 1e15, 0)])
def test_scaled_block(ns, dtype, scale, status):
    n3 = (20, 18, 17)
    nd = n3[0] * n3[1] * n3[2]
    g = np.random.default_rng(ns)
    V = g.uniform(-4.0, 1.0, nd)
    Y = g.uniform(-0.5, 0.5, (ns, nd)) * scale
    X = torch.from_numpy(Y).to("cuda:0", torch.float64 if dtype == "f64" else torch.float32)
    Y = X.double().cpu().numpy() / scale
    ctx = sparc.Context(n3, 0.4, veff=V)
    try:
        if status:
            with pytest.raises(sparc.SparcError) as e:
                ctx.orth_rr(X)
            assert e.value.status == status
            return
        ritz, _ = ctx.orth_rr(X)
    finally:
        ctx.close()
    H = oracle.Hamiltonian(n3, 0.4, V)
    lam = oracle.orth_rr(Y, H.apply(Y))[2]
    X = X.double().cpu().numpy()
    assert np.abs(ritz - lam).max() <= 1e-10
    assert np.abs(X @ X.T - np.eye(ns)).max() <= (1e-12 if dtype == "f64" else 1e-5)
