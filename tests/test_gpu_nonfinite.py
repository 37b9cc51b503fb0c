"""Calls on data with NaN return, with NaN in their results, as an operation on such data does;
what a caller learns of it is in the results (first_bounds alone refuses an interval of NaN)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from paper_1603_04334_gb300 import sparc  # noqa: E402


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_density(bad):
    n, maxit = 20, 700                         # more than one launch of the solver
    rho = np.random.default_rng(0).uniform(0.0, 1.0, n ** 3)
    rho[1234] = bad
    ctx = sparc.Context(n, 0.3, veff=np.zeros(n ** 3))
    phi, it, rel = ctx.poisson(torch.from_numpy(rho).to("cuda:0"), tol=1e-10, maxit=maxit)
    assert torch.isnan(phi).all() and it == maxit and rel == 0.0
    # and the context is as good as before
    phi, it, rel = ctx.poisson(torch.ones(n ** 3, dtype=torch.float64, device="cuda:0"), tol=1e-10)
    assert torch.isfinite(phi).all() and 0 < it < maxit and 0.0 < rel <= 1e-10
    ctx.close()


def test_potential():
    n = 20
    V = np.zeros(n ** 3)
    V[1234] = np.nan
    ctx = sparc.Context(n, 0.3, veff=V)
    assert np.isnan(ctx.lanczos_bounds(6)).all()
    with pytest.raises(sparc.SparcError) as e:
        ctx.first_bounds(6)
    assert e.value.status == sparc.SPARC_ERR_ARG
    ctx.close()
