"""sparc_poisson on densities near the ends of the FP64 range: r.r and p.Ap of CG are squares, which
leave it long before the density does. While tol^2 |f|^2 is above the smallest numbers the solve
is that of the same density times a power of ten (phi to 1e-6, iterations within 2); below, where
r.r runs out of bits before it meets the tolerance, and where it overflows, the call reports that it
did not converge."""
import functools

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from paper_1603_04334_gb300 import sparc  # noqa: E402

N3, H = (33, 19, 21), 0.4


def solve(scale, tol):
    nd = N3[0] * N3[1] * N3[2]
    rho = torch.from_numpy(np.random.default_rng(1).uniform(0.0, 1.0, nd) * scale).to("cuda:0")
    ctx = sparc.Context(N3, H, veff=np.zeros(nd))
    try:
        phi, it, rel = ctx.poisson(rho, tol=tol)
        return phi.cpu().numpy() / scale, it, rel
    finally:
        ctx.close()


reference = functools.lru_cache(None)(lambda tol: solve(1.0, tol))


@pytest.mark.parametrize("scale,tol", [(1e150, 1e-10), (1e-148, 1e-10), (1e-150, 1e-10),
                                       (1e-152, 1e-10), (1e-156, 1e-4), (1e-158, 1e-4)])
def test_solved(scale, tol):
    phi, it, rel = solve(scale, tol)
    ref, it_ref, _ = reference(tol)
    assert rel <= tol and abs(it - it_ref) <= 2
    assert np.abs(phi - ref).max() <= 1e-6 * np.abs(ref).max()


@pytest.mark.parametrize("scale,tol", [(1e156, 1e-4), (1e-156, 1e-10), (1e-160, 1e-4),
                                       (1e-161, 1e-4), (1e-162, 1e-4), (1e-163, 1e-10)])
def test_reported(scale, tol):
    with pytest.raises(sparc.SparcError) as e:
        solve(scale, tol)
    assert e.value.status == sparc.SPARC_ERR_TIMEOUT
