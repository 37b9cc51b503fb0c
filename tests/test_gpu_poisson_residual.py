"""The residual f - A phi of sparc_poisson's solution from its definition, not the solver's
recursion (which follows whatever operator it is given and passes any tolerance): the exact
rational weights in extended precision on the host, f from the oracle, at every stencil radius.

Tolerance: FP64 conjugate gradients stop getting closer at some ||f - A x|| / ||f|| of their own,
which the oracle's solver shows when run far below it (tol 1e-16). The library's residual may be
tol plus twice that."""
import functools

import numpy as np
import pytest

from oracle import lap_weights, lap_weights_exact
from oracle import poisson as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from paper_1603_04334_gb300 import sparc  # noqa: E402


def residual(f, phi, n3, h, radius):
    w = [np.longdouble(x.numerator) / np.longdouble(x.denominator)
         for x in lap_weights_exact(radius)]
    shape = n3[::-1]
    q = np.pad(phi.reshape(shape).astype(np.longdouble), radius)
    L = 6 * w[0] * q[tuple(slice(radius, radius + m) for m in shape)]
    for p in range(1, radius + 1):
        for ax in range(3):
            for s in (p, -p):
                ix = [slice(radius, radius + m) for m in shape]
                ix[ax] = slice(radius + s, radius + s + shape[ax])
                L = L + w[p] * q[tuple(ix)]
    r = f.astype(np.longdouble) + (L / (4 * np.longdouble(np.pi) * np.longdouble(h) ** 2)).reshape(-1)
    return float(np.sqrt((r * r).sum()) / np.linalg.norm(f))


def rhs(rho, b, n3, h, radius):
    return rho + b - P.charge_correction(n3, h, P.multipole_moments(rho + b, n3, h), radius)


@functools.lru_cache(None)
def system(n3, h, radius):
    """A neutral cluster of four charges, and how close the oracle's solver gets."""
    c, L = P.box_centre(n3, h), np.array(n3) * h
    R = c + np.random.default_rng(0).uniform(-0.25, 0.25, (4, 3)) * L
    Z = np.full(4, 2.0)
    X = P.node_coords(n3, h)
    rho = sum(np.exp(-np.sum((X - x0) ** 2, axis=1) / 1.5) for x0 in R)
    rho *= Z.sum() / (h ** 3 * rho.sum())
    f = rhs(rho, P.pseudocharge(n3, h, R, Z, 1.0, radius), n3, h, radius)
    x, _, _ = P.cg_solve(lambda v: P.poisson_apply(v, n3, h, radius), f,
                         -6.0 * lap_weights(radius, h)[0] / P.FOUR_PI, 1e-16, 3000)
    return R, Z, rho, residual(f, x, n3, h, radius)


@pytest.mark.parametrize("tol", [1e-12, 1e-13, 1e-14])
@pytest.mark.parametrize("n3,h,radius", [((40, 40, 40), 0.3, 6), ((37, 29, 23), 0.35, 6)] +
                         [((33, 40, 26), 0.3, r) for r in range(1, 6)])
def test_residual_from_definition(n3, h, radius, tol):
    R, Z, rho, floor = system(n3, h, radius)
    ctx = sparc.Context(n3, h, R, Z, np.zeros((4, 4)), veff=np.zeros(rho.size), rc_erf=1.0,
                        radius=radius)
    phi, it, rel, b = ctx.poisson(torch.from_numpy(rho).to("cuda:0"), tol=tol, want_b=True)
    ctx.close()
    assert rel <= tol
    f = rhs(rho, b.cpu().numpy(), n3, h, radius)
    assert residual(f, phi.cpu().numpy(), n3, h, radius) <= tol + 2.0 * floor
