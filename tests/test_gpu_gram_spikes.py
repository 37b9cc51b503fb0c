"""The 47-bit contraction of a column whose largest values stand out: in every 128-row chunk one
value 1, 126 values 2^-22 and a zero. All are single digits, so their products are exact in the
digits, and the small ones' sum lies in the last kept classes.

The norm of the rotated column shows M_s: M_s itself within 2^-50 per chunk sum, the coefficient
1 / sqrt(M_s) rounded to 47 bits (2^-47 in the square), so within 2^-45 of one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from paper_1603_04334_gb300 import sparc  # noqa: E402


@pytest.mark.parametrize("n3", [(16, 16, 16), (32, 32, 40)])
def test_norm(n3):
    nd = n3[0] * n3[1] * n3[2]
    Y = np.full((nd // 128, 128), 2.0 ** -22)
    Y[:, 0], Y[:, 64] = 1.0, 0.0
    X = torch.from_numpy(Y.reshape(1, nd).copy()).to("cuda:0")
    ctx = sparc.Context(n3, 0.5, veff=np.zeros(nd))
    ctx.orth_rr(X)
    ctx.close()
    x = X.cpu().numpy().astype(np.longdouble)
    assert abs(float((x * x).sum() - 1)) <= 2.0 ** -45
