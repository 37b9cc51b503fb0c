"""Equal and nearly equal eigenvalues where the dense step has more than one pair of 32-column
blocks and a third refinement (above 128 states), and products in FP32 pairs (above 256): the
problem, the reference and the tolerances of test_gpu_dense.test_close_eigenvalues."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from test_gpu_dense import test_close_eigenvalues as check_close_eigenvalues  # noqa: E402


@pytest.mark.parametrize("ns,spread", [(130, 0.0), (130, 1e-9), (300, 0.0), (300, 1e-9), (300, 1e-6)])
def test_multiplets(ns, spread):
    check_close_eigenvalues(ns, spread)
