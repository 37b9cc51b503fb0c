"""The batched FP32 filter with two rows per thread (more items than two CTAs per SM hold) on
clusters whose number of rows is odd, one row, or ends a row past a tile: equal to the filter of
each cluster (2e-6 of the largest value, as in test_gpu_batch.py), nothing written past a column."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytestmark = [pytest.mark.gpu, pytest.mark.skip(reason="no CUDA device")]

from paper_1603_04334_gb300 import batching, sparc  # noqa: E402


@pytest.mark.parametrize("shapes", [
    [((44, 29, 23), 60), ((32, 17, 40), 70), ((20, 33, 18), 80), ((36, 1, 30), 50)],
    [((24, 15, 9), 200), ((64, 47, 12), 60)]])
def test_odd_rows(shapes):
    items = sum(ns * -(-n[0] // 32) * -(-n[1] // 16) for n, ns in shapes)
    assert items > 2 * 152                     # at least one z range each
    g = np.random.default_rng(1)
    degree, pad = 7, 8
    ctxs, X, one = [], [], []
    for n, ns in shapes:
        nd = n[0] * n[1] * n[2]
        ctxs.append(sparc.Context(n, 0.45, veff=g.uniform(-3.0, 1.0, nd)))
        x = torch.full((ns, -(-nd // 4) * 4 + pad), 7.0, dtype=torch.float32, device="cuda:0")
        x[:, :nd] = torch.from_numpy(g.uniform(-0.5, 0.5, (ns, nd))).to("cuda:0", torch.float32)
        X.append(x)
    B = [(6.0 + i, 50.0 + i, -4.0) for i in range(len(shapes))]
    one = [x.clone() for x in X]
    W = [torch.full_like(x, 7.0) for x in X]
    batch = batching.Batch(ctxs)
    batch.filter(X, W, degree, B)
    torch.cuda.synchronize()
    for (n, ns), ctx, x, w, r, b in zip(shapes, ctxs, X, W, one, B):
        nd = n[0] * n[1] * n[2]
        ctx.cheb_filter(r, torch.empty_like(r), degree, *b)
        got, ref = x[:, :nd].double(), r[:, :nd].double()
        assert (got - ref).abs().max() <= 2e-6 * ref.abs().max()
        assert torch.all(x[:, nd:] == 7.0) and torch.all(w[:, nd:] == 7.0)
    batch.close()
    for c in ctxs:
        c.close()
