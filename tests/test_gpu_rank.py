"""Ranking and fused inference at the sizes where their tiles end: the k
smallest of n predictions are numpy's (ties by index), an ensemble's ranking
is the mean's, rows beyond the last full tile and descriptor rows at any
4-byte alignment give the same predictions."""
import math

import numpy as np
import pytest

from paper_2304_09953_gb300 import native as N

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def nets():
    hs = [N.ligate_surrogate_create(None, 40 + m) for m in range(10)]
    yield hs
    for h in hs:
        N.ligate_surrogate_destroy(h)


@pytest.mark.parametrize("n,keep,m", [(1, 1.0, 1), (2, 0.5, 10), (127, 1.0, 1), (128, 0.3, 2), (129, 1.0, 9),
                                      (2048, 1.0, 1), (2049, 1.0, 1), (4096, 0.01, 3), (16385, 1.0, 1),
                                      (40000, 0.418, 1), (131073, 0.02, 1)])
def test_rank_is_the_sorted_prediction(nets, n, keep, m):
    rng = np.random.default_rng(n)
    x = rng.normal(size=(n, 256)).astype(np.float32)
    x[n // 3:2 * n // 3] = x[0]  # equal predictions: ties go to the smaller index
    desc = torch.from_numpy(x).cuda()
    k = math.ceil(n * keep - 1e-9)
    idx = torch.full((max(k, 1) + 1,), -7, dtype=torch.int32, device="cuda")
    pred = torch.empty(n, dtype=torch.float32, device="cuda")
    if m == 1:
        N.ligate_surrogate_rank(nets[0], desc, n, keep, idx, pred)
    else:
        N.ligate_surrogate_rank_ensemble(nets[:m], desc, n, keep, idx, pred)
    p = pred.cpu().numpy()
    got = idx.cpu().numpy()
    assert np.array_equal(got[:k], np.lexsort((np.arange(n), p))[:k]) and got[k] == -7
    one = torch.empty(n, dtype=torch.float32, device="cuda")
    mean = np.zeros(n, np.float64)
    for h in nets[:m]:
        N.ligate_surrogate_predict(h, desc, n, one)
        mean += one.cpu().numpy().astype(np.float64) / m
    assert np.max(np.abs(mean - p)) <= 1e-6 * np.max(np.abs(p))  # the mean's own FP32 rounding
    if n <= 4096:  # the same rows behind a 4-byte offset
        buf = torch.empty(n * 256 + 1, dtype=torch.float32, device="cuda")
        buf[1:] = desc.reshape(-1)
        N.ligate_surrogate_predict(nets[0], desc, n, one)
        two = torch.empty_like(one)
        N.ligate_surrogate_predict(nets[0], buf.data_ptr() + 4, n, two)
        assert torch.equal(one, two)
