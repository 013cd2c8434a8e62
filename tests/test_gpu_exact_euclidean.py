"""The Euclidean exact variant where its groups change their way (scan_all and the
looks of fit_kernel in csrc/k_exact.cu): a few matches, numbers of matches around
the rule, dense matches whose first look takes in more than shared memory holds,
denser ones that need more, and matches crowded into a corner.  Lists and
distances equal those of a full sort, bit for bit (pixel centres are integers, so
the squared distances are exact in float32).  And dense matches do not take the
time of a scan of all of them."""

import time

import numpy as np
import pytest

from paper_1501_02565_gb300 import native

pytestmark = pytest.mark.gpu


def _frame(H, W, N, corner, seed):
    import torch
    rng = np.random.default_rng(seed)
    h, w = (min(H, 40), min(W, 40)) if corner else (H, W)
    flat = rng.permutation(h * w)[:N]
    xy = np.stack([flat % w, flat // w], 1).astype(np.float32)
    M = np.concatenate([xy, xy + rng.normal(0, 5, xy.shape)], 1).astype(np.float32)
    return torch.full((H, W), 0.01, device="cuda"), torch.from_numpy(M).cuda()


@pytest.mark.parametrize("H,W,N,K,corner", [
    (45, 70, 1, 1, False), (45, 70, 7, 7, False), (45, 70, 34, 10, False), (45, 70, 35, 10, False),
    (45, 70, 80, 80, False), (45, 70, 81, 81, False), (33, 50, 500, 30, False), (33, 50, 600, 30, False),
    (120, 130, 5400, 32, False), (100, 90, 4500, 32, False), (100, 90, 9000, 4, False), (100, 90, 9000, 32, False),
    (90, 300, 1500, 20, True), (90, 300, 700, 100, True),
])
def test_lists_are_those_of_a_full_sort(H, W, N, K, corner):
    import torch
    C, M = _frame(H, W, N, corner, N + K)
    eng = native.EpicInterp(0)
    _, idx, dist = eng.exact(C, M, K, 1.0, "euclidean", with_knn=True)
    eng.close()
    y, x = torch.meshgrid(torch.arange(H, device="cuda"), torch.arange(W, device="cuda"), indexing="ij")
    d2 = (x.reshape(-1, 1) - M[None, :, 0]) ** 2 + (y.reshape(-1, 1) - M[None, :, 1]) ** 2
    want, order = torch.sort(d2, dim=1, stable=True)   # by (distance, index)
    assert torch.equal(idx.reshape(-1, K).long(), order[:, :K])
    assert torch.equal(dist.reshape(-1, K), want[:, :K].sqrt())


def test_dense_matches_are_not_scanned():
    # (a match for four pixels, K = 100: 326 ms against 1.0 ms for K = 32 when
    # groups whose first look took in too much were scanned)
    import torch
    C, M = _frame(436, 1024, 436 * 256, False, 1)
    times = []
    for K in (32, 100):
        eng = native.EpicInterp(0)
        best = float("inf")
        for _ in range(4):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            eng.exact(C, M, K, 1.0, "euclidean")
            best = min(best, time.perf_counter() - t0)
        eng.close()
        times.append(best)
    assert times[1] < 20 * times[0], times
