"""The K-NN search (csrc/k_knn_fit.cu) among edges of weight zero, where every step
settles the smallest key alone: lists and distances against the oracle on the
GPU's own graph, with frontiers below and above the 64 entries that stay in
registers, neighbourhoods cut short and ones that exhaust the graph."""

import numpy as np
import pytest

from parity import check_knn, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("zeros", ["half", "plateau", "all"])
@pytest.mark.parametrize("H,W,N,K", [(40, 60, 12, 8), (64, 90, 150, 40), (64, 90, 150, 150), (120, 200, 300, 100)])
def test_lists_among_zero_weights(zeros, H, W, N, K):
    rng = np.random.default_rng(H + N + K)
    C = np.maximum(rng.normal(0.0, 0.02, (H, W)), 0.0)
    if zeros == "plateau":
        C += 1e-3
        C[H // 4:H // 2, W // 5:] = 0.0
    if zeros == "all":
        C[:] = 0.0
    flat = rng.choice(H * W, N, replace=False)
    xy = np.stack([flat % W, flat // W], 1).astype(np.float64)
    M = np.concatenate([xy, xy + rng.normal(0.0, 3.0, xy.shape)], 1).astype(np.float32)
    g = run_gpu((C.astype(np.float32), M), K=K, a=0.5)
    check_knn(M, g, {})
