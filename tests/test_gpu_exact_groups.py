"""The exact variant's kernels (csrc/k_single.cu, csrc/k_exact.cu) where they
change their path: groups of pixels with more candidates than shared memory
holds, matches outside the frame (Euclidean), distances beyond the 32-bit
window of a tile and steps longer than it, a budget of one key map, pools that
do not hold a match's tiles, frames of more tiles than the per-CTA tables hold, and runs that need more distance tiles
than are first set aside.

Against the FP64 oracle with the tolerances of test_gpu_exact.py, or, where the
oracle would be slow, against the assignment map of one match at a time, which
shares the unique fixed point of the same integer steps: equal bit for bit."""

import numpy as np
import pytest

from paper_1501_02565_gb300 import native
from test_gpu_exact import _check

pytestmark = pytest.mark.gpu


def _cost(kind, rng, H, W):
    if kind == "high":        # distances far beyond one cost unit
        return rng.uniform(0.3, 0.99, (H, W)).astype(np.float32)
    if kind == "wide":        # steps beyond 32 bits, narrow windows
        return rng.uniform(0.05, 1.99, (H, W)).astype(np.float32)
    if kind == "walls":       # strong edges with passages, weak texture between
        c = rng.uniform(0.002, 0.02, (H, W))
        c[:, ::9] = 1.4
        c[::7, ::9] = 0.01
        return c.astype(np.float32)
    c = 1e-3 + np.maximum(rng.normal(0.0, 0.02, (H, W)), 0.0)   # "edges"
    c[rng.random((H, W)) < 0.05] += 0.7
    return c.astype(np.float32)


def _matches(rng, xy):
    uv = rng.normal(0.0, 5.0, xy.shape)
    return np.concatenate([xy, xy + uv], 1).astype(np.float32)


def _spread(rng, H, W, N):
    flat = rng.choice(H * W, N, replace=False)
    return np.stack([flat % W, flat // W], 1).astype(np.float64)


@pytest.mark.parametrize("kind,H,W,N,K,cfg", [
    ("high", 41, 67, 60, 20, {}),
    ("wide", 37, 131, 40, 12, {}),
    ("wide", 70, 66, 25, 25, {}),
    ("walls", 66, 129, 90, 30, {}),
    ("edges", 33, 65, 50, 10, {"exact_chunk_bytes": 1}),
])
def test_geodesic_windows(kind, H, W, N, K, cfg):
    rng = np.random.Generator(np.random.PCG64(H * W + N))
    C = _cost(kind, rng, H, W)
    _check(C, _matches(rng, _spread(rng, H, W, N)), K, 1.0, "geodesic", **cfg)


@pytest.mark.parametrize("metric", ["geodesic", "euclidean"])
@pytest.mark.parametrize("K", [3, 300])
def test_dense_cluster(metric, K):
    # 620 of 640 matches in 26 x 26 pixels
    rng = np.random.Generator(np.random.PCG64(77))
    H, W = 45, 70
    xy = np.concatenate([_spread(rng, 26, 26, 620) + 5.0, np.stack(
        [rng.permutation(30)[:20] + 38.0, rng.permutation(40)[:20].astype(float)], 1)])
    _check(_cost("edges", rng, H, W), _matches(rng, xy), K, 0.5, metric)


def test_euclidean_matches_outside_the_frame():
    rng = np.random.Generator(np.random.PCG64(78))
    H, W = 35, 52
    xy = rng.permutation(4000)[:70]
    xy = np.stack([xy % 80 - 14.0, xy // 80 - 8.0], 1)
    C = _cost("edges", rng, H, W)
    _check(C, _matches(rng, xy), 9, 1.0, "euclidean")


@pytest.mark.parametrize("kind,H,W,N,K,budget", [
    ("edges", 530, 2100, 24, 2, 0),    # 33 x 17 tiles
    ("high", 300, 701, 40, 40, 0),     # every tile of every match: 4400 distance tiles
    ("high", 300, 701, 40, 40, 2 * 110 * 16384),   # three pools of 73 of the 110 tiles: all run again
    ("edges", 300, 701, 300, 20, 2 * 110 * 16384),
])
def test_lists_hold_the_single_match_maps(kind, H, W, N, K, budget):
    import torch
    rng = np.random.Generator(np.random.PCG64(H + W))
    M = _matches(rng, _spread(rng, H, W, N))
    C = torch.from_numpy(_cost(kind, rng, H, W)).cuda()
    eng = native.EpicInterp(0, exact_chunk_bytes=budget)
    _, idx, dist = eng.exact(C, torch.from_numpy(M).cuda(), K, 1.0, with_knn=True)
    eng.close()
    eng = native.EpicInterp(0, sweep=0)   # the apron tiles keep the unit 2^-31 on every frame
    D = torch.empty(N, H * W, device="cuda")
    out = torch.empty(H, W, 2, device="cuda")
    for m in range(N):
        eng.run(C, torch.from_numpy(M[m:m + 1]).cuda(), 1, 1.0, out)
        D[m] = eng.get_labels(0, H, W)[1].reshape(-1)
    eng.close()
    # by (distance, index): a stable sort
    want, order = torch.sort(D.T, dim=1, stable=True)
    assert torch.equal(dist.reshape(-1, K), want[:, :K])
    assert torch.equal(idx.reshape(-1, K).long(), order[:, :K])
