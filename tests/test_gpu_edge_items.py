"""The graph's edges (edges_kernel in csrc/k_graph.cu) where its work items
change: parts of a tile, tiles and stacks of tiles (chosen by the number of
tiles), tile heights that do not divide into parts, tiles taller than the rows
staged at once, frames narrower than a warp and cut tiles.  The set of edges must be the set of label pairs that touch in
the GPU's own assignment map, and each weight the smallest D(p) + step + D(q)
along the border, computed here in float64 from the float32 distances (parity.py's
tolerance of weights)."""

import numpy as np
import pytest

from parity import W_ATOL, W_RTOL, run_gpu

pytestmark = pytest.mark.gpu


def _edges(C, L, D):
    C, D = C.astype(np.float64), D.astype(np.float64)
    H, W = C.shape
    keys, ws = [], []
    for dx, dy in ((1, 0), (-1, 1), (0, 1), (1, 1)):
        p = (slice(0, H - dy), slice(max(0, -dx), W - max(0, dx)))
        q = (slice(dy, H), slice(max(0, dx), W + min(0, dx)))
        touch = L[p] != L[q]
        lo, hi = np.minimum(L[p], L[q])[touch], np.maximum(L[p], L[q])[touch]
        step = np.hypot(dx, dy) * (C[p] + C[q]) / 2
        keys.append(lo.astype(np.int64) << 32 | hi)
        ws.append((D[p] + step + D[q])[touch])
    keys, ws = np.concatenate(keys), np.concatenate(ws)
    uniq, inv = np.unique(keys, return_inverse=True)
    w = np.full(uniq.shape, np.inf)
    np.minimum.at(w, inv, ws)
    return uniq, w


@pytest.mark.parametrize("H,W,N,cfg", [
    (1, 40, 9, {}), (37, 5, 11, {}), (128, 256, 500, {}), (83, 150, 300, {"tile_w": 64, "tile_h": 1, "sweep": 2}),
    (100, 131, 300, {"tile_w": 64, "tile_h": 7, "sweep": 2}), (131, 300, 900, {"tile_w": 256, "tile_h": 16, "sweep": 0}),
    (61, 90, 200, {"tile_w": 8, "tile_h": 8, "sweep": 0}), (436, 1024, 5000, {}), (375, 1242, 4000, {}),
    (1100, 1500, 9000, {}), (1300, 2048, 20000, {}), (700, 64, 2, {}),
    (150, 300, 400, {"tile_w": 256, "tile_h": 70, "apron": 0, "sweep": 0}),
    (300, 200, 300, {"tile_w": 64, "tile_h": 256, "apron": 0, "sweep": 0}),
])
def test_edges_of_the_assignment_map(H, W, N, cfg):
    rng = np.random.default_rng(H + W)
    C = (1e-3 + np.maximum(rng.normal(0.0, 0.02, (H, W)), 0.0)).astype(np.float32)
    C[rng.random((H, W)) < 0.05] += np.float32(0.7)
    flat = rng.choice(H * W, N, replace=False)
    xy = np.stack([flat % W, flat // W], 1).astype(np.float32)
    M = np.concatenate([xy, xy + 1], 1).astype(np.float32)
    g = run_gpu((C, M), K=4, a=1.0, **cfg)
    keys, w = _edges(C, g["L"].reshape(H, W), g["D"].reshape(H, W))
    got = np.minimum(g["em"], g["en"]).astype(np.int64) << 32 | np.maximum(g["em"], g["en"])
    order = np.argsort(got)
    assert np.array_equal(got[order], keys)
    assert (np.abs(g["ew"][order] - w) <= W_RTOL * w + W_ATOL).all()
