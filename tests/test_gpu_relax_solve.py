"""The tile relaxation (csrc/k_relax.cu) against the apron-tile relaxation
(csrc/k_dt.cu), which shares none of its solve: labels and distances of every
pixel must be equal, bit for bit, since both end at the unique fixed point of
the same integer step costs.

The cases are where the tile solve changes its path: frames narrower and lower
than a block or a tile, tiles cut by the image, tile heights that are not whole
blocks, odd row pitches, plateaus of cost zero (no strictly nearer parent),
distances beyond a tile's 32-bit window, diagonal weights beyond 32 bits, and
batches large enough to be solved in stacks of two tiles."""

import numpy as np
import pytest

from paper_1501_02565_gb300 import native

pytestmark = pytest.mark.gpu


def _cost(kind, rng, H, W):
    if kind == "flat":
        return np.full((H, W), 1e-3, np.float32)
    if kind == "zero":        # plateaus of cost zero among weak texture
        c = np.maximum(rng.normal(0.0, 0.02, (H, W)), 0.0)
        c[H // 4: H // 2 + 1, :] = 0.0
        return c.astype(np.float32)
    if kind == "high":        # distances far beyond one cost unit
        return rng.uniform(0.3, 0.99, (H, W)).astype(np.float32)
    if kind == "wide":        # diagonal weights beyond 32 bits
        return rng.uniform(0.0, 1.99, (H, W)).astype(np.float32)
    c = 1e-3 + np.maximum(rng.normal(0.0, 0.02, (H, W)), 0.0)   # "edges"
    c[rng.random((H, W)) < 0.05] += 0.7
    return c.astype(np.float32)


def _pair(kind, H, W, N, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    flat = rng.choice(H * W, min(N, H * W), replace=False)
    xy = np.stack([flat % W, flat // W], 1).astype(np.float32)
    uv = rng.normal(0.0, 5.0, xy.shape).astype(np.float32)
    return _cost(kind, rng, H, W), np.concatenate([xy, xy + uv], 1).astype(np.float32)


def _labels(pairs, **cfg):
    import torch
    dev = torch.device("cuda", 0)
    eng = native.EpicInterp(0, max_pairs=len(pairs), **cfg)
    items = [(torch.from_numpy(C).to(dev), torch.from_numpy(M).to(dev), 8, 1.0,
              torch.empty(C.shape + (2,), device=dev)) for C, M in pairs]
    eng.run_batch(items)
    eng.sync()
    out = []
    for i, (C, _) in enumerate(pairs):
        L, D = eng.get_labels(i, *C.shape)
        out.append((L.cpu().numpy(), D.cpu().numpy()))
    eng.close()
    return out


def _same(a, b):
    for (La, Da), (Lb, Db) in zip(a, b):
        assert np.array_equal(La, Lb)
        assert np.array_equal(Da, Db)


@pytest.mark.parametrize("kind", ("edges", "flat", "zero", "high", "wide"))
@pytest.mark.parametrize("H, W, N", [(1, 1, 1), (1, 130, 3), (3, 2, 2), (17, 63, 9), (33, 65, 4),
                                     (50, 129, 40), (97, 322, 300), (130, 200, 2)])
def test_equals_the_apron_tile_relaxation(kind, H, W, N):
    pairs = [_pair(kind, H, W, N, 1000 + H + W)]
    _same(_labels(pairs), _labels(pairs, sweep=0))


@pytest.mark.parametrize("tile_h", (1, 2, 5, 8, 13, 16, 23, 32))
def test_every_tile_height(tile_h):
    pairs = [_pair("edges", 101, 201, 150, 7)]
    _same(_labels(pairs, tile_h=tile_h), _labels(pairs, sweep=0))


@pytest.mark.parametrize("kind", ("edges", "zero", "high"))
def test_stacked_batches(kind):
    # 1500 relaxation tiles of 64 x 16, heights that leave an odd tile row
    pairs = [_pair(kind, 470 + 7 * i, 640 + i, 2500, i) for i in range(5)]
    _same(_labels(pairs), [_labels([p])[0] for p in pairs])
    _same(_labels(pairs[:1]), _labels(pairs[:1], sweep=0))
