"""The windows of the exact variant's single-source runs (next_window in
csrc/k_single.cu) on frames that put them to the test: distances that jump from
window to window (lines of low cost through high ground, walls, plateaus with
gaps), distances of neighbours beyond 32 bits, caps as tight as K = 1 makes them,
and costs up to the largest.  Lists and distances
equal the assignment maps of one match at a time, bit for bit."""

import numpy as np
import pytest

from paper_1501_02565_gb300 import native

pytestmark = pytest.mark.gpu


def _cost(kind, rng, H, W):
    if kind == "edges":
        c = 1e-3 + np.maximum(rng.normal(0.0, 0.02, (H, W)), 0.0)
        c[rng.random((H, W)) < 0.05] += 0.7
    elif kind == "high":
        c = rng.uniform(0.3, 0.99, (H, W))
    elif kind == "wide":
        c = rng.uniform(0.0, 1.99, (H, W))
    elif kind == "mid":
        c = rng.uniform(0.05, 0.5, (H, W))
    elif kind == "walls":
        c = rng.uniform(0.002, 0.02, (H, W))
        step = rng.integers(7, 30)
        c[:, ::step] = 1.4
        c[::step] = 1.0
        c[rng.integers(0, H)] = 0.01
    elif kind == "blob":
        c = np.full((H, W), 0.01)
        y, x = rng.integers(0, H), rng.integers(0, W)
        c[max(0, y - 20):y + 20, max(0, x - 30):x + 30] = rng.uniform(0.5, 1.9)
        c = np.minimum(c + rng.uniform(0, 0.01, (H, W)), 1.98)
    elif kind == "lines":
        c = rng.uniform(0.3, 1.2, (H, W))
        for _ in range(6):
            c[rng.integers(0, H)] = 0.005
            c[:, rng.integers(0, W)] = 0.005
    else:   # "spikes"
        c = rng.uniform(0.001, 0.05, (H, W))
        c[rng.random((H, W)) < 0.3] = 1.95
    return c.astype(np.float32)


KINDS = ("edges", "high", "wide", "mid", "walls", "blob", "lines", "spikes")


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("K", (1, 3, 20))
def test_lists_hold_the_single_match_maps(kind, K):
    import torch
    ref = native.EpicInterp(0, sweep=0)   # the apron tiles keep the unit 2^-31 on every frame
    for case in range(6):
        rng = np.random.default_rng([KINDS.index(kind), K, case])
        H, W, N = int(rng.integers(20, 200)), int(rng.integers(20, 300)), int(rng.choice((20, 60, 120)))
        area = (min(H, 30), min(W, 30)) if case % 3 == 2 else (H, W)   # (matches in a corner)
        flat = np.unique(rng.integers(0, area[0], N) * W + rng.integers(0, area[1], N))
        xy = np.stack([flat % W, flat // W], 1).astype(np.float32)
        N, k = len(xy), min(K, len(xy))
        M = torch.from_numpy(np.concatenate([xy, xy + 1], 1)).cuda()
        C = torch.from_numpy(_cost(kind, rng, H, W)).cuda()
        eng = native.EpicInterp(0)
        _, idx, dist = eng.exact(C, M, k, 1.0, with_knn=True)
        eng.close()
        D = torch.empty(N, H * W, device="cuda")
        out = torch.empty(H, W, 2, device="cuda")
        for m in range(N):
            ref.run(C, M[m:m + 1], 1, 1.0, out)
            D[m] = ref.get_labels(0, H, W)[1].reshape(-1)
        # by (distance, index): a stable sort
        want, order = torch.sort(D.T, dim=1, stable=True)
        assert torch.equal(dist.reshape(-1, k), want[:, :k]), (H, W, N)
        assert torch.equal(idx.reshape(-1, k).long(), order[:, :k]), (H, W, N)
    ref.close()
