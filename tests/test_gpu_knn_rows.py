"""The K-NN search (csrc/k_knn_fit.cu) takes each node's adjacency row from the
entry that led to it, packed into a word: 22 bits for its start and 10 for its
degree, or a mark for what does not fit.  Lists and distances against the oracle
on the GPU's own graph, around the largest degree that fits (1022): hubs ringed
by as many matches, whose frontiers and batches also go far beyond a warp."""

import numpy as np
import pytest

from parity import check_knn, run_gpu

pytestmark = pytest.mark.gpu


def _hub(n, R, side, seed):
    # a match ringed by n others, one pixel each, with a cheap disk between, so
    # that the hub's cell touches the cells of (nearly) all of them
    rng = np.random.default_rng(seed)
    c = side // 2
    C = 0.5 + rng.uniform(-0.01, 0.01, size=(side, side))
    ys, xs = np.mgrid[0:side, 0:side]
    C[(xs - c) ** 2 + (ys - c) ** 2 < (R - 3.0) ** 2] *= 0.001
    ang = np.linspace(0.0, 2.0 * np.pi, n, endpoint=False)
    ring = np.stack([np.round(c + R * np.cos(ang)), np.round(c + R * np.sin(ang))], 1)
    p = np.concatenate([[[c, c]], np.unique(ring, axis=0)])
    M = np.stack([p[:, 0], p[:, 1], p[:, 0] + 1.5, p[:, 1] - 0.5], 1)
    return C.astype(np.float32), M.astype(np.float32)


@pytest.mark.parametrize("n,R,side,K,least", [(900, 160.0, 352, 20, 600), (1500, 236.0, 512, 40, 1023),
                                              (1700, 300.0, 640, 3, 1023), (1500, 236.0, 512, 200, 1023)])
def test_rows_around_the_largest_packed_degree(n, R, side, K, least):
    C, M = _hub(n, R, side, n)
    g = run_gpu((C, M), K=K, a=0.05)
    deg = np.bincount(np.r_[g["em"], g["en"]], minlength=len(M))
    print(f"\n[rows] {len(M)} matches, largest degree {deg.max()}")
    assert deg.max() > least
    check_knn(M, g, {})
