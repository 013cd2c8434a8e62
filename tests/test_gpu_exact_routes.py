"""The exact variant's single-source runs by each of their routes (single_few and
the rules beside it in csrc/epic_internal.cuh): few matches by pairs, caps that
reach far by pairs or by tiles with 64-bit keys (with pools that do not hold a
match's tiles too), and by tiles on frames of more tiles than the per-CTA tables
hold.  Lists and distances equal the assignment maps of one match at a time, bit
for bit.  And costs a hundred times higher, which change nothing but the scale,
do not take many times as long."""

import time

import numpy as np
import pytest

from paper_1501_02565_gb300 import native
from test_gpu_exact_groups import _cost, _matches, _spread

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,H,W,N,K,budget", [
    ("edges", 530, 2100, 70, 2, 0),                 # 561 tiles, by tiles
    ("edges", 530, 2101, 20, 20, 0),                # by pairs: few
    ("high", 301, 701, 60, 9, 0),                   # by pairs: far
    ("high", 301, 701, 60, 9, 3 * 301 * 701 * 8),   # a few pairs at a time
    ("high", 301, 700, 520, 60, 0),                 # by tiles, 64-bit keys
    ("wide", 97, 131, 520, 30, 0),
    ("high", 301, 700, 530, 60, 2 * 110 * 16384),   # pools that do not hold a match's tiles
    ("edges", 40, 70, 1, 1, 0),
    # 17 pools of 64 of the 110 tiles, which most matches outgrow
    ("edges", 301, 701, 20, 20, 10 * 110 * 16384),   # by pairs
    ("edges", 301, 701, 20, 7, 10 * 110 * 16384),    # by tiles
    ("zero", 301, 701, 60, 9, 10 * 110 * 16384),     # by pairs
    ("zero", 301, 701, 24, 9, 0),
])
def test_lists_hold_the_single_match_maps(kind, H, W, N, K, budget):
    import torch
    rng = np.random.Generator(np.random.PCG64(H + W + N))
    M = _matches(rng, _spread(rng, H, W, N))
    C = np.zeros((H, W), np.float32) if kind == "zero" else _cost(kind, rng, H, W)
    C = torch.from_numpy(C).cuda()
    eng = native.EpicInterp(0, exact_chunk_bytes=budget)
    for _ in range(2):   # the second call finds the first one's buffers
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


@pytest.mark.parametrize("H,W,N,K,pixels", [
    (45, 70, 60, 20, 60),
    (45, 70, 60, 60, 7),       # several matches on a pixel
    (45, 70, 600, 30, 600),    # more candidates than shared memory holds
    (301, 701, 300, 40, 300),
])
def test_equal_distances_go_by_index(H, W, N, K, pixels):
    import torch
    rng = np.random.Generator(np.random.PCG64(H + N + pixels))
    xy = _spread(rng, H, W, pixels)[np.arange(N) % pixels]
    C = torch.zeros(H, W, device="cuda")
    eng = native.EpicInterp(0)
    _, idx, dist = eng.exact(C, torch.from_numpy(_matches(rng, xy)).cuda(), K, 1.0, with_knn=True)
    eng.close()
    assert not dist.any()
    assert torch.equal(idx.reshape(-1, K).long(), torch.arange(K, device="cuda").expand(H * W, K))


def test_costs_of_zero_do_not_take_many_times_as_long():
    # (59 ms against 17 when the candidates of a group came in any order)
    import torch
    rng = np.random.Generator(np.random.PCG64(9))
    H, W, N, K = 436, 1024, 300, 200
    M = torch.from_numpy(_matches(rng, _spread(rng, H, W, N))).cuda()
    times = []
    for c in (1e-3, 0.0):
        C = torch.full((H, W), c, device="cuda")
        eng = native.EpicInterp(0)
        best = float("inf")
        for _ in range(4):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            eng.exact(C, M, K, 1.0)
            best = min(best, time.perf_counter() - t0)
        eng.close()
        times.append(best)
    assert times[1] < 2 * times[0], times


@pytest.mark.parametrize("c", [0.0, 1e-3])
def test_a_few_matches_more_than_there_are_full_pools(c):
    # 85 pools of every tile fit the budget.  By tiles most of 100 matches outgrow
    # theirs and run twice.
    import torch
    rng = np.random.Generator(np.random.PCG64(10))
    H, W, K = 1000, 1500, 50
    C = torch.full((H, W), c, device="cuda")
    times = []
    for N in (85, 100):
        M = torch.from_numpy(_matches(rng, _spread(rng, H, W, N))).cuda()
        eng = native.EpicInterp(0)
        best = float("inf")
        for _ in range(4):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            eng.exact(C, M, K, 1.0)
            best = min(best, time.perf_counter() - t0)
        eng.close()
        times.append(best)
    assert times[1] < 1.45 * times[0], times


@pytest.mark.parametrize("N,K", [(10, 10), (100, 10), (600, 10)])
def test_high_costs_do_not_take_many_times_as_long(N, K):
    # (by windows 85 ms against 2 ms for N = 100)
    import torch
    rng = np.random.Generator(np.random.PCG64(N))
    H, W = 436, 1024
    M = torch.from_numpy(_matches(rng, _spread(rng, H, W, N))).cuda()
    C = torch.from_numpy(_cost("high", rng, H, W)).cuda()
    times = []
    for c in (0.01 * C, C):
        eng = native.EpicInterp(0)
        best = float("inf")
        for _ in range(4):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            eng.exact(c, M, K, 1.0)
            best = min(best, time.perf_counter() - t0)
        eng.close()
        times.append(best)
    assert times[1] < 8 * times[0], times
