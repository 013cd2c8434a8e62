"""Pairs of high costs, whose relaxation is the settling alone (settles_only in
csrc/epic_internal.cuh): the assignment maps of batches in which they stand
beside others, pruned runs (whose tables are prepared twice) and means around
the line equal the apron tiles', bit for bit; and they take no longer than
frames of low cost, as with the kernel before the phases."""

import numpy as np
import pytest

from paper_1501_02565_gb300 import native
from test_gpu_relax_solve import _labels, _pair, _same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(97, 322, 300), (33, 65, 4), (130, 200, 2)], [(470, 640, 2500)] * 5])
def test_beside_other_pairs(sizes):
    kinds = ("high", "edges", "wide", "zero", "flat")
    pairs = [_pair(kinds[i % 5], H + i, W + i, N, i) for i, (H, W, N) in enumerate(sizes + sizes[:2])]
    _same(_labels(pairs), [_labels([p], sweep=0)[0] for p in pairs])


@pytest.mark.parametrize("tile_h", (1, 5, 8, 16, 32))
def test_tile_heights(tile_h):
    pairs = [_pair("high", 101, 201, 150, 7)]
    _same(_labels(pairs, tile_h=tile_h), _labels(pairs, sweep=0))


@pytest.mark.parametrize("mean", (0.13, 0.2499, 0.25, 0.2501, 0.5))
def test_means_around_the_line_and_pruning(mean):
    import torch
    rng = np.random.default_rng(8)
    _, M = _pair("flat", 150, 260, 300, 9)
    C = (mean * rng.uniform(0.9, 1.1, (150, 260))).astype(np.float32)
    _same(_labels([(C, M)]), _labels([(C, M)], sweep=0))
    C, M = torch.from_numpy(C).cuda(), torch.from_numpy(M).cuda()
    flows = []
    for sweep in (2, 0):
        eng = native.EpicInterp(0, prune=1, sweep=sweep)
        flows.append(eng.run(C, M, 16, 1.0))
        eng.sync()
        eng.close()
    assert torch.equal(*flows)


def test_constant_costs_take_the_same_time_at_any_height():
    # the frames differ in scale alone: 308 us of relaxation for either with the
    # row-closure kernel, 286 and 404 us when both went through all phases
    import torch
    _, M = _pair("flat", 436, 1024, 5000, 1)
    times = []
    for c in (1e-3, 1.0):
        C = torch.full((436, 1024), c, device="cuda")
        eng = native.EpicInterp(0, max_pairs=8)
        items = [(C, torch.from_numpy(M).cuda(), 16, 1.0, torch.empty(436, 1024, 2, device="cuda"))
                 for _ in range(8)]
        best = float("inf")
        for _ in range(12):
            eng.enable_stage_timing(True)
            eng.run_batch(items)
            eng.sync()
            best = min(best, eng.stage_times()[0]["relax"])
        eng.close()
        times.append(best)
    assert times[1] < 1.25 * times[0], times
