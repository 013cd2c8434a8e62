"""Seed binning (csrc/k_prepare.cu) on either side of the largest frame whose
tile counts fit in shared memory (4096 tiles), with several matches per thread
and duplicates: the assignment map equals the apron tiles' (few tiles), bit for
bit, and a match outside the frame is refused."""

import numpy as np
import pytest

from paper_1501_02565_gb300 import native
from test_gpu_relax_solve import _labels, _pair, _same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,N", [(4096, 64, 3000), (4097, 50, 5000), (436, 1024, 9000), (256, 1024, 2500)])
def test_tiles_around_the_shared_table(H, W, N):
    C, M = _pair("edges", H, W, N, 3)
    M = np.concatenate([M, M[:7]])   # duplicates: the smaller index owns the pixel
    _same(_labels([(C, M)], tile_w=64, tile_h=1, sweep=2), _labels([(C, M)], sweep=0))


@pytest.mark.parametrize("m", [0, 2047, 2999])
def test_a_match_outside_is_refused(m):
    import torch
    C, M = _pair("edges", 300, 200, 3000, 4)
    M[m, 0] = 200.0
    eng = native.EpicInterp(0)
    eng.run(torch.from_numpy(C).cuda(), torch.from_numpy(M).cuda(), 8, 1.0)
    with pytest.raises(native.EpicError):
        eng.sync()
    eng.close()
