"""epic_geodesic_labels_noalloc, which runs the tile relaxation of k_relax.cu
with the distance unit held at 2^-31, against the apron-tile relaxation
(k_dt.cu), which has that unit on every frame: labels and distances equal bit
for bit, at frames narrower and lower than a tile, ragged ones, the largest
that the entry point takes, plateaus of cost zero, and distances and costs so
large that the interpolator would take a coarser unit.  Costs of 2 and more and
those that are no cost stay refused."""

import numpy as np
import pytest

from paper_1501_02565_gb300 import native
from test_gpu_relax_solve import _pair
from test_zz_no_alloc import _noalloc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,H,W,N", [
    ("edges", 1, 1, 1), ("edges", 5000, 1, 7), ("flat", 3, 700, 5), ("zero", 33, 65, 20),
    ("wide", 131, 257, 60), ("edges", 436, 1024, 5000), ("high", 700, 748, 2),
    ("edges", 8192, 64, 900), ("high", 65536, 2, 3), ("zero", 512, 1024, 32768),
])
def test_same_as_the_apron_tiles(kind, H, W, N):
    import torch
    C, M = (torch.from_numpy(a).cuda() for a in _pair(kind, H, W, N, 5))
    rc, L, D = _noalloc(native.load(), C, M, H, W, M.shape[0])
    eng = native.EpicInterp(0, sweep=0)
    eng.run(C, M, 1, 1.0)
    Lr, Dr = (t.cpu().numpy().reshape(H, W) for t in eng.get_labels(0, H, W))
    eng.close()
    assert rc == native.EPIC_OK
    assert np.array_equal(L, Lr)
    assert np.array_equal(D.view(np.int32), Dr.view(np.int32))


@pytest.mark.parametrize("bad", [2.0, -1e-3, float("nan"), float("inf")])
def test_bad_costs_are_refused(bad):
    import torch
    C, M = _pair("edges", 40, 70, 9, 6)
    C[17, 33] = bad
    rc, _, _ = _noalloc(native.load(), torch.from_numpy(C).cuda(), torch.from_numpy(M).cuda(), 40, 70, 9)
    assert rc == native.EPIC_ERR_INVALID
