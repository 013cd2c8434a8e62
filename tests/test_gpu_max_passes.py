"""max_passes bounds the relaxation of the whole run, not the share of a CTA:
frames whose changes go to and fro between a few tiles, far more often than the
frame's average, end within the passes that their tile solves in all come to;
and a bound below these ends with EPIC_ERR_NOT_CONVERGED, after which the handle
goes on."""

import pytest

from paper_1501_02565_gb300 import native
from test_gpu_relax_solve import _pair

pytestmark = pytest.mark.gpu


def _run(C, M, **cfg):
    import torch
    eng = native.EpicInterp(0, **cfg)
    flow = eng.run(C, M, 8, 1.0)
    rc, passes = eng.sync_status(), eng.get_passes()
    eng.close()
    return rc, passes, flow


@pytest.mark.parametrize("kind,H,W,N", [("edges", 436, 1024, 5), ("high", 436, 1024, 50), ("wide", 436, 1024, 5000),
                                        ("wide", 130, 200, 2), ("high", 60, 130, 3)])
def test_the_bound_is_of_the_whole_run(kind, H, W, N):
    import torch
    C, M = (torch.from_numpy(a).cuda() for a in _pair(kind, H, W, N, 5))
    rc, passes, want = _run(C, M)
    assert rc == native.EPIC_OK
    # (either phase of the relaxation solves less than both together)
    rc, _, got = _run(C, M, max_passes=max(2, (passes + 2) // 2 + 1))
    assert rc == native.EPIC_OK and torch.equal(got, want)


def test_a_bound_too_low():
    import torch
    C, M = (torch.from_numpy(a).cuda() for a in _pair("edges", 436, 1024, 5, 5))
    eng = native.EpicInterp(0, max_passes=1)
    eng.run(C, M, 8, 1.0)
    assert eng.sync_status() == native.EPIC_ERR_NOT_CONVERGED
    C1, M1 = (torch.from_numpy(a).cuda() for a in _pair("edges", 16, 64, 3, 6))   # one tile
    eng.run(C1, M1, 8, 1.0)
    assert eng.sync_status() == native.EPIC_OK
    eng.close()
