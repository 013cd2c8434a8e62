"""The waits between thread blocks of the relaxation and of the refinement give up
in time (see epic_selftest_wait_timeout), record EPIC_ERR_TIMEOUT and leave the
handle usable; and what such a report means for the handle: a run queued behind it
does nothing, one queued after it has been read goes on."""

import time

import pytest

from paper_1501_02565_gb300 import synth
from paper_1501_02565_gb300.native import EPIC_ERR_INVALID, EPIC_ERR_TIMEOUT, EPIC_OK, EpicInterp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", range(2, 7))
def test_waits_give_up(which):
    import torch
    p = synth.config_pair(1, 0)
    C, M = torch.from_numpy(p.C).cuda(), torch.from_numpy(p.matches).cuda()
    eng = EpicInterp(0)
    want = eng.run(C, M, p.K, p.a)
    assert eng.sync_status() == EPIC_OK
    for limit_ms in (1, 60):
        t0 = time.monotonic()
        assert eng.selftest_wait_timeout(which, limit_ms) == EPIC_ERR_TIMEOUT
        took = time.monotonic() - t0
        assert 0.001 * limit_ms <= took < 1.0 + 0.001 * limit_ms
    got = eng.run(C, M, p.K, p.a)
    assert eng.sync_status() == EPIC_OK and torch.equal(got, want)
    img = torch.rand(C.shape, device="cuda")
    eng.refine(img, img, got, iterations=1)
    assert eng.sync_status() == EPIC_OK
    eng.close()


@pytest.mark.parametrize("which", (-1, 7))
def test_no_such_wait(which):
    eng = EpicInterp(0)
    assert eng.selftest_wait_timeout(which, 10) == EPIC_ERR_INVALID
    eng.close()
