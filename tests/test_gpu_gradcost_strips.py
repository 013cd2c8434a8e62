"""The cost-map kernel where its strips change: widths around a strip and a
lane's pixels, heights around a strip's rows, rows on 16-, 8- and 4-byte
boundaries, and images that do not start on a 16-byte boundary.  float32
arithmetic against 64 bits: within 1e-6 relative + 1e-7 absolute."""

import pytest

from paper_1501_02565_gb300.native import gradient_cost

pytestmark = pytest.mark.gpu


def _ref(x, floor):
    import torch
    x = x.double()

    def d(axis):
        n = x.shape[axis]
        i = torch.arange(n, device=x.device)
        return 0.5 * (x.index_select(axis, (i + 1).clamp(max=n - 1)) -
                      x.index_select(axis, (i - 1).clamp(min=0)))
    return floor + (d(2) ** 2 + d(1) ** 2).sum(-1).sqrt()


@pytest.mark.parametrize("ch", (1, 3, 4))
@pytest.mark.parametrize("W", (1, 2, 3, 4, 5, 59, 60, 61, 62, 119, 120, 121, 124, 241, 362))
@pytest.mark.parametrize("F, H", [(1, 1), (2, 2), (3, 7), (1, 40)])
@pytest.mark.parametrize("offset", (0, 1, 2))
def test_strip_edges(ch, W, F, H, offset):
    import torch
    g = torch.Generator(device="cuda").manual_seed(W * 7 + H)
    flat = torch.rand(F * H * W * ch + offset, generator=g, device="cuda")
    x = flat[offset:].view(F, H, W, ch)
    got = gradient_cost(x, 0.25)
    torch.testing.assert_close(got.double(), _ref(x, 0.25), rtol=1e-6, atol=1e-7)


def test_many_frames():
    import torch
    x = torch.rand((40, 97, 333, 3), device="cuda")
    torch.testing.assert_close(gradient_cost(x, 0.0).double(), _ref(x, 0.0), rtol=1e-6, atol=1e-7)
