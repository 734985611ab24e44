"""Workspaces of the splat: 32 bytes a photon place, the cell counters and the
visible points are enough; what pv_splat_workspace_bytes asks for may be more.
An image from the smallest workspace is that of the full one, and a byte less is
refused."""
import math

import pytest

import paper_2111_06906_gb300 as pv
import scenes
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2111_06906_gb300 import build
    build.build()
    pv.load()


def _least(photons, W, H):
    up = lambda x: (x + 255) & ~255
    cells = 4096
    while cells < photons:
        cells *= 2
    return up(up(up(32 * W * H) + 4 * cells) + 4 * (cells // 4096 + 1)) + up(32 * photons)


@pytest.mark.parametrize("paths", [1, 2, 1000, 4099, 30001])
@pytest.mark.parametrize("size", [(1, 1), (67, 41), (160, 90)])
def test_least_workspace(paths, size):
    import torch
    W, H = size
    sc = scenes.tiny_box(n_paths=paths)
    h = gu.lib_scene(sc)
    P = pv.Paths.allocate(paths, sc.max_bounces)
    pv.pv_trace_all(h, P, 4, 1)
    cam = pv.PvCamera.make((0.0, 1.0, 6.0), (0.0, 0.9, 0.0), (0.0, 1.0, 0.0), math.radians(25.0), W, H)
    least = _least(paths * sc.max_bounces, W, H)
    full = pv.pv_splat_workspace_bytes(h, W, H)
    assert full >= least
    img = [torch.full((H, W, 3), 7.0, device="cuda") for _ in range(2)]
    buf = torch.full((max(full, least) + 256,), 0xA5, dtype=torch.uint8, device="cuda")
    pv.pv_splat(h, P, cam, 0.3, img[0], buf[:full])
    buf.fill_(0xA5)
    for _ in range(2):                             # a second call finds the first one's workspace
        pv.pv_splat(h, P, cam, 0.3, img[1], buf[:least])
    assert bool((buf[least:] == 0xA5).all())       # and stays inside it
    # the same float32 sums in another order
    assert torch.allclose(img[0], img[1], rtol=1e-5, atol=1e-6 * float(img[0].max()))
    with pytest.raises(pv.PvError):
        pv.pv_splat(h, P, cam, 0.3, img[1], buf[:least - 1])
    pv.pv_destroy_scene(h)
