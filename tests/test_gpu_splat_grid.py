"""GPU splat over the sizes at which its grid and its pixel tiles can go wrong,
against the FP64 oracle on the oracle's own records: images smaller than a
tile and with ragged edges, radii for which the grid has its fewest cells per
axis or wraps around, and views whose pixels lie at very different depths.
Tolerance as in test_gpu_splat.py: float32 visible points and sums in any
order, 1e-4 of the image maximum + 1e-4 relative."""
import math

import numpy as np
import pytest

import oracle
import scenes
import paper_2111_06906_gb300 as pv
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

BOX = ((0.0, 1.0, 6.0), (0.0, 0.9, 0.0), (0.0, 1.0, 0.0))
SCENES = {
    "radius_of_the_room": (lambda: scenes.tiny_box(n_paths=3000), BOX, 25.0, 1.5),
    "grid_wraps": (lambda: scenes.tiny_box(n_paths=3000), BOX, 25.0, 0.02),
    "no_photons_seen": (lambda: scenes.tiny_box(n_paths=7), BOX, 25.0, 0.001),
    "depth_edges": (lambda: scenes.city(n_paths=6000, n_boxes=1500), ((0.0, 9.0, 30.0), (0.0, 2.0, 0.0), (0.0, 1.0, 0.0)),
                    50.0, 1.0),
}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2111_06906_gb300 import build
    build.build()
    pv.load()


@pytest.mark.parametrize("size", [(1, 1), (7, 5), (9, 33), (130, 47)])
@pytest.mark.parametrize("name", list(SCENES))
def test_splat_grid_matches_oracle(name, size):
    import torch
    make, (pos, target, up), fov, radius = SCENES[name]
    W, H = size
    sc = make()
    o = oracle.OracleScene(sc)
    o.set_frames(1, 1)
    op = o.trace(np.arange(sc.n_paths, dtype=np.uint32), 4, 1)
    want, amb = o.splat(op, oracle.Camera.make(pos, target, up, math.radians(fov), W, H), radius)
    h = gu.lib_scene(sc)
    P = pv.Paths.allocate(sc.n_paths, sc.max_bounces)
    gu.upload(P, op)
    cam = pv.PvCamera.make(pos, target, up, math.radians(fov), W, H)
    img = torch.full((H, W, 3), 7.0, dtype=torch.float32, device="cuda")
    work = torch.full((pv.pv_splat_workspace_bytes(h, W, H),), 0xA5, dtype=torch.uint8, device="cuda")
    for _ in range(2):                       # a second call finds the first one's workspace
        pv.pv_splat(h, P, cam, radius, img, work)
    err = np.abs(img.cpu().numpy().astype(np.float64) - want)[~amb]
    assert (err <= 1e-4 * want.max() + 1e-4 * np.abs(want)[~amb]).all(), (float(err.max()), float(want.max()))
    assert pv.pv_read_device_status(h) == 0
    pv.pv_destroy_scene(h)


def test_photons_out_of_reach_add_nothing_whatever_their_energy():
    """A photon with infinite energy shows where it is, and only there: the packed
    sums must not pick up infinity times a weight of zero."""
    import torch
    sc = scenes.tiny_box(n_paths=2000)
    h = gu.lib_scene(sc)
    P = pv.Paths.allocate(sc.n_paths, sc.max_bounces)
    pv.pv_trace_all(h, P, 4, 1)
    cam = pv.PvCamera.make(*BOX, math.radians(25.0), 64, 48)
    work = torch.empty(pv.pv_splat_workspace_bytes(h, 64, 48), dtype=torch.uint8, device="cuda")
    plain, odd = (torch.zeros(48, 64, 3, device="cuda") for _ in range(2))
    pv.pv_splat(h, P, cam, 0.2, plain, work)
    on_back = torch.nonzero((P.pa[0, :, 2] < -0.99) & (P.pa[0, :, 1] > 0.9)).flatten()
    P.pb[0, on_back[0], 0] = float("inf")
    pv.pv_splat(h, P, cam, 0.2, odd, work)
    assert not bool(torch.isnan(odd).any())
    bright = torch.isinf(odd[..., 0])
    assert 0 < int(bright.sum()) < bright.numel() // 2
    assert torch.allclose(odd[~bright], plain[~bright], rtol=1e-5, atol=1e-5 * float(plain.max()))
    pv.pv_destroy_scene(h)
