"""Radii small against the scene, where the photon grid is one row of places:
images against the FP64 oracle on both sides of the line, with as few places as
there can be (rows wrap, and places are shared), and the time of an image whose
photons lie on one plane.  Tolerance as in test_gpu_splat.py: 1e-4 of the image
maximum + 1e-4 relative."""
import math

import numpy as np
import pytest

import oracle
import scenes
import paper_2111_06906_gb300 as pv
from tests import gpu_util as gu
from tests import scene_kit as kit

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2111_06906_gb300 import build
    build.build()
    pv.load()


# 3900 photon places, so 4096 cells: by axes from a radius of 0.15 on, one row below
@pytest.mark.parametrize("radius", [0.03, 0.07, 0.1, 0.13, 0.15])
@pytest.mark.parametrize("size", [(1, 1), (9, 5), (130, 94)])
def test_either_side_of_the_line(size, radius):
    import torch
    W, H = size
    n = 1300
    sc = scenes.tiny_box(n_paths=n)
    o = oracle.OracleScene(sc)
    o.set_frames(1, 1)
    op = o.trace(np.arange(n, dtype=np.uint32), 4, 1)
    view = ((0.0, 1.0, 6.0), (0.0, 0.9, 0.0), (0.0, 1.0, 0.0), math.radians(25.0), W, H)
    want, amb = o.splat(op, oracle.Camera.make(*view), radius)
    h = gu.lib_scene(sc)
    P = pv.Paths.allocate(n, sc.max_bounces)
    gu.upload(P, op)
    img = torch.full((H, W, 3), 7.0, device="cuda")
    work = torch.full((pv.pv_splat_workspace_bytes(h, W, H),), 0xA5, dtype=torch.uint8, device="cuda")
    pv.pv_splat(h, P, pv.PvCamera.make(*view), radius, img, work)
    err = np.abs(img.cpu().numpy().astype(np.float64) - want)[~amb]
    assert (err <= 1e-4 * want.max() + 1e-4 * np.abs(want)[~amb]).all(), (float(err.max()), float(want.max()))
    assert pv.pv_read_device_status(h) == 0
    pv.pv_destroy_scene(h)


def _best_ms(sc, cam, radii):
    """Fastest of a dozen images at each radius."""
    import torch
    h = gu.lib_scene(sc)
    P = pv.Paths.allocate(sc.n_paths, sc.max_bounces)
    pv.pv_trace_all(h, P, 3, 1)
    img = torch.zeros(cam.height, cam.width, 3, device="cuda")
    work = torch.empty(pv.pv_splat_workspace_bytes(h, cam.width, cam.height), dtype=torch.uint8, device="cuda")
    out = []
    for radius in radii:
        ms = []
        for _ in range(12):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            pv.pv_splat(h, P, cam, radius, img, work)
            b.record()
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
        out.append(min(ms))
    pv.pv_destroy_scene(h)
    return out


def test_small_radius_on_a_plane_costs_no_more():
    """500k photons spread over a floor: at a hundredth of the radius a point has a ten-thousandth of the photons
    in reach.  (With a grid whose cells of a plane fell on each other the image took four times as long.)"""
    cam = pv.PvCamera.make((0.0, 4.0, 12.0), (0.0, 0.5, 0.0), (0.0, 1.0, 0.0), math.radians(60.0), 700, 500)
    small, large = _best_ms(kit.rect_light_over_floor(500_000, B=1, R=20.0), cam, (0.002, 0.2))
    assert small < 2.0 * large, (small, large)


def test_points_far_apart_cost_little_more():
    """A large image of a room whose points lie many radii apart.  (With the pixels of a tile taken one after the
    other it took nearly four times as long as at a thousand times the radius; it takes 1.5 times.)"""
    cam = pv.PvCamera.make((0.0, 1.5, 0.95), (0.0, 0.2, -0.4), (0.0, 1.0, 0.0), math.radians(60.0), 1920, 1080)
    small, large = _best_ms(scenes.tiny_box(n_paths=10_000), cam, (0.0001, 0.1))
    assert small < 2.5 * large, (small, large)
