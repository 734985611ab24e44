"""Pixels that see nothing are zero, whatever the radius."""
import math

import pytest

import paper_2111_06906_gb300 as pv
from tests import gpu_util as gu
from tests import scene_kit as kit

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2111_06906_gb300 import build
    build.build()
    pv.load()


@pytest.mark.parametrize("radius", [1.0, 1e-15, 1e-21, 1e-40, 1e30])      # from 1e-21 on, 1 / (pi radius^2) is infinite
def test_background_is_zero(radius):
    import torch
    sc = kit.rect_light_over_floor(500, B=1, R=3.0)
    h = gu.lib_scene(sc)
    P = pv.Paths.allocate(sc.n_paths, sc.max_bounces)
    pv.pv_trace_all(h, P, 3, 1)
    cam = pv.PvCamera.make((0.0, 2.0, 0.0), (0.0, 9.0, 1.0), (0.0, 0.0, 1.0), math.radians(50.0), 33, 21)
    img = torch.full((21, 33, 3), 7.0, device="cuda")
    work = torch.empty(pv.pv_splat_workspace_bytes(h, 33, 21), dtype=torch.uint8, device="cuda")
    pv.pv_splat(h, P, cam, radius, img, work)
    assert bool((img == 0).all())
    pv.pv_destroy_scene(h)
