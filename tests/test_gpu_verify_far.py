"""Box tests of segments that leave the range of float32: a moved object's group
with free places must not count them as objects."""
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


@pytest.mark.parametrize("y,meets", [(1.7, False), (0.9, True)])      # above the moved torus, and at its height
def test_infinite_segment(y, meets):
    import torch
    n = 70
    sc = kit.box_with_torus(n, B=2)
    h = gu.lib_scene(sc)
    P = pv.Paths.allocate(n, sc.max_bounces)
    pv.pv_trace_all(h, P, 3, 1)
    # one photon per path, infinitely far along +x from a point beside the torus
    P.info.copy_((P.info & ~(15 << pv.PV_INFO_NSEG_SHIFT)) | (1 << pv.PV_INFO_NSEG_SHIFT))
    P.origin[0], P.origin[1], P.origin[2] = -0.9, y, 0.0
    P.pa[0, :, 0], P.pa[0, :, 1], P.pa[0, :, 2] = float("inf"), y, 0.0
    P.pa[0, :, 3] = 0.0                            # on triangle 0 of the room, which does not move
    gu.advance(h, sc, 2)
    lst = torch.zeros(n, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    pv.pv_verify_paths(h, P, pv.PV_MODE_NAIVE_AABB, 0.01, 0, lst, cnt, seed=3, frame=2)
    assert int(cnt.item()) == (n if meets else 0)
    pv.pv_destroy_scene(h)
