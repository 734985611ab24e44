"""The first batch of a scene reads the tree's child references to see how deep it
is: 16 of a node's 128 bytes.  Its time over that of a second batch of the scene
(which finds the depth known), and the depth itself, by the stack that the batch
accepts, for trees of few and of many nodes."""
import time

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


def _create_twice(sc):
    import torch
    h = gu.lib_scene(sc)
    P = pv.Paths.allocate(sc.n_paths, sc.max_bounces)
    pv.pv_trace_all(h, P, 3, 1)
    torch.cuda.synchronize()
    t = []
    for _ in range(2):
        a = time.perf_counter()
        b = pv.pv_batch_create([(h, P, None, None, None, 3)], pv.PV_MODE_ERROR, sc.tau)
        t.append(time.perf_counter() - a)
        stack = pv.pv_batch_get_config(b)["stack"]
        pv.pv_batch_destroy(b)
    pv.pv_destroy_scene(h)
    return t, stack


def test_first_batch_of_a_large_scene():
    """Two million triangles: 19 ms; 40 ms when whole nodes were copied."""
    sc = scenes.villa(n_paths_per_light=1000)
    assert min(t[0] - t[1] for t, _ in (_create_twice(sc) for _ in range(4))) < 0.032


@pytest.mark.parametrize("n_boxes,stack", [(0, 32), (60, 32), (1500, 64), (16_666, 64)])
def test_depth_of_trees(n_boxes, stack):
    sc = scenes.city(n_paths=1000, n_boxes=n_boxes) if n_boxes else scenes.tiny_box(n_paths=1000)
    assert _create_twice(sc)[1] == stack
