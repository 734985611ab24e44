"""Counters of queries that reach the traversal cap: a step that the cap refuses
is no node visit, and Alg. 1 counts the same by itself and in the fused frame."""
import pytest

import paper_2111_06906_gb300 as pv
import scenes
from tests import gpu_util as gu
from tests import scene_kit as kit

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2111_06906_gb300 import build
    build.build()
    pv.load()


@pytest.mark.parametrize("limit", [1, 2, 3, 6])
def test_no_ray_counts_more_visits_than_the_cap(limit):
    sc = scenes.city(n_paths=5000, n_boxes=1500)
    h = gu.lib_scene(sc)
    P = pv.Paths.allocate(sc.n_paths, sc.max_bounces)
    pv.pv_set_traversal_limit(h, limit)
    st = pv.new_stats()
    pv.pv_trace_all(h, P, 3, 1, st)
    s = pv.stats_dict(st)
    assert pv.pv_read_device_status(h) == -5
    assert 0 < s["node_visits"] + s["tri_tests"] <= limit * s["trace_rays"]      # a step is a node or a leaf
    pv.pv_destroy_scene(h)


@pytest.mark.parametrize("limit", [2, 4, 7])
def test_fused_and_separate_calls_count_alike(limit):
    import torch
    sc = kit.box_with_torus(6000, B=4)
    out = []
    for fused in (False, True):
        h = gu.lib_scene(sc)
        P = pv.Paths.allocate(sc.n_paths, sc.max_bounces)
        pv.pv_trace_all(h, P, 3, 1)
        gu.advance(h, sc, 2)
        pv.pv_set_traversal_limit(h, limit)
        st = pv.new_stats()
        if fused:
            pv.pv_verify_retrace(h, P, pv.PV_MODE_ERROR, 0.01, 0, 3, 2, st)
        else:
            lst = torch.zeros(sc.n_paths, dtype=torch.int32, device="cuda")
            cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
            pv.pv_verify_paths(h, P, pv.PV_MODE_ERROR, 0.01, 0, lst, cnt, st)
            pv.pv_retrace_invalid(h, P, lst, cnt, 3, 2, st)
        out.append((pv.stats_dict(st), P.info.cpu().tolist()))
        assert pv.pv_read_device_status(h) == -5
        pv.pv_destroy_scene(h)
    assert out[0][0]["cont_rays"] > 0 and out[0] == out[1]
