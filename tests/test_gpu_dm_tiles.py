"""Distribution maps at the sizes where the tiled prefix of the deficits and
the per-block counts of the free paths can go wrong: maps of one cell, of one
cell less and more than a tile of 2048 and of several tiles, with two moving
lights whose path ranges end inside a block.  Info words, maps, lists and
records are compared with the oracle bit for bit, as in test_gpu_dm.py."""
import numpy as np
import pytest

import oracle
import paper_2111_06906_gb300 as pv
from scenes import LIGHT_RECT, Light
from tests import gpu_util as gu
from tests import scene_kit as kit

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2111_06906_gb300 import build
    build.build()
    pv.load()


def _two_lights(n0, n1):
    sc = kit.rect_light_over_floor(n0 + n1, B=2, R=3.0)

    def lights(f):
        return [Light(LIGHT_RECT, (0.11 * (f - 1), 3.0, 0.07 * (f - 1)), (0.0, -1.0, 0.0), (1.0, 0.0, 0.0), (1.0, 1.0),
                      (100.0,) * 3, n0),
                Light(LIGHT_RECT, (0.3 - 0.05 * (f - 1), 2.5, 0.1), (0.0, -1.0, 0.0), (1.0, 0.0, 0.0), (0.5, 0.7),
                      (50.0,) * 3, n1)]
    sc._light_fn = lights
    return sc


@pytest.mark.parametrize("res", [(1, 1, 1, 1), (1, 1, 23, 89), (2, 4, 16, 16), (3, 1, 683, 1), (17, 241, 1, 1),
                                 (5, 7, 31, 9)])
def test_map_sizes_match_oracle(res):
    import torch
    seed, n0, n1 = 41, 1301, 2459
    sc = _two_lights(n0, n1)
    n = n0 + n1
    o = oracle.OracleScene(sc)
    o.set_frames(1, 1)
    o.set_dm(res, (0, 0))
    op = o.trace(np.arange(n, dtype=np.uint32), seed, 1)
    o.dm_reset()
    h = gu.lib_scene(sc, dm_rect=res)
    P = pv.Paths.allocate(n, sc.max_bounces)
    pv.pv_trace_all(h, P, seed, 1)
    gu.upload(P, op)
    lst = torch.zeros(n, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    filled = 0
    for f in (2, 3):
        gu.advance(h, sc, f)
        st = pv.new_stats()
        pv.pv_verify_paths(h, P, pv.PV_MODE_ERROR, 0.01, 0, lst, cnt, st, seed=seed, frame=f)
        o.set_frames(f - 1, f)
        _, ost = o.verify(op, pv.PV_MODE_ERROR, 0.01, seed=seed, frame=f)
        assert np.array_equal(gu.download(P).info, op.info)
        for l in range(2):
            assert np.array_equal(pv.pv_read_distribution_map(h, l), o.dm_counts(l)), l
        s = pv.stats_dict(st)
        assert (s["n_pruned"], s["n_filled"]) == (ost["n_pruned"], ost["n_filled"])
        filled += s["n_filled"]
        assert np.array_equal(lst[:int(cnt.item())].cpu().numpy().view(np.uint32), oracle.compact(op.info))
        pv.pv_retrace_invalid(h, P, lst, cnt, seed, f)
        o.retrace(op, seed, f)
        gu.upload(P, op)
    assert filled > 0
    assert pv.pv_read_device_status(h) == 0
    pv.pv_destroy_scene(h)
