"""Lists that leave lanes without work.  The persistent kernels spread a list
shorter than their lanes over their warps; a path's new record must not depend on
how long the list was or which lane took it."""
import numpy as np
import pytest

import paper_2111_06906_gb300 as pv
import scenes
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

SEED = 11


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2111_06906_gb300 import build
    build.build()
    pv.load()


def _listed(n):
    """A scene whose second frame lists most of its n paths, the records after verification, and the list."""
    import torch
    sc = scenes.city(n_paths=n, n_boxes=1500)
    h = gu.lib_scene(sc)
    P = pv.Paths.allocate(n, sc.max_bounces)
    pv.pv_trace_all(h, P, SEED, 1)
    gu.advance(h, sc, 9)
    lst = torch.zeros(n, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    pv.pv_verify_paths(h, P, pv.PV_MODE_NAIVE_AABB, 0.0, 0, lst, cnt)
    return sc, h, P, lst[:int(cnt.item())].clone()


@pytest.fixture(scope="module")
def case():
    import torch
    sc, h, P, lst = _listed(200_000)
    base = [t.clone() for t in (P.info, P.origin, P.pa, P.pb)]
    cnt = torch.tensor([lst.numel()], dtype=torch.int32, device="cuda")
    st = pv.new_stats()
    pv.pv_retrace_invalid(h, P, lst, cnt, SEED, 9, st)
    yield sc, h, P, lst, base, [t.clone() for t in (P.info, P.origin, P.pa, P.pb)], pv.stats_dict(st)
    pv.pv_destroy_scene(h)


# lengths around multiples of a full grid's warps (eight blocks of four warps per SM), down to one path
@pytest.mark.parametrize("times,more", [(0, 1), (0, 2), (1, -1), (1, 0), (1, 1), (2, 0), (2, 1), (5, 3), (8, -1), (8, 1),
                                        (31, 1), (32, -1), (32, 0), (32, 1)])
def test_retraced_records_do_not_depend_on_the_list(case, times, more):
    import torch
    sc, h, P, lst, base, full, _ = case
    warps = 32 * torch.cuda.get_device_properties(0).multi_processor_count
    m = min(times * warps + more, lst.numel())
    pick = torch.as_tensor(np.sort(np.random.default_rng(m).choice(lst.numel(), m, replace=False)), device="cuda")
    some = lst[pick].contiguous()
    for t, b in zip((P.info, P.origin, P.pa, P.pb), base):
        t.copy_(b)
    room = torch.zeros(P.n, dtype=torch.int32, device="cuda")
    room[:m] = some
    st = pv.new_stats()
    pv.pv_retrace_invalid(h, P, room, torch.tensor([m], dtype=torch.int32, device="cuda"), SEED, 9, st)
    done = torch.zeros(P.n, dtype=torch.bool, device="cuda")
    done[some.long()] = True
    i32 = torch.int32
    for t, b, f, path_dim in zip((P.info, P.origin, P.pa, P.pb), base, full, (0, 1, 1, 1)):
        shape = [1] * t.dim()
        shape[path_dim] = P.n
        want = torch.where(done.view(shape), f.view(i32) if t.dtype != i32 else f, b.view(i32) if t.dtype != i32 else b)
        assert torch.equal(t.view(i32) if t.dtype != i32 else t, want)
    assert pv.stats_dict(st)["trace_rays"] > 0
    assert pv.pv_read_device_status(h) == 0


@pytest.mark.parametrize("n", [1, 31, 33, 1023, 4864, 40_000])
def test_fused_frame_equals_separate_calls(n):
    """Short and long lists of Alg. 1 and of the re-trace, and the deposits after them, in one kernel."""
    import torch
    sc = scenes.city(n_paths=n, n_boxes=1500)
    out = []
    for fused in (False, True):
        h = gu.lib_scene(sc)
        P = pv.Paths.allocate(n, sc.max_bounces)
        pv.pv_trace_all(h, P, SEED, 1)
        gu.advance(h, sc, 2)
        atlas = torch.zeros(40, 40, 3, dtype=torch.int64, device="cuda")
        st = pv.new_stats()
        if fused:
            pv.pv_verify_retrace_deposit(h, P, pv.PV_MODE_ERROR, 0.01, 0, SEED, 2, atlas, sc.atlas_rect, 32, st)
        else:
            lst = torch.zeros(n, dtype=torch.int32, device="cuda")
            cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
            pv.pv_verify_paths(h, P, pv.PV_MODE_ERROR, 0.01, 0, lst, cnt, st, seed=SEED, frame=2)
            pv.pv_retrace_invalid(h, P, lst, cnt, SEED, 2, st)
            pv.pv_deposit(h, P, atlas, sc.atlas_rect, 32)
        out.append([P.info, P.origin.view(torch.int32), P.pa.view(torch.int32), P.pb.view(torch.int32), atlas, st])
        assert pv.pv_read_device_status(h) == 0
        pv.pv_destroy_scene(h)
    for a, b in zip(*out):
        assert torch.equal(a, b)
