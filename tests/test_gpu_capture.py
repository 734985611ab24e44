"""A frame captured into a CUDA graph and replayed gives what the same calls
give on a stream: the frame's kernels are dependent launches with the clears
between them in one kernel, and both must order the same way as graph nodes."""
import numpy as np
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


@pytest.mark.parametrize("dm", [(0, 0, 0, 0), (3, 2, 9, 31)])
@pytest.mark.parametrize("n", [1, 2049, 30011])
def test_captured_frame_matches_stream(n, dm):
    import torch
    seed = 23
    sc = kit.rect_light_over_floor(n, shift=lambda f: (0.07 * (f - 1), 0.0, 0.05 * (f - 1)), B=2, R=3.0)
    out = []
    for captured in (False, True):
        h = gu.lib_scene(sc, dm_rect=dm)
        P = pv.Paths.allocate(n, sc.max_bounces)
        pv.pv_trace_all(h, P, seed, 1)
        lst = torch.zeros(n, dtype=torch.int32, device="cuda")
        cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
        st = pv.new_stats()
        gu.advance(h, sc, 2)
        torch.cuda.synchronize()

        def frame(stream):
            pv.pv_verify_paths(h, P, pv.PV_MODE_ERROR, 0.01, 0, lst, cnt, st, stream=stream, seed=seed, frame=2)
            pv.pv_retrace_invalid(h, P, lst, cnt, seed, 2, st, stream=stream)

        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                frame(torch.cuda.current_stream())
            g.replay()
        else:
            frame(torch.cuda.current_stream())
        torch.cuda.synchronize()
        k = int(cnt.item())
        p = gu.download(P)
        out.append((k, lst[:k].cpu().numpy().copy(), p.info.copy(), P.pa.cpu().numpy(), pv.stats_dict(st)))
        assert pv.pv_read_device_status(h) == 0
        pv.pv_destroy_scene(h)
    (k0, l0, i0, a0, s0), (k1, l1, i1, a1, s1) = out
    assert k0 == k1 and np.array_equal(l0, l1) and np.array_equal(i0, i1)
    assert np.array_equal(a0.view(np.uint32), a1.view(np.uint32))
    assert s0 == s1
