"""Every call of a frame captured into a CUDA graph gives what it gives on a
stream, also where a memset stands before its first kernel, where the call is the
first one after a fork or a join of the capture, and when the graph is replayed."""
import math

import numpy as np
import pytest

import paper_2111_06906_gb300 as pv
import scenes
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

N, SEED = 20011, 7


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2111_06906_gb300 import build
    build.build()
    pv.load()


class _Frame:
    """A small district advanced to its second pose, with buffers for every call."""

    def __init__(self):
        import torch
        self.sc = sc = scenes.district(12_000, N, 2, 4, 2, seed=5)
        self.h = gu.lib_scene(sc)
        self.P = P = pv.Paths.allocate(N, sc.max_bounces)
        pv.pv_trace_all(self.h, P, SEED, 1)
        self.atlas = torch.zeros(96, 96, 3, dtype=torch.int64, device="cuda")
        pv.pv_deposit(self.h, P, self.atlas, sc.atlas_rect, 32)
        self.list, self.kept = (torch.zeros(N, dtype=torch.int32, device="cuda") for _ in range(2))
        self.count, self.kept_count = (torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(2))
        self.score = torch.as_tensor(np.random.default_rng(1).random(N).astype(np.float32), device="cuda")
        self.theta = torch.as_tensor(pv.pv_theta_current(self.h), device="cuda")
        self.model = torch.zeros(64, 64, 3, device="cuda")
        self.grad = torch.as_tensor(np.random.default_rng(2).random((64, 64, 3)).astype(np.float32), device="cuda")
        self.dtheta = torch.zeros_like(self.theta)
        self.image = torch.zeros(90, 160, 3, device="cuda")
        self.work = torch.full((pv.pv_splat_workspace_bytes(self.h, 160, 90),), 0xA5, dtype=torch.uint8, device="cuda")
        hz = sc.atlas_rect[2]
        self.cam = pv.PvCamera.make((0.0, 0.9 * hz, 0.7 * hz), (0.0, 0.0, 0.0), (0.0, 1.0, 0.0), math.radians(60.0),
                                    160, 90)
        self.st = pv.new_stats()
        gu.advance(self.h, sc, 2)
        torch.cuda.synchronize()

    def call(self, kind, stream):
        h, P, sc = self.h, self.P, self.sc
        if kind == "update":
            pv.pv_update_dynamic(h, sc.xforms(2), sc.lights(2), stream=stream)
            pv.pv_trace_all(h, P, SEED, 2, self.st, stream=stream)
        elif kind == "fused":
            pv.pv_verify_retrace_deposit(h, P, pv.PV_MODE_ERROR, 0.01, 0, SEED, 2, self.atlas, sc.atlas_rect, 32,
                                         self.st, stream=stream)
        elif kind == "carried":
            pv.pv_verify_retrace_deposit_delta(h, P, pv.PV_MODE_ERROR, 0.01, 0, SEED, 2, self.atlas, sc.atlas_rect,
                                               32, self.st, stream=stream)
        elif kind == "trace":
            pv.pv_trace_all_deposit(h, P, SEED, 2, self.atlas, sc.atlas_rect, 32, stream=stream)
        elif kind == "deposit":
            pv.pv_deposit(h, P, self.atlas, sc.atlas_rect, 32, stream=stream)
        elif kind == "splat":
            pv.pv_splat(h, P, self.cam, 0.3, self.image, self.work, stream=stream)
        elif kind == "budget":
            pv.pv_compact_replace(h, P, self.list, self.count, stream=stream)
            self.list.copy_(self.ids())
            self.count.fill_(N)
            pv.pv_budget_list(h, self.list, self.count, self.score, N // 3, self.kept, self.kept_count, stream=stream)
        elif kind == "model":
            self.model.zero_()
            self.dtheta.zero_()
            pv.pv_model_deposit(h, P, self.theta, self.model, sc.atlas_rect, stream=stream)
            pv.pv_adjoint_deposit(h, P, self.theta, self.grad, sc.atlas_rect, self.dtheta, stream=stream)

    def ids(self):
        import torch
        if not hasattr(self, "_ids"):
            self._ids = torch.arange(N, dtype=torch.int32, device="cuda")
        return self._ids

    def results(self):
        import torch
        torch.cuda.synchronize()
        whole = [t.cpu().numpy() for t in (self.P.info, self.P.origin, self.P.pa, self.P.pb, self.atlas, self.kept,
                                           self.kept_count, self.st)]
        sums = [t.cpu().numpy() for t in (self.image, self.model, self.dtheta)]
        assert pv.pv_read_device_status(self.h) == 0
        pv.pv_destroy_scene(self.h)
        return whole, sums


# the frames advance the records, so they are replayed once; the other calls give the same again
@pytest.mark.parametrize("fork", [False, True])
@pytest.mark.parametrize("kind,replays", [("update", 2), ("fused", 1), ("carried", 1), ("trace", 2), ("deposit", 3),
                                          ("splat", 3), ("budget", 3), ("model", 3)])
def test_captured_call_matches_stream(kind, replays, fork):
    import torch
    a, b = _Frame(), _Frame()
    a.ids(), b.ids()
    torch.cuda.synchronize()
    a.call(kind, torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        main = torch.cuda.current_stream()
        if fork:
            # the call's first node follows two others, and the capture joins its last one
            other = torch.cuda.Stream()
            x, y = torch.zeros(64, device="cuda"), torch.zeros(64, device="cuda")
            other.wait_stream(main)
            with torch.cuda.stream(other):
                y.add_(1.0)
            x.add_(1.0)
            main.wait_stream(other)
            b.call(kind, main)
            other.wait_stream(main)
            with torch.cuda.stream(other):
                y.add_(1.0)
            main.wait_stream(other)
        else:
            b.call(kind, main)
    for _ in range(replays):
        g.replay()
    (wa, fa), (wb, fb) = a.results(), b.results()
    if kind == "update":
        wa[-1], wb[-1] = wa[-1] * 0, wb[-1] * 0    # its counters add up over the replays
    for i, (p, q) in enumerate(zip(wa, wb)):
        assert np.array_equal(p.view(np.uint32), q.view(np.uint32)), i
    for p, q in zip(fa, fb):
        assert np.abs(p - q).max() <= 1e-5 * max(np.abs(p).max(), 1e-30)      # float32 sums in any order
