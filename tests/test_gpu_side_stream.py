"""A call made under a side stream waits for that stream's work and for nothing
less: it sees what the stream wrote just before."""
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


def test_calls_under_a_side_stream_see_its_writes():
    import torch
    sc = scenes.tiny_box(n_paths=20_000)
    h = gu.lib_scene(sc)
    P, Q = (pv.Paths.allocate(sc.n_paths, sc.max_bounces) for _ in range(2))
    pv.pv_trace_all(h, P, 3, 1)
    want = torch.zeros(64, 64, 3, dtype=torch.int64, device="cuda")
    pv.pv_deposit(h, P, want, sc.atlas_rect, 32)
    got, big = torch.zeros_like(want), torch.ones(1 << 28, device="cuda")
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        for _ in range(10):
            big.mul_(1.0)                         # some milliseconds of work before the records are written
        for a, b in zip((Q.info, Q.origin, Q.pa, Q.pb), (P.info, P.origin, P.pa, P.pb)):
            a.copy_(b)
        pv.pv_deposit(h, Q, got, sc.atlas_rect, 32)
    side.synchronize()
    assert torch.equal(got, want)
    pv.pv_destroy_scene(h)
