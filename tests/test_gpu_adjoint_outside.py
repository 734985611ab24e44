"""The adjoint at photons outside the atlas: they are no part of the loss, so
their energy must not reach the gradient or a score, not even an infinite one."""
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


@pytest.mark.parametrize("off", [0, 1])           # an array at and off a 16-byte boundary
@pytest.mark.parametrize("axis", [0, 2])
def test_infinite_energy_outside_adds_nothing(axis, off):
    import torch
    W = H = 24
    sc = kit.box_with_torus(900, B=3)
    h = gu.lib_scene(sc)
    P = pv.Paths.allocate(sc.n_paths, sc.max_bounces)
    pv.pv_trace_all(h, P, 3, 1)
    # the atlas covers half of the room: along ``axis`` half of the photons lie outside, far from its last texels
    rect = (-1.1, -1.1, 0.0, 1.1) if axis == 0 else (-1.1, -1.1, 1.1, 0.0)
    th = torch.as_tensor(pv.pv_theta_current(h), device="cuda")
    G = torch.zeros(3 * W * H + 1, device="cuda")[off:off + 3 * W * H].view(H, W, 3)
    G.copy_(torch.as_tensor(np.random.default_rng(5).standard_normal((H, W, 3)).astype(np.float32)))
    out = P.pa[..., axis] > 0.3                    # more than two texels beyond the edge
    assert int(out.sum()) > 100

    def adjoint(energy):
        P.pb[..., :3] = torch.where(out[..., None], torch.full_like(P.pb[..., :3], energy), P.pb[..., :3])
        d, s = torch.zeros_like(th), torch.zeros(sc.n_paths, device="cuda")
        pv.pv_adjoint_deposit(h, P, th, G, rect, d, s)
        return d.cpu().numpy(), s.cpu().numpy()

    d0, s0 = adjoint(0.0)
    d1, s1 = adjoint(float("inf"))
    assert np.isfinite(d0).all() and np.abs(d0).max() > 0
    # the same sums, their atomics in any order
    assert np.abs(d1 - d0).max() <= 1e-5 * np.abs(d0).max()
    assert np.array_equal(s1, s0)
    pv.pv_destroy_scene(h)
