"""The differentiable deposit and its adjoint where their texel rows can go
wrong: atlases narrower than a photon's four taps, of every width modulo four
and of a single row (rows that end at the array's last floats), arrays that
start off a 16-byte boundary, photons that fall outside, warps with one path
and with paths of up to 15 photons.  Reference: the FP64 oracle on the same
records; tolerances as in test_gpu_adjoint.py (1e-4 of the atlas maximum;
2e-3 of the largest gradient entry + 1e-3 relative; scores 1e-4 + 1e-4)."""
import numpy as np
import pytest

import oracle
import scenes
import paper_2111_06906_gb300 as pv
from tests import gpu_util as gu
from tests import scene_kit as kit

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2111_06906_gb300 import build
    build.build()
    pv.load()


@pytest.mark.parametrize("paths,bounces", [(1, 3), (33, 15), (700, 7)])
@pytest.mark.parametrize("size", [(1, 1), (2, 3), (3, 1), (4, 4), (5, 2), (6, 9), (7, 1), (31, 17)])
def test_texel_rows_match_oracle(paths, bounces, size):
    import torch
    W, H = size
    sc = kit.box_with_torus(paths, B=bounces)
    rect = (-0.7, -0.6, 0.8, 0.9)                # part of the photons lie outside
    o = oracle.OracleScene(sc)
    o.set_frames(1, 1)
    op = o.trace(np.arange(paths, dtype=np.uint32), 3, 1)
    h = gu.lib_scene(sc)
    P = pv.Paths.allocate(paths, sc.max_bounces)
    gu.upload(P, op)
    th = o.theta_current()
    d_th = torch.as_tensor(th, dtype=torch.float32, device="cuda")
    G = np.random.default_rng(W * 100 + H).standard_normal((H, W, 3)).astype(np.float32)
    want = o.model_deposit(op, th, W, H, rect)
    dth_o, score_o = o.adjoint(op, th, G, rect)
    for off in (0, 1, 2):                        # floats past the allocation's 256-byte boundary
        buf = torch.zeros(3 * W * H + off + 8, dtype=torch.float32, device="cuda")
        A = buf[off:off + 3 * W * H].view(H, W, 3)
        pv.pv_model_deposit(h, P, d_th, A, rect)
        err = np.abs(A.cpu().numpy() - want).max()
        assert err <= 1e-4 * max(want.max(), 1e-30), (off, err)
        assert not bool(buf[:off].any()) and not bool(buf[off + 3 * W * H:].any())
        gbuf = torch.full((3 * W * H + off + 8,), float("nan"), device="cuda")
        gbuf[off:off + 3 * W * H] = torch.as_tensor(G.reshape(-1), device="cuda")
        dth = torch.zeros_like(d_th)
        score = torch.zeros(paths, device="cuda")
        pv.pv_adjoint_deposit(h, P, d_th, gbuf[off:off + 3 * W * H].view(H, W, 3), rect, dth, score)
        e = np.abs(dth.cpu().numpy() - dth_o)
        assert np.all(e <= 2e-3 * np.abs(dth_o).max() + 1e-3 * np.abs(dth_o) + 1e-30), (off, e)
        s = np.abs(score.cpu().numpy() - score_o)
        assert np.all(s <= 1e-4 * score_o.max() + 1e-4 * score_o + 1e-30), (off, s.max())
    assert pv.pv_read_device_status(h) == 0
    pv.pv_destroy_scene(h)
