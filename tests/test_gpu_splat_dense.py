"""Splat tiles around the number of photons (1024) from which a tile is shared by
several warps: every tile of the image meets exactly K photons (the radius spans
the room), and a city view has sparse and shared tiles side by side.  Oracle and
tolerance as in test_gpu_splat.py: 1e-4 of the image maximum + 1e-4 relative."""
import math

import numpy as np
import pytest

import oracle
import scenes
import paper_2111_06906_gb300 as pv
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2111_06906_gb300 import build
    build.build()
    pv.load()


def _keep_first(op, photons):
    """Shorten the paths, last first, until ``photons`` photons are left."""
    sh = np.uint32(pv.PV_INFO_NSEG_SHIFT)
    nseg = (op.info >> sh) & np.uint32(15)
    before = np.cumsum(nseg) - nseg
    left = np.clip(photons - before.astype(np.int64), 0, nseg).astype(np.uint32)
    assert int(left.sum()) == photons
    op.info[:] = (op.info & ~(np.uint32(15) << sh)) | (left << sh)


def _compare(sc, op, view, size, radius):
    import torch
    (pos, target, up), fov = view
    W, H = size
    o = oracle.OracleScene(sc)
    o.set_frames(1, 1)
    want, amb = o.splat(op, oracle.Camera.make(pos, target, up, math.radians(fov), W, H), radius)
    h = gu.lib_scene(sc)
    P = pv.Paths.allocate(sc.n_paths, sc.max_bounces)
    gu.upload(P, op)
    cam = pv.PvCamera.make(pos, target, up, math.radians(fov), W, H)
    img = torch.full((H, W, 3), 7.0, dtype=torch.float32, device="cuda")
    work = torch.full((pv.pv_splat_workspace_bytes(h, W, H),), 0xA5, dtype=torch.uint8, device="cuda")
    pv.pv_splat(h, P, cam, radius, img, work)
    err = np.abs(img.cpu().numpy().astype(np.float64) - want)[~amb]
    assert (err <= 1e-4 * want.max() + 1e-4 * np.abs(want)[~amb]).all(), (float(err.max()), float(want.max()))
    assert pv.pv_read_device_status(h) == 0
    pv.pv_destroy_scene(h)


@pytest.mark.parametrize("size", [(1, 1), (8, 4), (9, 5), (67, 41)])
@pytest.mark.parametrize("photons", [1023, 1024, 1025, 4097])
def test_tile_of_k_photons(photons, size):
    sc = scenes.tiny_box(n_paths=4000)
    o = oracle.OracleScene(sc)
    o.set_frames(1, 1)
    op = o.trace(np.arange(sc.n_paths, dtype=np.uint32), 4, 1)
    _keep_first(op, photons)
    _compare(sc, op, (((0.0, 1.0, 6.0), (0.0, 0.9, 0.0), (0.0, 1.0, 0.0)), 25.0), size, 3.0)


def test_sparse_and_dense_tiles_of_one_image():
    sc = scenes.city(n_paths=12000, n_boxes=1500)
    o = oracle.OracleScene(sc)
    o.set_frames(1, 1)
    op = o.trace(np.arange(sc.n_paths, dtype=np.uint32), 4, 1)
    _compare(sc, op, (((0.0, 9.0, 30.0), (0.0, 2.0, 0.0), (0.0, 1.0, 0.0)), 50.0), (203, 117), 2.0)
