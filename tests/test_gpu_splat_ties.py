"""Primary rays at surfaces that lie on each other.  Of two triangles at the same
distance a query takes the one of lower index, whichever it meets first; so of two
copies of a triangle the same one is seen in every pixel."""
import math

import numpy as np
import pytest

import paper_2111_06906_gb300 as pv
from tests import gpu_util as gu
from tests import scene_kit as kit

pytestmark = pytest.mark.gpu

N, R, W, H = 6, 1.0, 240, 200
CAM = ((0.13, 1.37, 1.21), (0.02, 0.0, 0.05), (0.0, 1.0, 0.0))


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2111_06906_gb300 import build
    build.build()
    pv.load()


def _scene(copy_albedo, shift):
    """A floor of 2 N^2 triangles, twice; every second copy has ``copy_albedo``."""
    quad = np.asarray(kit.quad((-R, 0, -R), (0, 0, 2 * R), (2 * R, 0, 0), N), np.float64)
    quad = quad + np.array([0.0, shift, 0.0])
    lights = lambda f: [kit.Light(kit.LIGHT_POINT, (0.1, 1.0, 0.2), power=(20.0,) * 3, n_paths=4000)]
    return kit.build([(quad, (0.5, 0.5, 0.5), False), (quad, (copy_albedo,) * 3, False)], lights, B=1, diag=4.0)


def _image(sc):
    import torch
    h = gu.lib_scene(sc)
    P = pv.Paths.allocate(sc.n_paths, sc.max_bounces)
    pv.pv_trace_all(h, P, 3, 1)
    img = torch.zeros(H, W, 3, device="cuda")
    work = torch.empty(pv.pv_splat_workspace_bytes(h, W, H), dtype=torch.uint8, device="cuda")
    pv.pv_splat(h, P, pv.PvCamera.make(*CAM, math.radians(70.0), W, H), 0.4, img, work)
    pv.pv_destroy_scene(h)
    return img.cpu().numpy()[..., 0]


def _floor_points(shift):
    pos, target, up = (np.asarray(v, np.float64) for v in CAM)
    f = (target - pos) / np.linalg.norm(target - pos)
    r = np.cross(f, up)
    r /= np.linalg.norm(r)
    u = np.cross(r, f)
    ty = math.tan(math.radians(35.0))
    x = (2 * (np.arange(W) + 0.5) / W - 1) * ty * W / H
    y = (1 - 2 * (np.arange(H) + 0.5) / H) * ty
    d = f + x[None, :, None] * r + y[:, None, None] * u
    t = (shift - pos[1]) / d[..., 1]
    return (pos + t[..., None] * d)[..., [0, 2]]


@pytest.mark.parametrize("shift", [0.0, 0.1, 1.0 / 3.0])
def test_one_of_two_copies_is_seen_everywhere(shift):
    both = _image(_scene(0.5, shift))              # either copy looks the same
    img = _image(_scene(0.0, shift))               # a copy seen is black
    xz = (_floor_points(shift) + R) * N / (2 * R)  # in cells
    cell, at = np.floor(xz).astype(int), xz - np.floor(xz)
    # which triangle: pixels near an edge or a diagonal (of either direction) are left out
    edge = np.minimum(at, 1 - at).min(-1)
    clear = (edge > 0.02) & (np.abs(at[..., 0] - at[..., 1]) > 0.03) & (np.abs(at.sum(-1) - 1) > 0.03)
    clear &= (cell >= 0).all(-1) & (cell < N).all(-1) & (both > 0)
    part = (at[..., 0] > at[..., 1]) * 2 + (at.sum(-1) > 1)      # quarter of the cell, within one triangle
    key = (cell[..., 0] * N + cell[..., 1]) * 4 + part
    seen = img > 0.5 * both
    mixed = [k for k in np.unique(key[clear]) if len(np.unique(seen[clear & (key == k)])) > 1]
    assert clear.sum() > 5000 and not mixed, mixed
