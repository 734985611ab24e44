"""Workloads of the path-verification library, each one pass through its public entry points.

``listed()`` names the workloads, ``draw(rng)`` gives one more of the same ranges, ``prepare(case, seed)``
builds what a renderer has in hand before a frame (scene handle, traced paths, atlas, marshalled poses),
``run(state)`` makes one pass, ``work(case)`` is the least traffic and arithmetic of that pass and
``exact(case, seed)`` its result in 64 bits where that can be had.

Scenes are the repository's seeded ones (``scenes``).  The seed picks the random numbers of the paths
and the frame of the motion at which the pass starts.  A pass that advances the scene takes the next
pose of a stretch of the scene's motion, walked forth and back, and the next frame number.
"""
from __future__ import annotations

import functools
import math
from dataclasses import replace

import numpy as np
import torch

import paper_2111_06906_gb300 as pv
import scenes

SCALE_LOG2 = 32          # fixed point of the atlas
POSES = 12               # poses of the motion that a state walks forth and back
MODES = {"error": (pv.PV_MODE_ERROR, 0), "error_exact": (pv.PV_MODE_ERROR, pv.PV_FLAG_ERROR_EXACT),
         "naive_aabb": (pv.PV_MODE_NAIVE_AABB, 0), "naive_exact": (pv.PV_MODE_NAIVE_EXACT, 0)}


def _case(kind, scene, paths, **kw):
    c = {"kind": kind, "scene": scene, "tris": 0, "paths": paths, "lights": 1, "bounces": 7, "tori": 4, "atlas": 1024,
         "mode": "error", "point_moves": False, "maps": 0, "width": 0, "height": 0, "radius": 0.0, "budget": 0,
         "scenes": 1}
    c.update(kw)
    return c


def listed():
    def named(name, c):
        return {"name": name, **c}

    return [
        # the smallest frame: one room, a moving cube, a point light; a tool or a preview, bound by launches
        named("box_frame", _case("frame", "box", 10_000, bounces=3, atlas=128)),
        # an ordinary frame: verification, re-trace and deposit of a million paths in a city of 200k triangles
        named("city_frame", _case("frame", "city", 1_000_000)),
        # the largest frame: an interior of two million triangles, three lights, three million paths
        named("villa_frame", _case("frame", "villa", 3_000_000, lights=3)),
        # a lamp carried through the scene: a moving point light needs a visibility ray per path; the atlas is
        # carried from frame to frame instead of cleared
        named("lamp_frame", _case("carried", "district", 600_011, tris=60_000, lights=2, bounces=5, tori=3, atlas=777,
                                  point_moves=True)),
        # the separate calls of a renderer that needs the list of pruned paths, with the exact segment test
        named("calls_frame", _case("calls", "district", 300_007, tris=30_000, lights=3, bounces=4, tori=2, atlas=500,
                                   mode="naive_exact")),
        # distribution maps on the moving area light (count, prune and fill beside the verification)
        named("maps_frame", _case("maps", "city", 1_000_000, maps=64)),
        # the first frame of a scene, and the frame without any reuse: every path traced and deposited
        named("trace_all", _case("trace", "city", 1_000_000)),
        # the picture of a frame: photons splatted at the visible points of a full-HD camera
        named("splat_city", _case("splat", "city", 1_000_000, width=1920, height=1080, radius=0.3)),
        # a small preview window of a room
        named("splat_box", _case("splat", "box", 10_000, bounces=3, width=641, height=361, radius=0.12)),
        # one step of fitting lights and object positions: the differentiable atlas and its gradient
        named("fit_step", _case("model", "city", 1_000_000)),
        # a frame under a ray budget: the listed paths of largest score are re-traced, the others wait
        named("budget_frame", _case("budget", "district", 400_003, tris=100_000, lights=2, bounces=6, tori=4,
                                    budget=20_000)),
        # several scenes of uneven size advanced by one call (a server, or several levels of one game)
        named("batch", _case("batch", "district", 1_600_000, tris=100_000, scenes=6, bounces=0, lights=0, tori=0)),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "carried", "calls", "maps", "trace", "splat", "model", "budget", "batch"])
    c = _case(kind, "district", _log(rng, 10_000, 1_000_000), tris=_log(rng, 12_000, 200_000),
              lights=rng.randint(1, 3), bounces=rng.randint(1, 7), tori=rng.randint(1, 4), atlas=_log(rng, 128, 1024))
    if kind in ("frame", "carried", "calls"):
        c["mode"] = rng.choice(["error", "error", "naive_aabb", "naive_exact", "error_exact"])
        c["point_moves"] = c["lights"] > 1 and rng.random() < 0.3
    elif kind == "maps":
        c["maps"] = rng.choice([8, 16, 33, 64])
    elif kind == "splat":
        c["width"], c["height"] = _log(rng, 320, 1920), _log(rng, 180, 1080)
        c["radius"] = round(rng.uniform(0.1, 0.4), 3)
    elif kind == "budget":
        c["budget"] = _log(rng, 100, 50_000)
    elif kind == "batch":
        c.update(scenes=rng.randint(2, 6), bounces=0, lights=0, tori=0)
    return c


# ---------------------------------------------------------------- scenes
@functools.lru_cache(maxsize=6)
def _scene(kind, tris, paths, lights, bounces, tori):
    if kind == "box":
        return scenes.tiny_box(n_paths=paths)
    if kind == "city":
        return scenes.city(n_paths=paths)
    if kind == "villa":
        return scenes.villa(n_paths_per_light=paths // 3)
    return scenes.district(tris, paths, lights, bounces, tori, seed=5)


def _scene_of(c):
    return _scene(c["scene"], c["tris"], c["paths"], c["lights"], c["bounces"], c["tori"])


def _batch_scenes(c):
    """Uneven districts: triangles and paths log-spaced, the most triangles with the fewest paths."""
    k = c["scenes"]
    tri = np.geomspace(max(12_000, c["tris"] // 8), c["tris"], k)
    w = np.geomspace(12.0, 1.0, k)
    return [_scene("district", int(tri[i]), max(1000, int(c["paths"] * w[i] / w.sum())), 1 + i % 3, 1 + (3 * i + 3) % 7,
                   1 + i % 4) for i in range(k)]


def _lights(sc, c, f):
    ls = sc.lights(f)
    if c["point_moves"]:       # the point light walks 0.05 m a frame, the other lights stand still
        ls = [replace(l, pos=(l.pos[0] + 0.05 * (f - 1), l.pos[1], l.pos[2])) if l.type == scenes.LIGHT_POINT else l
              for l in sc.lights(1)]
    return [l.as_f32() for l in ls]


def _maps(c):
    m = c["maps"]
    return {"dm_rect": (8, 8, m, m), "dm_point": (m, m)} if m else {}


class _Scene:
    """A built scene, the paths traced at its first pose, and the motion that follows."""

    def __init__(self, sc, c, seed):
        self.sc, self.seed = sc, int(seed)
        self.first = 1 + int(seed) % 8
        self.handle = pv.pv_build_scene(sc.verts, sc.tri_object, sc.object_dynamic, sc.object_albedo,
                                        _lights(sc, c, self.first), sc.max_bounces, sc.diag,
                                        object_xform=sc.xforms(self.first), **_maps(c))
        self.paths = pv.Paths.allocate(sc.n_paths, sc.max_bounces)
        self.poses = [(np.ascontiguousarray(sc.xforms(self.first + i), np.float32), _lights(sc, c, self.first + i))
                      for i in range(POSES)]
        self.packed = [pv.make_lights(l) for _, l in self.poses]
        self.at, self.frame = 0, 1
        pv.pv_trace_all(self.handle, self.paths, self.seed, self.frame)

    def next_pose(self):
        """Index of the next pose, forth and back."""
        self.at, self.frame = self.at + 1, self.frame + 1
        i = self.at % (2 * POSES - 2)
        return i if i < POSES else 2 * POSES - 2 - i

    def records(self):
        p = self.paths
        return {"info": p.info, "origin": p.origin, "position": p.pa[..., :3], "prim": p.pa.view(torch.int32)[..., 3],
                "energy": p.pb}

    def __del__(self):
        h, self.handle = getattr(self, "handle", None), None
        if h:
            pv.pv_destroy_scene(h)


class _State:
    def __init__(self, c):
        self.case, self.batch = c, None

    def __del__(self):
        if self.batch:
            pv.pv_batch_destroy(self.batch)


def _camera(c, sc):
    if c["scene"] == "box":
        pos, target = (0.0, 1.5, 0.95), (0.0, 0.2, -0.4)
    else:
        h = sc.atlas_rect[2]
        pos, target = (0.0, 0.9 * h, 0.7 * h), (0.0, 0.0, 0.0)
    return pv.PvCamera.make(pos, target, (0.0, 1.0, 0.0), math.radians(60.0), c["width"], c["height"])


def _fit_inputs(c, sc, theta, seed):
    """The parameters a fit has reached, and the gradient of its loss with respect to the atlas."""
    n_lights = len(sc.lights(1))
    th = scenes.perturbed_theta(theta, n_lights, seed=2111 + int(seed))
    g = torch.Generator().manual_seed(int(seed))
    grad = torch.randn(c["atlas"] // 8 + 1, c["atlas"] // 8 + 1, 3, generator=g).cuda()
    grad = torch.nn.functional.interpolate(grad.permute(2, 0, 1)[None], size=(c["atlas"], c["atlas"]), mode="bilinear",
                                           align_corners=True)[0].permute(1, 2, 0).contiguous()
    return torch.as_tensor(th, dtype=torch.float32, device="cuda"), grad


def prepare(case, seed):
    c = case
    st = _State(c)
    st.mode, st.flags = MODES[c["mode"]]
    if c["kind"] == "batch":
        st.scenes = [_Scene(sc, c, seed + 7 * i) for i, sc in enumerate(_batch_scenes(c))]
        st.batch = pv.pv_batch_create([(s.handle, s.paths, None, None, None, s.seed) for s in st.scenes], st.mode,
                                      st.scenes[0].sc.tau)
        st.poses = []
        for _ in range(2 * POSES - 2):
            now = [s.poses[s.next_pose()] for s in st.scenes]
            st.poses.append(pv.BatchPoses(len(now), [x for x, _ in now], [l for _, l in now]))
        st.step = 0
        return st
    sc = _scene_of(c)
    s = st.scene = _Scene(sc, c, seed)
    n = sc.n_paths
    if c["kind"] in ("frame", "carried", "calls", "trace", "maps"):
        st.atlas = torch.zeros(c["atlas"], c["atlas"], 3, dtype=torch.int64, device="cuda")
    if c["kind"] == "carried":
        pv.pv_deposit(s.handle, s.paths, st.atlas, sc.atlas_rect, SCALE_LOG2)
    if c["kind"] in ("calls", "budget"):
        st.list = torch.zeros(n, dtype=torch.int32, device="cuda")
        st.count = torch.zeros(1, dtype=torch.int32, device="cuda")
    if c["kind"] == "budget":
        st.kept = torch.zeros_like(st.list)
        st.kept_count = torch.zeros_like(st.count)
        # scores of an earlier gradient: most paths carry a little, a few much, some nothing
        g = torch.Generator().manual_seed(int(seed))
        st.score = (torch.randn(n, generator=g).mul_(2.0).exp_() * (torch.rand(n, generator=g) < 0.9)).cuda()
    if c["kind"] == "splat":
        st.camera = _camera(c, sc)
        st.image = torch.zeros(c["height"], c["width"], 3, dtype=torch.float32, device="cuda")
        st.work = torch.empty(pv.pv_splat_workspace_bytes(s.handle, c["width"], c["height"]), dtype=torch.uint8,
                              device="cuda")
    if c["kind"] == "model":
        st.theta, st.grad = _fit_inputs(c, sc, pv.pv_theta_current(s.handle), seed)
        st.theta.requires_grad_(True)
    return st


def run(state):
    st, c = state, state.case
    kind = c["kind"]
    if kind == "batch":
        st.step += 1
        pv.pv_batch_frame(st.batch, st.poses[(st.step - 1) % len(st.poses)], None, 1 + st.step)
        return [s.records() for s in st.scenes]
    s = st.scene
    sc, h, P = s.sc, s.handle, s.paths
    if kind == "splat":
        pv.pv_splat(h, P, st.camera, c["radius"], st.image, st.work)
        return st.image
    if kind == "model":
        atlas = pv.model_deposit(h, P, st.theta, c["atlas"], c["atlas"], sc.atlas_rect)
        (g,) = torch.autograd.grad(atlas, st.theta, st.grad)
        return {"atlas": atlas.detach(), "theta_grad": g}
    i = s.next_pose()
    pv.pv_update_dynamic(h, s.poses[i][0], s.packed[i])
    if kind == "frame":
        pv.pv_verify_retrace_deposit(h, P, st.mode, sc.tau, st.flags, s.seed, s.frame, st.atlas, sc.atlas_rect,
                                     SCALE_LOG2)
    elif kind == "carried":
        pv.pv_verify_retrace_deposit_delta(h, P, st.mode, sc.tau, st.flags, s.seed, s.frame, st.atlas, sc.atlas_rect,
                                           SCALE_LOG2)
    elif kind == "maps":
        pv.pv_verify_retrace(h, P, st.mode, sc.tau, st.flags, s.seed, s.frame)
        pv.pv_deposit(h, P, st.atlas, sc.atlas_rect, SCALE_LOG2)
    elif kind == "trace":
        pv.pv_trace_all_deposit(h, P, s.seed, s.frame, st.atlas, sc.atlas_rect, SCALE_LOG2)
    elif kind == "calls":
        pv.pv_verify_paths(h, P, st.mode, sc.tau, st.flags, st.list, st.count, seed=s.seed, frame=s.frame)
        pv.pv_retrace_invalid(h, P, st.list, st.count, s.seed, s.frame)
        pv.pv_deposit(h, P, st.atlas, sc.atlas_rect, SCALE_LOG2)
        return {**s.records(), "atlas": st.atlas, "list": st.list, "count": st.count}
    elif kind == "budget":
        pv.pv_verify_paths(h, P, st.mode, sc.tau, st.flags, st.list, st.count, seed=s.seed, frame=s.frame)
        pv.pv_budget_list(h, st.list, st.count, st.score, c["budget"], st.kept, st.kept_count)
        pv.pv_retrace_invalid(h, P, st.kept, st.kept_count, s.seed, s.frame)
        return {**s.records(), "list": st.list, "count": st.count, "kept": st.kept, "kept_count": st.kept_count}
    return {**s.records(), "atlas": st.atlas}


# ---------------------------------------------------------------- least work of a pass
# Photons a path stores, rays that a reuse frame traces per path, and 4-wide node visits and triangle
# tests of a ray, as measured per scene (a node visit is 80 operations, a triangle test 35).
_PER = {"box": (2.1, 0.02, 4.0, 6.0), "city": (2.0, 0.48, 15.3, 2.1), "villa": (3.1, 0.44, 21.7, 2.4),
        "district": (1.9, 0.4, 14.0, 2.1)}


def _photons(c):
    return min(_PER[c["scene"]][0], float(c["bounces"] or 4)) * c["paths"]


def work(case):
    c = case
    n, ph = c["paths"], _photons(c)
    _, rays, nodes, tris = _PER[c["scene"]]
    per_ray = 80.0 * nodes + 35.0 * tris
    atlas = 24.0 * c["atlas"] ** 2
    kind = c["kind"]
    if kind == "trace":            # every path written, the atlas written
        return {"bytes": 16.0 * n + 32.0 * ph + atlas, "flops": (n + ph) * per_ray}
    if kind == "splat":            # every photon and its predecessor's position read, the image written
        px = c["width"] * c["height"]
        return {"bytes": 16.0 * n + 32.0 * ph + 12.0 * px, "flops": px * per_ray + 60.0 * ph}
    if kind == "model":            # paths read forward and backward, atlas written, its gradient read
        return {"bytes": 2.0 * (16.0 * n + 32.0 * ph) + 24.0 * c["atlas"] ** 2, "flops": 2.0 * ph * 250.0}
    least = 16.0 * n + 16.0 * ph + rays * n * 48.0          # verification reads, re-traced paths written
    if kind == "batch":
        return {"bytes": least, "flops": rays * n * per_ray + 40.0 * ph}
    if kind == "budget":
        return {"bytes": 16.0 * n + 16.0 * ph + 12.0 * n, "flops": c["budget"] * 2.0 * per_ray + 40.0 * ph}
    return {"bytes": least + 16.0 * ph + atlas, "flops": rays * n * per_ray + 40.0 * ph}


# ---------------------------------------------------------------- results in 64 bits
def exact(case, seed):
    """The splat of a small room and the model with its gradient, in float64 by plain torch.

    Frames and traces give None: they follow every path of large scenes through all triangles, far over
    twenty seconds in 64 bits, and what they decide is in whole numbers (info, primitives, lists, the
    fixed-point atlas).  So does the splat of a large scene (a primary ray per pixel through all
    triangles)."""
    if case["kind"] == "model":
        return _exact_model(case, seed)
    if case["kind"] == "splat" and case["scene"] == "box":
        return _exact_splat(case, seed)
    return None


def _world(sc, frame):
    """World corners [T, 3, 3] and unit-less normals [T, 3] at a frame, float64 on the GPU."""
    v = torch.as_tensor(sc.world_verts(frame), dtype=torch.float64, device="cuda")
    return v, torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])


def _stored(s):
    r = s.records()
    nseg = torch.bitwise_and(r["info"] >> pv.PV_INFO_NSEG_SHIFT, 15).long()
    light = torch.bitwise_and(r["info"] >> 20, 3).long()
    return nseg, light, r["origin"].double().T, r["position"].double(), r["prim"].long(), r["energy"][..., :3].double()


def _exact_model(c, seed):
    st = prepare(c, seed)
    s = st.scene
    sc = s.sc
    _, normal = _world(sc, s.first)
    nseg, light, o0, x, prim, energy = _stored(s)
    lights = _lights(sc, c, s.first)
    f64 = dict(dtype=torch.float64, device="cuda")
    th = st.theta.detach().double().requires_grad_(True)
    dyn = np.nonzero(sc.object_dynamic)[0]
    slot_of = np.full(sc.n_objects, -1)
    slot_of[dyn] = np.arange(len(dyn))
    slot = torch.as_tensor(slot_of[sc.tri_object], device="cuda")
    now = torch.as_tensor(sc.xforms(s.first)[dyn][:, [3, 7, 11]].astype(np.float64), **f64)
    moved = th[7 * len(lights):].reshape(-1, 3) - now
    W = H = c["atlas"]
    x0, z0, x1, z1 = (float(np.float32(v)) for v in sc.atlas_rect)
    atlas = torch.zeros(H * W, 3, **f64)

    def taps(f):
        return torch.stack([(1 - f) ** 3 / 6, (3 * f ** 3 - 6 * f ** 2 + 4) / 6,
                            (-3 * f ** 3 + 3 * f ** 2 + 3 * f + 1) / 6, f ** 3 / 6], -1)

    for li, lt in enumerate(lights):
        ids = torch.nonzero((light == li) & (nseg > 0)).flatten()
        tl = th[7 * li:7 * li + 7]
        d = x[0, ids] - o0[ids]
        if lt.type == scenes.LIGHT_POINT:
            prev = tl[:3].expand_as(d)
        else:
            pos, n, t = (torch.tensor(v, **f64) for v in (lt.pos, lt.normal, lt.tangent))
            b = torch.linalg.cross(n, t)
            rel = o0[ids] - pos
            bl = torch.linalg.cross(tl[3:6], t)
            prev = tl[:3] + (rel @ t)[:, None] * t + (rel @ b)[:, None] * bl
            d = (d @ t)[:, None] * t + (d @ b)[:, None] * bl + (d @ n)[:, None] * tl[3:6]
        for k in range(sc.max_bounces):
            on = nseg[ids] > k
            ids, prev, d = ids[on], prev[on], d[on]
            pr = prim[k, ids]
            nu = torch.nn.functional.normalize(normal[pr], dim=1)
            q = x[k, ids] + torch.where(slot[pr][:, None] >= 0, moved[slot[pr].clamp(min=0)], torch.zeros_like(prev))
            y = prev + ((nu * (q - prev)).sum(1) / (nu * d).sum(1))[:, None] * d
            u = (y[:, 0] - x0) * (W / (x1 - x0)) - 0.5
            v = (y[:, 2] - z0) * (H / (z1 - z0)) - 0.5
            wx, wz = taps(u - u.detach().floor()), taps(v - v.detach().floor())
            i0, j0 = u.detach().floor().long() - 1, v.detach().floor().long() - 1
            e = tl[6] * energy[k, ids]
            for r in range(4):
                for q4 in range(4):
                    ti, tj = i0 + q4, j0 + r
                    ok = (ti >= 0) & (ti < W) & (tj >= 0) & (tj < H)
                    atlas = atlas.index_add(0, (tj * W + ti)[ok], (e * (wx[:, q4] * wz[:, r])[:, None])[ok])
            if k + 1 < sc.max_bounces:
                d = x[k + 1, ids] - x[k, ids]
            prev = y
    atlas = atlas.reshape(H, W, 3)
    (g,) = torch.autograd.grad(atlas, th, st.grad.double())
    return {"atlas": atlas.detach(), "theta_grad": g}


def _exact_splat(c, seed):
    st = prepare(c, seed)
    s = st.scene
    sc = s.sc
    f64 = dict(dtype=torch.float64, device="cuda")
    tri, normal = _world(sc, s.first)
    nseg, _, o0, x, _, energy = _stored(s)
    cam = st.camera
    unit = torch.nn.functional.normalize
    pos = torch.tensor(list(cam.pos), **f64)
    fwd = unit(torch.tensor(list(cam.target), **f64) - pos, dim=0)
    right = unit(torch.linalg.cross(fwd, torch.tensor(list(cam.up), **f64)), dim=0)
    up = torch.linalg.cross(right, fwd)
    ty = math.tan(0.5 * cam.fov_y)
    tx = ty * cam.width / cam.height
    px = (2 * (torch.arange(cam.width, **f64) + 0.5) / cam.width - 1) * tx
    py = (1 - 2 * (torch.arange(cam.height, **f64) + 0.5) / cam.height) * ty
    d = unit((fwd + px[None, :, None] * right + py[:, None, None] * up).reshape(-1, 3), dim=1)
    best = torch.full((d.shape[0],), math.inf, **f64)
    hit = torch.full((d.shape[0],), -1, dtype=torch.long, device="cuda")
    for i in range(tri.shape[0]):
        e1, e2, sv = tri[i, 1] - tri[i, 0], tri[i, 2] - tri[i, 0], pos - tri[i, 0]
        p = torch.linalg.cross(d, e2.expand_as(d))
        q = torch.linalg.cross(sv, e1)
        det = p @ e1
        u, v, t = (p @ sv) / det, (d @ q) / det, (e2 @ q) / det
        ok = (det != 0) & (u >= 0) & (v >= 0) & (u + v <= 1) & (t > 0) & (t < best)
        best, hit = torch.where(ok, t, best), torch.where(ok, torch.full_like(hit, i), hit)
    seen = hit >= 0
    P = pos + best[seen, None] * d[seen]
    nrm = unit(normal[hit[seen]], dim=1)
    nrm = torch.where(((nrm * d[seen]).sum(1) > 0)[:, None], -nrm, nrm)
    alb = torch.as_tensor(sc.object_albedo[sc.tri_object].astype(np.float64), **f64)[hit[seen]]
    r = float(np.float32(c["radius"]))
    at, came, e = [], [], []
    for k in range(sc.max_bounces):
        ids = torch.nonzero(nseg > k).flatten()
        at.append(x[k, ids])
        came.append(x[k, ids] - (x[k - 1, ids] if k else o0[ids]))
        e.append(energy[k, ids])
    at, came, e = torch.cat(at), torch.cat(came), torch.cat(e)
    near = (at - pos) @ fwd - r * fwd.abs().sum()
    front = near > 1e-3 * sc.diag
    at, came, e = at[front], came[front], e[front]
    total = torch.zeros_like(P)
    for b in range(0, P.shape[0], 4096):
        Pb, nb = P[b:b + 4096], nrm[b:b + 4096]
        s2 = sum((Pb[:, a, None] - at[None, :, a]) ** 2 for a in range(3)) / (r * r)
        total[b:b + 4096] = torch.where((s2 < 1) & (nb @ came.T < 0), 1 - s2, torch.zeros_like(s2)) @ e
    image = torch.zeros(cam.height * cam.width, 3, **f64)
    image[seen] = alb / math.pi * total * (2 / (math.pi * r * r))
    return image.reshape(cam.height, cam.width, 3)
