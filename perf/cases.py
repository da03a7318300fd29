"""The work a user of this framework has it do, as cases that can be timed.

Each case goes through the public entry points (paper_2008_00326_gb300.perch,
the binding of include/perch.h).  Scenes are the seeded synthetic ones of
paper_2008_00326_gb300.scenes at the sizes of the repository's workloads, and
ragged sizes between them.  Kinds of call:

    argmin   the per-object argmin alone over resident costs
    search   score + argmin per object, poses and costs resident (device mode)
    few      a handful of poses scored from host memory, and their argmin
    refine   generalised-ICP refinement of resident poses
    batch    many scenes' searches in one call
    tree     the scene-generation tree search (host mode)
    served   a burst of requests to the continuous-batching server
    frame    a camera frame from host arrays to the best poses, then released
    errors   ADD-S / ADD of pose pairs
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2008_00326_gb300 import perch as P
from paper_2008_00326_gb300 import scenes as S


def listed():
    return [
        # the argmin of each of five objects over a long search, with the caller's ids
        {"name": "argmin_300k", "kind": "argmin", "objects": 5, "n": 300001, "ids": True},
        # the smallest search of the repository: one coarse box on a small image, colour off
        {"name": "search_small", "kind": "search", "scene": "small", "W": 160, "H": 120, "tri": 1.0, "objects": 1,
         "grid": 5, "yaws": 8, "colour": False, "stride": 1, "jo_mode": 0, "margin": 100},
        # a few candidate poses checked again (after refinement or tracking): latency
        {"name": "few_vga", "kind": "few", "scene": "table", "W": 640, "H": 480, "tri": 1.0, "object": 0, "n": 24,
         "colour": True, "stride": 1},
        # the benchmark: three objects on a table, 43 x 43 positions x 16 yaws each, colour on
        {"name": "search_table", "kind": "search", "scene": "table", "W": 640, "H": 480, "tri": 1.0, "objects": 3,
         "grid": 21, "yaws": 16, "colour": True, "stride": 1, "jo_mode": 0, "margin": 100},
        # the 6-DoF workload: five 30k-triangle objects, labels and regions of interest
        {"name": "search_sixdof", "kind": "search", "scene": "sixdof", "W": 640, "H": 480, "tri": 1.0, "objects": 5,
         "n": 4096, "colour": True, "stride": 1, "jo_mode": 0, "margin": 100},
        # an odd image and an odd search, both clouds down-sampled, Eq. 3 as written, no occluder marking
        {"name": "search_eq3_odd", "kind": "search", "scene": "table", "W": 517, "H": 389, "tri": 0.35, "objects": 2,
         "grid": 9, "yaws": 7, "colour": True, "stride": 2, "jo_mode": 1, "margin": -1},
        # the 6-DoF workload's poses refined against the observation at stride 2
        {"name": "refine_sixdof", "kind": "refine", "W": 640, "H": 480, "tri": 1.0, "objects": 5, "n": 4096,
         "stride": 2, "iters": 10},
        # sixteen quarter-size scenes of one to six objects (500-30k triangles), uneven searches
        {"name": "batch_16", "kind": "batch", "scenes": 16, "W": 320, "H": 240, "lo": 500, "hi": 40000},
        # the tree over three objects, beam 4
        {"name": "tree_beam4", "kind": "tree", "W": 640, "H": 480, "tri": 1.0, "grid": 10, "yaws": 16, "beam": 4},
        # requests of uneven size from two resident scenes, arriving at once
        {"name": "served_burst", "kind": "served", "requests": 24, "lo": 120, "hi": 4096, "W": 640, "H": 480,
         "tri": 1.0},
        # one camera frame: observation, proposals, scores and best pose of each of its five objects
        {"name": "frame_vga", "kind": "frame", "W": 640, "H": 480, "tri": 1.0, "objects": 5, "M": 42, "N": 8, "K": 3,
         "stride": 1},
        # pose errors of an evaluation: symmetric, 10k vertices
        {"name": "errors_adds", "kind": "errors", "verts": 10001, "n": 200, "symmetric": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo_w=160, hi_w=640):
    w = rng.randint(lo_w, hi_w)
    return w, max(90, int(w * rng.uniform(0.6, 0.8)))


def draw(rng):
    kind = rng.choice(("argmin", "search", "search", "search", "few", "refine", "batch", "tree", "served", "frame",
                       "errors"))
    w, h = _size(rng)
    tri = round(math.exp(rng.uniform(math.log(0.05), 0.0)), 4)
    if kind == "argmin":
        return {"kind": kind, "objects": rng.randint(2, 6), "n": _log(rng, 500, 2000000), "ids": rng.random() < 0.5}
    if kind == "search":
        scene = rng.choice(("small", "table", "sixdof"))
        c = {"kind": kind, "scene": scene, "W": w, "H": h, "tri": tri, "colour": rng.random() < 0.7,
             "stride": rng.choice((1, 1, 1, 2, 3)), "jo_mode": int(rng.random() < 0.2),
             "margin": rng.choice((100, 100, 60, -1))}
        if scene == "small":
            w = rng.randint(120, 320)
            c.update(W=w, H=3 * w // 4, tri=1.0, objects=1, grid=rng.randint(2, 9), yaws=rng.randint(3, 16))
        elif scene == "table":
            c.update(objects=rng.randint(1, 3), grid=_log(rng, 1, 14), yaws=rng.randint(1, 16))
        else:
            c.update(objects=rng.randint(1, 5), n=_log(rng, 8, 4096))
        return c
    if kind == "few":
        return {"kind": kind, "scene": rng.choice(("small", "table", "sixdof")), "W": w, "H": h, "tri": tri, "object": 0,
                "n": rng.randint(1, 200), "colour": rng.random() < 0.7, "stride": rng.choice((1, 1, 2))}
    if kind == "refine":
        return {"kind": kind, "W": w, "H": h, "tri": tri, "objects": rng.randint(1, 5), "n": _log(rng, 8, 2048),
                "stride": rng.choice((1, 2, 2, 3)), "iters": rng.randint(3, 20)}
    if kind == "batch":
        return {"kind": kind, "scenes": rng.randint(2, 16), "W": rng.randint(200, 320), "H": rng.randint(150, 240),
                "lo": 100, "hi": _log(rng, 500, 20000)}
    if kind == "tree":
        return {"kind": kind, "W": w, "H": h, "tri": tri, "grid": rng.randint(1, 8), "yaws": rng.randint(2, 16),
                "beam": rng.randint(1, 6)}
    if kind == "served":
        return {"kind": kind, "requests": rng.randint(4, 40), "lo": 30, "hi": _log(rng, 200, 4000), "W": w, "H": h,
                "tri": tri}
    if kind == "frame":
        return {"kind": kind, "W": w, "H": h, "tri": tri, "objects": rng.randint(1, 5), "M": rng.randint(6, 42),
                "N": rng.randint(2, 8), "K": rng.randint(1, 4), "stride": rng.choice((1, 1, 2))}
    return {"kind": "errors", "verts": _log(rng, 300, 10000), "n": rng.randint(3, 200), "symmetric": rng.random() < 0.8}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

# camera distances of the tabletop scenes (metres)
_SMALL_DIST, _TABLE_DIST = 0.53, 1.05


def _scene(kind, c, seed):
    """A Scene whose requests hold no pose set yet (one placeholder pose)."""
    if kind == "small":
        return S.tabletop_small(seed=seed, W=c["W"], H=c["H"])
    if kind == "table":
        return S.tabletop_3obj(seed=seed, W=c["W"], H=c["H"], grid_half=0, n_yaw=16, tri_scale=c["tri"])
    return S.sixdof_5obj(seed=seed, W=c["W"], H=c["H"], n_hyp=1, tri_scale=c["tri"])


def _grid(dist, gt, half, yaws, step):
    """(2 half + 1)^2 positions around the pose gt times `yaws` yaws, on the table."""
    r_wc, t_wc = S.look_at(dist, 50.0)
    at = r_wc.T @ (np.asarray(gt).reshape(3, 4)[:, 3] - t_wc)
    off = np.arange(-half, half + 1) * step
    x, y = np.meshgrid(at[0] + off, at[1] + off, indexing="ij")
    xy = np.stack([x.ravel(), y.ravel(), np.zeros(x.size)], 1)
    t = xy @ r_wc.T + t_wc
    r = np.stack([r_wc @ S.rot_z(2 * math.pi * k / yaws) for k in range(yaws)])
    out = np.empty((len(t), yaws, 3, 4))
    out[:, :, :, :3] = r[None]
    out[:, :, :, 3] = t[:, None]
    return out.reshape(-1, 12).astype(np.float32)


def _around(rng, gt, n, sigma_t=0.02, sigma_deg=15.0):
    """n poses around gt: N(0, sigma_t) translations, N(0, sigma_deg) rotations about random axes."""
    g = np.asarray(gt).reshape(3, 4)
    r = S.rodrigues_batch(rng.normal(size=(n, 3)), np.radians(rng.normal(0.0, sigma_deg, size=n))) @ g[:, :3]
    t = g[:, 3] + rng.normal(0.0, sigma_t, size=(n, 3))
    return np.concatenate([r, t[:, :, None]], 2).reshape(n, 12).astype(np.float32)


def _poses(kind, c, sc, k, rng, half=None, yaws=None, n=None):
    if kind == "sixdof" or n is not None:
        return _around(rng, sc.gt_poses[k], n if n is not None else c["n"])
    if kind == "small":
        return _grid(_SMALL_DIST, sc.gt_poses[k], half, yaws, 0.02)
    return _grid(_TABLE_DIST, sc.gt_poses[k], half, yaws, 0.01)


class _State:
    """What a user's program holds: a context with resident meshes (and scenes), its stream and buffers."""

    def __init__(self, case):
        self.case = case
        self.ctx = P.Context(0)
        self.stream = torch.cuda.Stream()
        self.server = None

    def __del__(self):
        try:
            if self.server is not None:
                self.server.stop()
            torch.cuda.synchronize()
            self.ctx.close()
        except Exception:
            pass


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    st = _State(case)
    if kind == "argmin":
        n = case["n"]
        st.objs = [(_dev(rng.integers(150, 6000, size=(n, 2)).astype(np.int32)),
                    _dev(rng.permutation(n).astype(np.int64)) if case["ids"] else None,
                    torch.zeros(1, dtype=torch.int64, device="cuda"),
                    torch.zeros(1, dtype=torch.int32, device="cuda")) for _ in range(case["objects"])]
    elif kind == "search":
        sc = _scene(case["scene"], case, seed)
        st.sid = st.ctx.set_observation(sc, color_check=int(case["colour"]), stride=case["stride"],
                                        jo_mode=case["jo_mode"], occ_margin_units=case["margin"])
        st.objs = []
        for k, r in enumerate(sc.requests[:case["objects"]]):
            poses = _poses(case["scene"], case, sc, k, rng, case.get("grid"), case.get("yaws"))
            st.objs.append((st.ctx.load_mesh(sc.meshes[k]), r.label, r.roi, _dev(poses),
                            torch.zeros((len(poses), 2), dtype=torch.int32, device="cuda"),
                            torch.zeros(1, dtype=torch.int64, device="cuda"),
                            torch.zeros(1, dtype=torch.int32, device="cuda")))
    elif kind == "few":
        sc = _scene(case["scene"], case, seed)
        r = sc.requests[case["object"]]
        st.sid = st.ctx.set_observation(sc, color_check=int(case["colour"]), stride=case["stride"])
        st.obj = (st.ctx.load_mesh(sc.meshes[case["object"]]), r.label, r.roi)
        st.poses = _poses(case["scene"], case, sc, case["object"], rng, n=case["n"])
    elif kind == "refine":
        sc = _scene("sixdof", case, seed)
        st.sid = st.ctx.set_observation(sc, stride=case["stride"])
        st.params = P.perch_default_gicp_params(max_iterations=case["iters"])
        st.objs = []
        for k, r in enumerate(sc.requests[:case["objects"]]):
            poses = _dev(_poses("sixdof", case, sc, k, rng))
            st.objs.append((st.ctx.load_mesh(sc.meshes[k]), r.label, r.roi, poses, torch.empty_like(poses),
                            torch.zeros((len(poses), 2), dtype=torch.int32, device="cuda")))
    elif kind == "batch":
        scs = S.batched_scenes(seed=seed, n_scenes=case["scenes"], W=case["W"], H=case["H"],
                               hyp_range=(8, 8), pool=_pool())
        mids = {id(m): st.ctx.load_mesh(m) for m in _pool()}
        specs, poses, at = [], [], 0
        for sc, total in zip(scs, _totals(case, case["scenes"])):
            sid = st.ctx.set_observation(sc)
            k = len(sc.requests)
            share = rng.multinomial(total - k, np.ones(k) / k) + 1
            for r, gt, n in zip(sc.requests, sc.gt_poses, share):
                specs.append((sid, mids[id(sc.meshes[r.mesh_index])], r.label, r.roi, at, int(n)))
                poses.append(_around(rng, gt, int(n)))
                at += int(n)
        st.items = P.work_items(specs)
        st.poses = _dev(np.concatenate(poses))
        st.costs = torch.zeros((at, 2), dtype=torch.int32, device="cuda")
    elif kind == "tree":
        sc = _scene("table", case, seed)
        st.sid = st.ctx.set_observation(sc)
        st.objs = [(st.ctx.load_mesh(sc.meshes[k]), r.label, r.roi,
                    _poses("table", case, sc, k, rng, case["grid"], case["yaws"])) for k, r in enumerate(sc.requests)]
    elif kind == "served":
        kinds = []
        for name in ("table", "sixdof"):
            sc = _scene(name, case, seed)
            sid = st.ctx.set_observation(sc)
            kinds += [(sid, st.ctx.load_mesh(sc.meshes[k]), r.label, r.roi, sc.gt_poses[k])
                      for k, r in enumerate(sc.requests)]
        st.requests = []
        for n in _totals(case, case["requests"], log=True):
            sid, mid, label, roi, gt = kinds[int(rng.integers(len(kinds)))]
            st.requests.append((sid, mid, label, roi, _around(rng, gt, n)))
        st.server = P.Server(st.ctx, slots=2, max_batch_hypotheses=1 << 15)
    elif kind == "frame":
        st.scene = _scene("sixdof", case, seed)
        st.objs = [(st.ctx.load_mesh(st.scene.meshes[k]), r.label, r.roi)
                   for k, r in enumerate(st.scene.requests[:case["objects"]])]
    else:
        mesh, true, est = _error_inputs(case, seed)
        st.mid = st.ctx.load_mesh(mesh)
        st.true, st.est = _dev(true), _dev(est)
        st.out = torch.zeros(case["n"], dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return st


def _totals(case, count, log=False):
    """Uneven hypothesis counts between lo and hi, the same for every seed (outputs keep their shapes)."""
    f = np.random.default_rng(count).uniform(size=count)
    lo, hi = case["lo"], case["hi"]
    return [int(round(x)) for x in (lo * (hi / lo) ** f if log else lo + (hi - lo) * f)]


@functools.lru_cache(maxsize=None)
def _pool():
    return S.mesh_pool()


def _error_inputs(case, seed):
    """An ellipsoid of about case["verts"] vertices, true poses, and estimates a few degrees and millimetres off."""
    rng = np.random.default_rng(seed)
    nlon = max(4, int(round(math.sqrt(case["verts"]))))
    nlat = max(3, (case["verts"] - 2 + nlon // 2) // nlon + 1)
    mesh = S.ellipsoid_mesh(*rng.uniform(0.03, 0.06, size=3), nlat, nlon)
    n = case["n"]
    true = np.empty((n, 3, 4))
    true[:, :, :3] = S.rodrigues_batch(rng.normal(size=(n, 3)), rng.uniform(0.0, math.pi, size=n))
    true[:, :, 3] = rng.normal(size=(n, 3)) * 0.1 + [0.0, 0.0, 0.9]
    est = true.copy()
    est[:, :, :3] = S.rodrigues_batch(rng.normal(size=(n, 3)), np.radians(rng.normal(0.0, 10.0, size=n))) @ true[:, :, :3]
    est[:, :, 3] += rng.normal(size=(n, 3)) * 0.01
    return mesh, true.reshape(n, 12).astype(np.float32), est.reshape(n, 12).astype(np.float32)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    case, ctx = st.case, st.ctx
    kind = case["kind"]
    if kind == "argmin":
        for costs, ids, best, cost in st.objs:
            ctx.best(costs, ids, stream=st.stream, out_index=best, out_cost=cost)
        return [[best, cost] for _, _, best, cost in st.objs]
    if kind == "search":
        out = []
        for mid, label, roi, poses, costs, best, cost in st.objs:
            ctx.score(st.sid, mid, label, roi, poses, costs, stream=st.stream)
            ctx.best(costs, stream=st.stream, out_index=best, out_cost=cost)
            out.append([costs, best, cost])
        return out
    if kind == "few":
        costs = ctx.score(st.sid, *st.obj, st.poses)
        return [costs, *ctx.best(costs)]
    if kind == "refine":
        out = []
        for mid, label, roi, poses, refined, info in st.objs:
            ctx.refine(st.sid, mid, label, roi, poses, st.params, poses_out=refined, info=info, stream=st.stream)
            out.append([refined, info])
        return out
    if kind == "batch":
        return P.perch_score_batch(ctx.ctx, st.items, st.poses, st.costs, stream=st.stream)
    if kind == "tree":
        order, pose, cost, edges = P.perch_tree_search(ctx.ctx, st.sid, st.objs, case["beam"])
        return [np.array(order), np.array(pose), np.array(cost), edges]
    if kind == "served":
        tickets = [st.server.submit(*r)[0] for r in st.requests]
        out = []
        for t in tickets:
            out.append(st.server.wait(t))
            st.server.release(t)
        return out
    if kind == "frame":
        sid = ctx.set_observation(st.scene, stride=case["stride"])
        out = []
        for mid, label, roi in st.objs:
            poses, zr = P.perch_pose_proposals(ctx.ctx, sid, mid, label, roi, case["M"], case["N"], case["K"])
            costs = ctx.score(sid, mid, label, roi, poses)
            out.append([poses, costs, *zr, *ctx.best(costs)])
        P.perch_release_scene(ctx.ctx, sid)
        return out
    return P.perch_add_s(ctx.ctx, st.mid, st.est, st.true, case["symmetric"], out=st.out, stream=st.stream)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

# 32-bit operations by definition: per vertex transformed and projected, per
# triangle set up, per rendered point (depth, back-projection, its neighbour
# search over about 40 candidates at 8 each), more with the colour test
_VERTEX, _TRIANGLE, _POINT, _COLOUR = 27, 11, 27 + 20 + 320, 150
_TRIS = {"small": 516, "table": 13300, "sixdof": 30000}
_SIZE = {"small": (0.09, 0.53), "table": (0.075, 1.05), "sixdof": (0.08, 0.85)}


def _per_pose(scene, case, colour):
    """(operations per pose, triangles) of an object of the scene at the case's image and mesh size."""
    tris = _TRIS[scene] * (case["tri"] if scene != "small" else 1.0)
    size, dist = _SIZE[scene]
    focal = (150.0 / 160.0 if scene == "small" else 615.0 / 640.0) * case["W"]
    px = (focal * size / dist) ** 2 / case.get("stride", 1) ** 2
    return tris / 2 * _VERTEX + tris * _TRIANGLE + px * (_POINT + (_COLOUR if colour else 0)), tris


def work(case):
    kind = case["kind"]
    px = case.get("W", 0) * case.get("H", 0)
    if kind == "argmin":
        n = case["objects"] * case["n"]
        return {"bytes": n * (16 if case["ids"] else 8) + 12 * case["objects"], "flops": 2 * n}
    if kind == "errors":
        v, n = case["verts"], case["n"]
        return {"bytes": 16 * v + 104 * n, "flops": n * (v * 30 + (8.0 * v * v if case["symmetric"] else 8 * v))}
    if kind == "search":
        n = case["n"] if case["scene"] == "sixdof" else (2 * case["grid"] + 1) ** 2 * case["yaws"]
        ops, tris = _per_pose(case["scene"], case, case["colour"])
        return {"bytes": case["objects"] * (56 * n + 20 * tris) + 9 * px, "flops": case["objects"] * n * ops}
    if kind == "few":
        ops, tris = _per_pose(case["scene"], case, case["colour"])
        return {"bytes": 56 * case["n"] + 20 * tris + 9 * px, "flops": case["n"] * ops}
    if kind == "refine":
        ops, tris = _per_pose("sixdof", case, False)
        return {"bytes": case["objects"] * (104 * case["n"] + 20 * tris) + 9 * px,
                "flops": case["objects"] * case["n"] * ops * 2}
    if kind == "batch":
        n = case["scenes"] * 0.5 * (case["lo"] + case["hi"])
        ops, tris = _per_pose("sixdof", dict(case, tri=0.375), True)
        return {"bytes": 56 * n + case["scenes"] * 9 * px + 20 * 67500, "flops": n * ops}
    if kind == "tree":
        n = (2 * case["grid"] + 1) ** 2 * case["yaws"]
        ops, tris = _per_pose("table", case, True)
        edges = n * (3 + 2 * case["beam"] + case["beam"])
        return {"bytes": 3 * (48 * n + 20 * tris) + 8 * edges + 9 * px, "flops": edges * ops}
    if kind == "served":
        n = case["requests"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        ops, tris = _per_pose("sixdof", case, True)
        return {"bytes": 56 * n + 2 * 9 * px + 8 * 20 * tris, "flops": n * ops}
    n = case["objects"] * case["M"] * case["N"] * case["K"]
    ops, tris = _per_pose("sixdof", case, True)
    return {"bytes": 104 * n + 9 * px + case["objects"] * 20 * tris, "flops": n * ops + 60 * px}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _proposals64(sc, mesh, r, M, N, K):
    """Viewpoints of a Fibonacci lattice x in-plane angles x depths of the labelled box (poses, M N K x 12)."""
    u0, v0, u1, v1 = (max(0, r.roi[0]), max(0, r.roi[1]), min(sc.W, r.roi[2]), min(sc.H, r.roi[3]))
    d = sc.depth[v0:v1, u0:u1][sc.labels[v0:v1, u0:u1] == r.label]
    d = d[d > 0]
    z0, z1 = (d.min() / 1e4, d.max() / 1e4) if d.size else (0.0, 0.0)
    i = np.arange(M)
    y = 1.0 - (2.0 * i + 1.0) / M
    rad = np.sqrt(np.maximum(0.0, 1.0 - y * y))
    phi = math.pi * (3.0 - math.sqrt(5.0)) * i
    fwd = -np.stack([rad * np.cos(phi), y, rad * np.sin(phi)], 1)
    right = np.cross(fwd, [0.0, 0.0, 1.0])
    flat = np.linalg.norm(right, axis=1) < 1e-6
    right[flat] = np.cross(fwd[flat], [0.0, 1.0, 0.0])
    right /= np.linalg.norm(right, axis=1, keepdims=True)
    view = np.stack([right, np.cross(fwd, right), fwd], 1)
    spin = np.stack([S.rot_z(2 * math.pi * k / N) for k in range(N)])
    R = np.einsum("kab,ibc->ikac", spin, view)
    z = z0 + (z1 - z0) * np.arange(K) / (K - 1) if K > 1 else np.array([0.5 * (z0 + z1)])
    c = np.stack([(0.5 * (u0 + u1 - 1) - sc.cx) * z / sc.fx, (0.5 * (v0 + v1 - 1) - sc.cy) * z / sc.fy, z], 1)
    m = 0.5 * (mesh.verts.min(0).astype(np.float64) + mesh.verts.max(0).astype(np.float64))
    out = np.empty((M, N, K, 3, 4))
    out[..., :3] = R[:, :, None]
    out[..., 3] = c[None, None] - np.einsum("ikab,b->ika", R, m)[:, :, None]
    return out.reshape(-1, 12)


def exact(case, seed):
    if case["kind"] == "frame":
        sc = _scene("sixdof", case, seed)
        return [[_proposals64(sc, sc.meshes[k], r, case["M"], case["N"], case["K"]), None, None, None, None, None]
                for k, r in enumerate(sc.requests[:case["objects"]])]
    if case["kind"] != "errors":
        return None          # whole numbers, and poses that follow from a chain of discrete matches
    mesh, true, est = _error_inputs(case, seed)
    v = _dev(mesh.verts.astype(np.float64))
    out = []
    for a, b in zip(est.astype(np.float64).reshape(-1, 3, 4), true.astype(np.float64).reshape(-1, 3, 4)):
        x = v @ _dev(a[:, :3]).T + _dev(a[:, 3])
        y = v @ _dev(b[:, :3]).T + _dev(b[:, 3])
        if case["symmetric"]:
            near = [((x[i:i + 1024, None] - y[None]) ** 2).sum(-1).amin(1).sqrt() for i in range(0, len(x), 1024)]
            out.append(torch.cat(near).mean())
        else:
            out.append((x - y).norm(dim=1).mean())
    return torch.stack(out)
