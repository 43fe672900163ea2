"""The work that a simulator has the renderer do, one case per kind and size of call.

A simulator keeps one renderer with one scene resident and asks it, step after
step, for the views of its agents from wherever they have walked to: the
handle (scene, work buffers, settings) is what a program keeps, so it is built
once per scene and settings here, and what differs from seed to seed is the
cameras, requests, maps or keys of a call. Scenes are multi-room floors (floor,
walls on a 4 m grid, furniture blobs) and a small uniform box, as octrees with
moment-matched interior nodes."""
import ctypes
import math
import types

import numpy as np
import torch

from paper_2603_15186_gb300 import Renderer, Server, _lib, camera_array

FLOOR1M, FLOOR4M = 1_000_000, 4_000_000
MIXED = ((320, 240), (640, 480), (640, 480), (1280, 720))   # one 1:2:1 round of resolutions


def listed():
    return [
        # one small view of a small scene, every leaf: the smallest render a program asks for
        views("view_box10k_128", "box", 10_000, "f32", 1, 128, 128, 0.0),
        # a short stretch of one agent's trajectory, view by view on the plain float32 path
        views("plain_floor1m_640x480", "floor", FLOOR1M, "f32", 4, 640, 480, 3.0, mode="plain"),
        # a few agents on a floor, float32, at an odd size
        views("views8_floor1m_333x187", "floor", FLOOR1M, "f32", 8, 333, 187, 4.0),
        # smooth transitions between levels, bfloat16 attributes
        views("blend16_floor1m_bf16", "floor", FLOOR1M, "bf16", 16, 640, 480, 4.0, blend=True),
        # one large view of a large scene: what a person looks at
        views("view_floor4m_720p", "floor", FLOOR4M, "f16", 1, 1280, 720, 3.0),
        # every agent of a large simulation in one call: mixed resolutions and granularities
        views("batch256_floor4m_mixed", "floor", FLOOR4M, "f16", 256, 0, 0, 5.0, tile=32, cta=16),
        # agents' requests arriving together at the serving loop
        {"name": "serve64_floor4m_mixed", "kind": "serve", "layout": "floor", "leaves": FLOOR4M,
         "dtype": "f16", "n": 64, "width": 0, "height": 0, "tau": 5.0, "tile": 32, "cta": 16},
        # the level-of-detail cuts of many agents, as lists of nodes
        {"name": "cut64_floor4m", "kind": "cut", "layout": "floor", "leaves": FLOOR4M,
         "dtype": "f16", "n": 64, "width": 0, "height": 0, "tau": 5.0},
        # one frustum-culled cut per group of consecutive poses (what a group needs resident)
        {"name": "shared_cut64_floor4m", "kind": "shared", "layout": "floor", "leaves": FLOOR4M,
         "dtype": "f16", "n": 64, "width": 0, "height": 0, "tau": 5.0, "group": 8, "guard": 0.0},
        # floor occupancy from horizontal slices over the robot's height, 5 cm cells
        {"name": "slice_floor4m_5cm", "kind": "slice", "layout": "floor", "leaves": FLOOR4M,
         "dtype": "f16", "cell": 0.05, "planes": 13},
        # distance fields to a building's landmarks and the agents' shortest paths
        {"name": "nav_528x276_9goals", "kind": "nav", "nx": 528, "ny": 276, "planes": 13,
         "goals": 9, "agents": 64, "inflate": 2},
        # sorting keyed data of a user's own, in place
        {"name": "sort_12m_u32", "kind": "sort", "n": 12_345_678, "key_bytes": 4, "bits": 32},
    ]


def views(name, layout, leaves, dtype, n, width, height, tau, mode="batched", blend=False,
          tile=16, cta=0):
    return {"name": name, "kind": "views", "layout": layout, "leaves": leaves, "dtype": dtype,
            "n": n, "width": width, "height": height, "tau": tau, "mode": mode, "blend": blend,
            "tile": tile, "cta": cta}


def draw(rng):
    kind = rng.choice(["views"] * 5 + ["serve", "cut", "shared", "slice", "nav", "sort"])

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "nav":
        return {"kind": kind, "nx": log(40, 900), "ny": log(40, 700), "planes": rng.randint(1, 16),
                "goals": rng.randint(1, 24), "agents": log(1, 400), "inflate": rng.randint(0, 6)}
    if kind == "sort":
        kb = rng.choice([4, 8])
        return {"kind": kind, "n": log(1_000, 16_000_000), "key_bytes": kb,
                "bits": rng.choice([8, 13, 16, 24, 32]) if kb == 4 else rng.choice([17, 32, 48, 64])}
    layout = rng.choice(["box", "floor", "floor", "floor"])
    leaves = log(1_000, 60_000) if layout == "box" else log(30_000, 1_500_000)
    case = {"kind": kind, "layout": layout, "leaves": leaves,
            "dtype": rng.choice(["f32", "f16", "bf16"])}
    if kind == "slice":
        return {**case, "cell": rng.choice([0.025, 0.04, 0.05, 0.1]), "planes": rng.randint(1, 24)}
    mixed = rng.random() < 0.4
    case.update(n=log(1, 64), width=0 if mixed else log(64, 1400),
                height=0 if mixed else log(48, 900), tau=rng.choice([0.0, rng.uniform(1.0, 12.0)]))
    if kind == "shared":
        return {**case, "group": rng.randint(1, 12), "guard": rng.choice([0.0, 16.0, 40.0])}
    if kind == "cut":
        return case
    tile = rng.choice([16, 16, 32])
    case.update(tile=tile, cta=16 if tile == 32 else 0)
    if kind == "views":
        mode = rng.choice(["batched"] * 4 + ["plain"])
        case.update(mode=mode, blend=rng.random() < 0.2)
        if mode == "plain":
            case["n"] = min(case["n"], 8)
    return case


# ---------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------

def floor_size(leaves):
    return (25.0, 12.0, 3.0) if leaves > 2_000_000 else (20.0, 15.0, 3.0)


def leaf_positions(rng, layout, n):
    if layout == "box":
        return rng.random((n, 3), dtype=np.float32) * np.float32([4.0, 4.0, 3.0])
    sx, sy, sz = floor_size(n)
    clusters, size = (160, 5000) if n > 2_000_000 else (40, 5000)
    n_furn = min(clusters * size, n // 2)
    segs = []          # (axis, coordinate, from, to) of the wall pieces around the doorways
    for axis, across, along in ((0, sx, sy), (1, sy, sx)):
        grid = np.arange(0.0, across + 1e-6, 4.0)
        cuts = np.append(np.arange(0.0, along, 4.0), along)
        for c in np.unique(np.append(grid, across)):
            for a, b in zip(cuts[:-1], cuts[1:]):
                half = 0.5 * min(1.0, 0.5 * (b - a))
                segs += [(axis, c, a, 0.5 * (a + b) - half), (axis, c, 0.5 * (a + b) + half, b)]
    segs = np.array([s for s in segs if s[3] > s[2]])
    length = segs[:, 3] - segs[:, 2]
    rest = n - n_furn
    n_wall = int(round(rest * length.sum() * sz / (length.sum() * sz + sx * sy)))
    n_floor = rest - n_wall
    ground = np.stack([rng.uniform(0, sx, n_floor), rng.uniform(0, sy, n_floor),
                       rng.normal(0.0, 0.01, n_floor)], 1)
    which = rng.choice(len(segs), size=n_wall, p=length / length.sum())
    on = segs[which, 2] + rng.random(n_wall) * length[which]
    off = segs[which, 1] + rng.normal(0.0, 0.01, n_wall)
    isx = segs[which, 0] == 0
    wall = np.stack([np.where(isx, off, on), np.where(isx, on, off), rng.uniform(0, sz, n_wall)], 1)
    k = max(1, n_furn // size)
    centre = np.stack([rng.uniform(0.6, sx - 0.6, k), rng.uniform(0.6, sy - 0.6, k),
                       np.full(k, 0.4)], 1)
    furn = centre[rng.integers(0, k, n_furn)] + rng.normal(0.0, 0.3, (n_furn, 3))
    furn[:, 2] = np.abs(furn[:, 2])
    return np.concatenate([ground, wall, furn]).astype(np.float32)


def morton(pos):
    lo = pos.min(0).astype(np.float64)
    side = float((pos.max(0) - lo).max()) * (1 + 1e-9) or 1.0
    g = np.clip((pos - lo) / side * (1 << 21), 0, (1 << 21) - 1).astype(np.uint64)
    for shift, mask in ((32, 0x1F00000000FFFF), (16, 0x1F0000FF0000FF), (8, 0x100F00F00F00F00F),
                        (4, 0x10C30C30C30C30C3), (2, 0x1249249249249249)):
        g = (g | (g << np.uint64(shift))) & np.uint64(mask)
    return (g[:, 0] << np.uint64(2)) | (g[:, 1] << np.uint64(1)) | g[:, 2]


def octree(codes):
    """Tree over leaves sorted by Morton code: cells of more than 8 leaves split
    into their non-empty octants, chains of single children collapse. Returns
    (depth, first leaf, number of leaves, is leaf) in breadth-first order (depth,
    then first leaf)."""
    n = len(codes)
    out = []

    def add(depth, lo, cnt, leaf):
        out.append((np.broadcast_to(depth, lo.shape), lo, cnt, np.full(lo.shape, leaf)))

    def leaves_of(depth, lo, cnt):
        at = np.repeat(lo - np.append(0, np.cumsum(cnt)[:-1]), cnt) + np.arange(cnt.sum())
        add(np.repeat(depth, cnt), at, np.ones_like(at), True)

    lo, cnt, depth = np.array([0]), np.array([n]), np.array([0])
    add(depth, lo, cnt, n == 1)
    if n <= 8:
        if n > 1:
            leaves_of(depth + 1, lo, cnt)
        lo = lo[:0]
    for level in range(21):
        if not len(lo):
            break
        cell = np.repeat(np.arange(len(lo)), cnt)
        at = np.repeat(lo - np.append(0, np.cumsum(cnt)[:-1]), cnt) + np.arange(len(cell))
        octant = (codes[at] >> np.uint64(3 * (20 - level))) & np.uint64(7)
        start = np.flatnonzero(np.append(True, (cell[1:] != cell[:-1]) | (octant[1:] != octant[:-1])))
        s_lo, s_cell, s_cnt = at[start], cell[start], np.diff(np.append(start, len(cell)))
        chain = np.bincount(s_cell, minlength=len(lo))[s_cell] == 1
        s_depth = depth[s_cell] + np.where(chain, 0, 1)
        one, some = ~chain & (s_cnt == 1), ~chain & (s_cnt > 1)
        add(s_depth[one], s_lo[one], s_cnt[one], True)
        add(s_depth[some], s_lo[some], s_cnt[some], False)
        small = some & (s_cnt <= 8)
        leaves_of(s_depth[small] + 1, s_lo[small], s_cnt[small])
        more = chain | (s_cnt > 8)
        lo, cnt, depth = s_lo[more], s_cnt[more], s_depth[more]
    if len(lo):        # coincident leaves at the finest level: one node holds them all
        leaves_of(depth + 1, lo, cnt)
    depth, lo, cnt, leaf = (np.concatenate(v) for v in zip(*out))
    order = np.lexsort((lo, depth))
    return depth[order], lo[order], cnt[order], leaf[order]


def rotations(q):
    q = q / np.linalg.norm(q, axis=1, keepdims=True)
    w, x, y, z = q.T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)],
                    1).reshape(-1, 3, 3)


def quaternions(R):
    """Unit quaternions (w, x, y, z) of rotation matrices, each from its largest component."""
    d0, d1, d2 = R[:, 0, 0], R[:, 1, 1], R[:, 2, 2]
    four = np.stack([1 + d0 + d1 + d2, 1 + d0 - d1 - d2, 1 - d0 + d1 - d2, 1 - d0 - d1 + d2], 1)
    a, b, c = R[:, 2, 1] - R[:, 1, 2], R[:, 0, 2] - R[:, 2, 0], R[:, 1, 0] - R[:, 0, 1]
    p, q, r = R[:, 0, 1] + R[:, 1, 0], R[:, 0, 2] + R[:, 2, 0], R[:, 1, 2] + R[:, 2, 1]
    rows = np.stack([np.stack([four[:, 0], a, b, c], 1), np.stack([a, four[:, 1], p, q], 1),
                     np.stack([b, p, four[:, 2], r], 1), np.stack([c, q, r, four[:, 3]], 1)], 1)
    v = rows[np.arange(len(R)), four.argmax(1)]
    return v / np.linalg.norm(v, axis=1, keepdims=True)


def make_scene(layout, n):
    """Leaves: log-scales ~ N(-3.5, 0.5), uniform rotations, opacity = sigmoid(N(0,
    1.5)), SH DC ~ N(0, 0.5), higher bands ~ N(0, 0.05). Interior nodes: opacity-
    weighted moments of their children; boxes: 3 sigma of a leaf, else the union."""
    rng = np.random.default_rng(n)
    lpos = leaf_positions(rng, layout, n)
    codes = morton(lpos)
    order = np.argsort(codes, kind="stable")
    depth, lo, cnt, leaf = octree(codes[order])
    m = len(depth)
    # a node's parent: the last node one level up that starts at or before it
    parent = np.full(m, -1, np.int64)
    begin = np.searchsorted(depth, np.arange(int(depth.max()) + 2))
    for d in range(1, int(depth.max()) + 1):
        up, me = slice(begin[d - 1], begin[d]), slice(begin[d], begin[d + 1])
        parent[me] = begin[d - 1] + np.searchsorted(lo[up], lo[me], side="right") - 1
    count = np.bincount(parent[1:], minlength=m).astype(np.int64)
    first = np.full(m, -1, np.int64)
    first[parent[1:][::-1]] = np.arange(1, m)[::-1]

    pos, quat = np.zeros((m, 3), np.float32), np.zeros((m, 4), np.float32)
    logs, opac = np.zeros((m, 3), np.float32), np.zeros(m, np.float32)
    sh = np.empty((m, 16, 3), np.float32)
    bmin, bmax = np.zeros((m, 3), np.float32), np.zeros((m, 3), np.float32)
    cov = np.zeros((m, 3, 3))
    pos[leaf] = lpos[order[lo[leaf]]]
    q = rng.standard_normal((n, 4), dtype=np.float32)
    quat[leaf] = q / np.linalg.norm(q, axis=1, keepdims=True)
    logs[leaf] = np.float32(0.5) * rng.standard_normal((n, 3), dtype=np.float32) - np.float32(3.5)
    opac[leaf] = 1 / (1 + np.exp(np.float32(-1.5) * rng.standard_normal(n, dtype=np.float32)))
    c = rng.standard_normal((n, 16, 3), dtype=np.float32) * np.float32(0.05)
    c[:, 0] *= 10
    sh[leaf] = c
    M = rotations(quat[leaf].astype(np.float64)) * np.exp(logs[leaf].astype(np.float64))[:, None, :]
    cov[leaf] = M @ M.transpose(0, 2, 1)
    sig = np.sqrt((M * M).sum(2))
    bmin[leaf], bmax[leaf] = pos[leaf] - 3 * sig, pos[leaf] + 3 * sig
    for d in range(int(depth.max()) - 1, -1, -1):
        at = begin[d] + np.flatnonzero(~leaf[begin[d]:begin[d + 1]])
        if not len(at):
            continue
        kids = np.arange(first[at[0]], first[at[-1]] + count[at[-1]])
        seg, own = first[at] - kids[0], np.repeat(np.arange(len(at)), count[at])
        w = opac[kids].astype(np.float64)
        total = np.add.reduceat(w, seg)
        share = w / total[own]
        mean = np.add.reduceat(share[:, None] * pos[kids], seg, axis=0)
        off = pos[kids] - mean[own]
        cov[at] = np.add.reduceat(share[:, None, None] *
                                  (cov[kids] + off[:, :, None] * off[:, None, :]), seg, axis=0)
        pos[at], opac[at] = mean, np.add.reduceat(share * w, seg)
        sh[at] = np.add.reduceat(share.astype(np.float32)[:, None, None] * sh[kids], seg, axis=0)
        bmin[at] = np.minimum.reduceat(bmin[kids], seg, axis=0)
        bmax[at] = np.maximum.reduceat(bmax[kids], seg, axis=0)
        val, vec = np.linalg.eigh(cov[at])
        vec[np.linalg.det(vec) < 0, :, 0] *= -1
        quat[at], logs[at] = quaternions(vec), 0.5 * np.log(np.maximum(val, 1e-12))
    i32 = np.int32
    return types.SimpleNamespace(
        pos=pos, quat=quat, log_scale=logs, opacity=opac, sh=sh, parent=parent.astype(i32),
        child_begin=first.astype(i32), child_count=count.astype(i32), aabb_min=bmin, aabb_max=bmax)


def stored_attributes(scene, dtype):
    if dtype == "f16":
        return {k: getattr(scene, k).astype(np.float16) for k in ("sh", "log_scale", "opacity")}
    if dtype == "bf16":
        got = {}
        for k in ("sh", "log_scale", "opacity"):
            b = getattr(scene, k).view(np.uint32)
            got[k] = ((b + ((b >> 16) & 1) + 0x7FFF) >> 16).astype(np.uint16)
        return got
    return None


_scene = {}     # the last scene built
_handle = {}    # the renderer (and its serving loop) that the program keeps


def scene_of(case):
    key = (case["layout"], case["leaves"])
    if key not in _scene:
        _scene.clear()
        _scene[key] = make_scene(*key)
    return _scene[key]


def release():
    for server, renderer in _handle.values():
        if server is not None:
            server.stop()
        renderer.close()
    _handle.clear()


def handle(case):
    """The renderer of the case's scene, set up as the case has it, and for a
    serving case the running serving loop over it."""
    serve = case["kind"] == "serve"
    key = (case["layout"], case["leaves"], case["dtype"], serve)
    if key not in _handle:
        release()
        scene = scene_of(case)
        large = case["leaves"] > 2_000_000
        renderer = Renderer(record_capacity=1 << (28 if large else 26),
                            pair_capacity=1 << (30 if large else 29))
        renderer.load_scene(scene, attr_dtype=case["dtype"],
                            stored=stored_attributes(scene, case["dtype"]))
        server = None
        if serve:
            renderer.set_tile(case["tile"], case["tile"])
            renderer.set_cta(case["cta"], case["cta"])
            server = Server(renderer, lanes=2, max_cams=64,
                            lane_record_capacity=1 << (27 if large else 26),
                            lane_pair_capacity=1 << 29)
        _handle[key] = (server, renderer)
    server, renderer = _handle[key]
    if case["kind"] == "views":
        renderer.set_mode(case["mode"])
        renderer.set_tile(case["tile"], case["tile"])
        renderer.set_cta(case["cta"], case["cta"])
        renderer.set_lod_blend(case["blend"])
    return server, renderer


# ---------------------------------------------------------------------------
# inputs of a call
# ---------------------------------------------------------------------------

def cameras(case, seed):
    """Views at 1.2 m from walks of 32 steps of 0.11 m that keep 0.3 m from the walls; in
    the box, views from near its middle. Resolutions and the order they come in belong
    to the case (a simulation's agents keep their cameras), poses and granularities to
    the seed (tau of the case +- 60 %)."""
    rng = np.random.default_rng(seed)
    n = case["n"]
    size = (4.0, 4.0) if case["layout"] == "box" else floor_size(case["leaves"])[:2]

    def free(p):
        return all(0.3 <= p[k] % 4.0 <= 3.7 and 0.3 <= p[k] <= size[k] - 0.3 for k in (0, 1))

    poses = []
    while len(poses) < n:
        if case["layout"] == "box":
            poses.append((rng.uniform(1.5, 2.5, 2), rng.uniform(-math.pi, math.pi)))
            continue
        p, heading = np.zeros(2), rng.uniform(-math.pi, math.pi)
        while not free(p):
            p = rng.uniform(0.0, size)
        for _ in range(32):
            for _ in range(64):
                h = heading + rng.normal(0.0, 0.14)
                q = p + 0.11 * np.array([math.cos(h), math.sin(h)])
                if free(q):
                    p, heading = q, h
                    break
                heading += rng.uniform(1.0, math.pi)
            poses.append((p, heading + rng.normal(0.0, 0.17)))
    out = []
    for i in range(n):
        w, h = (case["width"], case["height"]) if case["width"] else MIXED[i * 7 % 4]
        (x, y), a = poses[i]
        ca, sa = math.cos(a), math.sin(a)
        out.append(types.SimpleNamespace(
            pos=np.float32([x, y, 1.2]), width=w, height=h, cx=w / 2.0, cy=h / 2.0,
            R_wc=np.float32([[sa, -ca, 0.0], [0.0, 0.0, -1.0], [ca, sa, 0.0]]),
            fx=0.9375 * w, fy=0.9375 * w,
            tau=float(np.float32(case["tau"] * rng.uniform(0.4, 1.6)))))
    return out


def grid_of(case):
    size = (4.0, 4.0, 3.0) if case["layout"] == "box" else floor_size(case["leaves"])
    c = case["cell"]
    return types.SimpleNamespace(x0=-0.7, y0=-0.9, cell=c, nx=int((size[0] + 1.4) / c),
                                 ny=int((size[1] + 1.8) / c), z0=0.05, dz=0.1,
                                 nz=case["planes"], threshold=0.5)


def occupancy(case, seed):
    """A building's occupancy: walls every 80 cells with doorways, furniture, per plane."""
    rng = np.random.default_rng(seed)
    nx, ny, nz = case["nx"], case["ny"], case["planes"]
    j, i = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    wall = ((i % 80 < 2) & (np.abs(j % 80 - 40) > 10)) | ((j % 80 < 2) & (np.abs(i % 80 - 40) > 10))
    occ = np.broadcast_to(wall, (nz, ny, nx)).copy()
    for _ in range(1 + nx * ny // 3000):
        x, y, r, top = rng.uniform(0, nx), rng.uniform(0, ny), rng.uniform(1, 9), rng.integers(1, nz + 1)
        x0, x1, y0, y1 = (int(v) for v in (max(x - r, 0), x + r + 1, max(y - r, 0), y + r + 1))
        ys, xs = np.mgrid[y0:min(y1, ny), x0:min(x1, nx)]
        occ[:top, y0:y1, x0:x1] |= (xs - x) ** 2 + (ys - y) ** 2 <= r * r
    goals = np.stack([rng.integers(0, nx, case["goals"]), rng.integers(0, ny, case["goals"])], 1)
    for x, y in goals:     # a landmark stands free
        b = case["inflate"] + 4
        occ[:, max(y - b, 0):y + b + 1, max(x - b, 0):x + b + 1] = False
    starts = np.stack([rng.integers(0, nx, case["agents"]), rng.integers(0, ny, case["agents"]),
                       rng.integers(0, case["goals"], case["agents"])], 1)
    return occ.astype(np.uint8), goals.astype(np.int32), starts.astype(np.int32)


def images_of(cams):
    """One buffer for all images of a call, and each image's view of it."""
    flat = torch.zeros(sum(3 * c.width * c.height for c in cams), device="cuda")
    views_, at = [], 0
    for c in cams:
        k = 3 * c.width * c.height
        views_.append(flat[at:at + k].view(3, c.height, c.width))
        at += k
    return flat, views_


def prepare(case, seed):
    s = types.SimpleNamespace(case=case)
    kind = case["kind"]
    if kind in ("nav", "sort"):
        key = ("plain",)
        if key not in _handle:
            release()
            _handle[key] = (None, Renderer(record_capacity=1 << 22, pair_capacity=1 << 25))
        s.renderer = _handle[key][1]
    if kind == "nav":
        occ, s.goals, s.starts = occupancy(case, seed)
        s.occ = torch.from_numpy(occ).cuda()
    elif kind == "sort":
        g = torch.Generator(device="cuda").manual_seed(seed)
        n, wide = case["n"], case["key_bytes"] == 8
        s.fresh = torch.randint(-(1 << 63) if wide else -(1 << 31), (1 << 63) - 1 if wide else (1 << 31) - 1,
                                (n,), generator=g, device="cuda", dtype=torch.int64 if wide else torch.int32)
        s.index = torch.arange(n, device="cuda", dtype=torch.int32)
        s.keys, s.vals = torch.empty_like(s.fresh), torch.empty_like(s.index)
    else:
        s.server, s.renderer = handle(case)
        if kind == "slice":
            s.grid = grid_of(case)
            # the survey's origin shifts from scan to scan by up to a cell
            dx, dy, dz = np.random.default_rng(seed).uniform(0.0, 1.0, 3)
            s.grid.x0 += case["cell"] * dx
            s.grid.y0 += case["cell"] * dy
            s.grid.z0 += 0.05 * dz
        else:
            s.cams = cameras(case, seed)
        if kind in ("views", "serve"):
            s.flat, s.images = images_of(s.cams)
        if kind in ("cut", "shared"):
            # the program's own buffers, sized for the largest cut (every leaf, per list)
            step = case.get("group", 1)
            s.groups = np.int32(list(range(0, case["n"], step)) + [case["n"]])
            lists = len(s.groups) - 1
            s.ids = torch.zeros(lists * case["leaves"], dtype=torch.int32, device="cuda")
            s.offsets = torch.zeros(lists + 1, dtype=torch.int64, device="cuda")
    return s


def run(s):
    case, r = s.case, s.renderer
    kind = case["kind"]
    if kind == "views":
        r.render(s.cams, s.images)
        return s.flat
    if kind == "serve":
        for cam, image in zip(s.cams, s.images):
            s.server.submit(cam, image)
        s.server.wait_all()
        return s.flat
    if kind in ("cut", "shared"):
        # the library's C entry points, which write into the caller's buffers
        cams, n = camera_array(s.cams), case["n"]
        into = (ctypes.c_void_p(s.ids.data_ptr()), ctypes.c_void_p(s.offsets.data_ptr()), s.ids.numel(),
                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if kind == "cut":
            _lib.check(r.L.ngs_select_cut(r.h, cams, n, *into), "ngs_select_cut")
        else:
            _lib.check(r.L.ngs_select_cut_shared(
                r.h, cams, n, s.groups.ctypes.data_as(ctypes.c_void_p), len(s.groups) - 1,
                _lib.CUT_FRUSTUM, case["guard"], *into), "ngs_select_cut_shared")
        return s.ids, s.offsets
    if kind == "slice":
        return r.slice_occupancy(s.grid)
    if kind == "nav":
        top = min(case["planes"] - 1, 9)
        blocked, dist = r.nav_fields(s.occ, s.goals, min(1, top), top, case["inflate"])
        paths, lengths = r.nav_paths(dist, s.starts, 2048)
        return blocked, dist, paths, lengths
    # the keys come from the program's last step: sorted in place, new ones each time
    s.keys.copy_(s.fresh)
    s.vals.copy_(s.index)
    r.sort_pairs(s.keys, s.vals, 0, case["bits"])
    return s.keys, s.vals


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: the boxes of all nodes (the cut looks at each) once, the attributes of the
    Gaussians that a call draws or slices once, every output once. Operations: about 250
    blended Gaussians a pixel at 21 operations each, 20 a node and camera for a cut, 20 a
    cell a slice reaches."""
    kind = case["kind"]
    if kind == "sort":
        return {"bytes": 2 * case["n"] * (case["key_bytes"] + 4), "flops": 0}
    if kind == "nav":
        cells = case["nx"] * case["ny"]
        return {"bytes": cells * (min(case["planes"] - 1, 9) + 1 + 4 * case["goals"]) +
                case["agents"] * 2048 * 8, "flops": 0}
    nodes = 1.31 * case["leaves"]
    attr = 32 + (208 if case["dtype"] == "f32" else 104)
    if kind == "slice":
        g = grid_of(case)
        return {"bytes": case["leaves"] * (attr - (96 if case["dtype"] != "f32" else 192) + 4) +
                5 * g.nx * g.ny * g.nz, "flops": 300.0 * case["leaves"]}
    if kind in ("cut", "shared"):
        lists = case["n"] if kind == "cut" else -(-case["n"] // case["group"])
        kept = 0.7 if kind == "cut" else 0.2
        return {"bytes": 32 * nodes + 4 * kept * case["leaves"] * lists,
                "flops": 20.0 * nodes * case["n"]}
    pixels = sum(w * h for w, h in ((case["width"], case["height"]) if case["width"] else MIXED[i * 7 % 4]
                                    for i in range(case["n"])))
    drawn = min(1.0, 0.1 * case["n"]) * case["leaves"]
    return {"bytes": 32 * nodes + attr * drawn + 12 * pixels,
            "flops": 250.0 * 21 * pixels + 20.0 * nodes * case["n"]}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def exact(case, seed):
    kind = case["kind"]
    if kind in ("cut", "shared", "nav", "sort"):
        return None        # whole numbers
    if kind == "slice":
        g = prepare_grid(case, seed)
        return slice_exact(case, g), None
    pixels = work(case)["flops"] / 5250.0
    if pixels > 1.3e6:
        return None        # minutes rather than seconds
    scene = attributes64(case)
    return torch.cat([view_exact(scene, c, case.get("blend", False)).reshape(-1)
                      for c in cameras(case, seed)])


def prepare_grid(case, seed):
    g = grid_of(case)
    dx, dy, dz = np.random.default_rng(seed).uniform(0.0, 1.0, 3)
    g.x0 += case["cell"] * dx
    g.y0 += case["cell"] * dy
    g.z0 += 0.05 * dz
    return g


def attributes64(case):
    """The scene as stored (reduced types widened again), in 64 bits on the GPU."""
    scene = scene_of(case)
    got = {k: torch.from_numpy(getattr(scene, k)).cuda().double()
           for k in ("pos", "quat", "aabb_min", "aabb_max")}
    got["parent"] = torch.from_numpy(scene.parent).cuda().long()
    got["leaf"] = torch.from_numpy(scene.child_count).cuda() == 0
    stored = stored_attributes(scene, case["dtype"])
    for k in ("sh", "log_scale", "opacity"):
        a = getattr(scene, k) if stored is None else stored[k]
        if case["dtype"] == "bf16":
            a = (a.astype(np.uint32) << 16).view(np.float32)
        got[k] = torch.from_numpy(np.ascontiguousarray(a)).cuda()     # widened where used
    return types.SimpleNamespace(**got)


def axes64(quat, log_scale):
    """R diag(scale) of each Gaussian: its covariance is this times its transpose."""
    w, x, y, z = (quat / quat.norm(dim=1, keepdim=True)).unbind(1)
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1)
    return R.view(-1, 3, 3) * log_scale.double().exp()[:, None, :]


def sh_basis64(d):
    """Real spherical harmonics to degree 3 times (-1)^|m|, in the order l^2 + l + m."""
    x, y, z = d.unbind(1)
    pi = math.pi
    c1, c2 = math.sqrt(3 / (4 * pi)), math.sqrt(15 / (4 * pi))
    c3a, c3b, c3c = math.sqrt(35 / (32 * pi)), math.sqrt(105 / (4 * pi)), math.sqrt(21 / (32 * pi))
    return torch.stack([
        torch.full_like(x, math.sqrt(1 / (4 * pi))), -c1 * y, c1 * z, -c1 * x,
        c2 * x * y, -c2 * y * z, math.sqrt(5 / (16 * pi)) * (3 * z * z - 1), -c2 * x * z,
        c2 / 2 * (x * x - y * y), -c3a * y * (3 * x * x - y * y), c3b * x * y * z,
        -c3c * y * (5 * z * z - 1), math.sqrt(7 / (16 * pi)) * z * (5 * z * z - 3),
        -c3c * x * (5 * z * z - 1), c3b / 2 * z * (x * x - y * y), -c3a * x * (x * x - 3 * y * y)], 1)


def view_exact(sc, cam, blend):
    """One view: the cut at tau, the projection with its 0.3 dilation, SH colour, and every
    pixel blended front to back over the Gaussians whose alpha reaches 1/255."""
    dev = sc.pos.device
    eye = torch.from_numpy(cam.pos).to(dev).double()
    R = torch.from_numpy(cam.R_wc).to(dev).double()
    fx, fy, cx, cy = (float(np.float32(v)) for v in (cam.fx, cam.fy, cam.cx, cam.cy))
    gap = torch.clamp(torch.maximum(sc.aabb_min - eye, eye - sc.aabb_max), min=0).norm(dim=1)
    s = fx * (sc.aabb_max - sc.aabb_min).amax(1) / gap          # infinite inside the box
    above = s[sc.parent.clamp(min=0)]
    at = torch.nonzero((sc.leaf | (s <= cam.tau)) & ((sc.parent < 0) | (above > cam.tau)))[:, 0]
    mean, M, o, sh = sc.pos[at], axes64(sc.quat[at], sc.log_scale[at]), sc.opacity[at].double(), sc.sh[at]
    cov = M @ M.transpose(1, 2)
    if blend:
        up = sc.parent[at].clamp(min=0)
        sn, sp = s[at], above[at]
        v = 1 - ((sp - cam.tau) / (sp - sn)).clamp(0, 1)
        v = torch.where(torch.isfinite(sp) & (sp > sn) & (sc.parent[at] >= 0), v, torch.zeros_like(v))
        mean = mean + v[:, None] * (sc.pos[up] - mean)
        Mp = axes64(sc.quat[up], sc.log_scale[up])
        cov = cov + v[:, None, None] * (Mp @ Mp.transpose(1, 2) - cov)
        o = o + v * (sc.opacity[up].double() - o)
        sh = sh.double() + v[:, None, None] * (sc.sh[up].double() - sh.double())
    d = mean - eye
    t = d @ R.T
    keep = (t[:, 2] > 0.2) & (255 * o >= 1)
    d, t, cov, o, sh = d[keep], t[keep], cov[keep], o[keep], sh[keep]
    iz = 1 / t[:, 2]
    T = torch.stack([(fx * iz)[:, None] * R[0] - (fx * t[:, 0] * iz * iz)[:, None] * R[2],
                     (fy * iz)[:, None] * R[1] - (fy * t[:, 1] * iz * iz)[:, None] * R[2]], 1)
    c2 = T @ cov @ T.transpose(1, 2)
    a, b, c = c2[:, 0, 0] + 0.3, c2[:, 0, 1], c2[:, 1, 1] + 0.3
    det = a * c - b * b
    u, v = fx * t[:, 0] * iz + cx, fy * t[:, 1] * iz + cy
    K = 2 * torch.log(255 * o)
    hx, hy = (K * a).sqrt() + 1 / 64, (K * c).sqrt() + 1 / 64
    W, H = cam.width, cam.height
    keep = (u + hx >= 0) & (u - hx <= W) & (v + hy >= 0) & (v - hy <= H)
    order = torch.nonzero(keep)[:, 0]
    order = order[torch.sort(t[order, 2], stable=True)[1]]
    rgb = torch.einsum("nk,nkc->nc", sh_basis64(d[order] / d[order].norm(dim=1, keepdim=True)),
                       sh[order].double())
    rgb = (rgb + 0.5).clamp(min=0)
    u, v, a, b, c, det, o, hx, hy = (q[order] for q in (u, v, a, b, c, det, o, hx, hy))
    out = torch.zeros((3, H, W), dtype=torch.float64, device=dev)
    side = 64
    for y0 in range(0, H, side):
        band = torch.nonzero((v + hy >= y0) & (v - hy <= y0 + side))[:, 0]
        for x0 in range(0, W, side):
            mine = band[(u[band] + hx[band] >= x0) & (u[band] - hx[band] <= x0 + side)]
            ys, xs = torch.meshgrid(torch.arange(y0, min(y0 + side, H), device=dev) + 0.5,
                                    torch.arange(x0, min(x0 + side, W), device=dev) + 0.5, indexing="ij")
            X, Y = xs.reshape(-1).double(), ys.reshape(-1).double()
            left = torch.ones_like(X)
            colour = torch.zeros((3, len(X)), dtype=torch.float64, device=dev)
            for k in range(0, len(mine), 512):
                g = mine[k:k + 512]
                ex, ey = X[None] - u[g, None], Y[None] - v[g, None]
                e = (c[g, None] * ex * ex - 2 * b[g, None] * ex * ey + a[g, None] * ey * ey) / det[g, None]
                alpha = (o[g, None] * torch.exp(-0.5 * e)).clamp(max=0.99)
                alpha = torch.where(alpha >= 1 / 255, alpha, torch.zeros_like(alpha))
                after = left[None] * torch.cumprod(1 - alpha, 0)
                before = torch.cat([left[None], after[:-1]])
                colour += rgb[g].T @ (alpha * before * (after >= 1e-4))
                left = torch.where(after[-1] >= 1e-4, after[-1], torch.zeros_like(left))
                if not bool((left > 0).any()):
                    break
            out[:, y0:y0 + side, x0:x0 + side] = colour.view(3, *xs.shape)
    return out


def slice_exact(case, g):
    """The largest slice value of any leaf at each cell centre, from Sigma^-1 directly."""
    scene = scene_of(case)
    stored = stored_attributes(scene, case["dtype"]) or vars(scene)
    leaf = scene.child_count == 0

    def wide(k):
        a = stored[k][leaf]
        return (a.astype(np.uint32) << 16).view(np.float32) if case["dtype"] == "bf16" else a

    def put(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda().double()

    o = put(wide("opacity"))
    mean, M = put(scene.pos[leaf]), axes64(put(scene.quat[leaf]), put(wide("log_scale")))
    x0, y0, z0, cell, dz = (float(np.float32(v)) for v in (g.x0, g.y0, g.z0, g.cell, g.dz))
    keep = 255 * o >= 1
    o, mean, cov = o[keep], mean[keep], (M @ M.transpose(1, 2))[keep]
    inv = torch.linalg.inv(cov)
    K = 2 * torch.log(255 * o)
    out = torch.zeros((g.nz, g.ny * g.nx), dtype=torch.float64, device="cuda")
    for k in range(g.nz):
        z = z0 + k * dz
        near = torch.nonzero((z - mean[:, 2]) ** 2 <= K * cov[:, 2, 2] * 1.001)[:, 0]
        for part in near.split(1 << 19):
            m, P = mean[part], inv[part]
            half = (K[part, None] * cov[part][:, [0, 1], [0, 1]]).sqrt() + 1e-6
            first = torch.ceil((m[:, :2] - half - torch.tensor([x0, y0], device="cuda")) / cell - 0.5).long()
            last = torch.floor((m[:, :2] + half - torch.tensor([x0, y0], device="cuda")) / cell - 0.5).long()
            first = first.clamp(min=0)
            last = torch.minimum(last, torch.tensor([g.nx - 1, g.ny - 1], device="cuda"))
            span = (last - first + 1).clamp(min=0)
            cnt = span[:, 0] * span[:, 1]
            who = torch.repeat_interleave(torch.arange(len(part), device="cuda"), cnt)
            j = torch.arange(len(who), device="cuda") - (cnt.cumsum(0) - cnt)[who]
            cxs = first[who, 0] + j % span[who, 0]
            cys = first[who, 1] + j // span[who, 0]
            e = torch.stack([x0 + (cxs + 0.5) * cell - m[who, 0], y0 + (cys + 0.5) * cell - m[who, 1],
                             z - m[who, 2]], 1)
            q = torch.einsum("ni,nij,nj->n", e, P[who], e)
            value = (o[part][who] * torch.exp(-0.5 * q)).clamp(max=0.99)
            value = torch.where(value >= 1 / 255, value, torch.zeros_like(value))
            out[k].scatter_reduce_(0, cys * g.nx + cxs, value, "amax")
    return out.view(g.nz, g.ny, g.nx)
