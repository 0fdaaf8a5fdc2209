"""What the performance of this framework is measured on.

A case is a dict of plain values; ``listed()`` gives the fixed ones and
``draw()`` more of the same ranges. Each stands for a call that a program
using the library makes again and again: a frame of the adaptive update with
its vertices for the renderer, a batch or a served tick of such frames, the
indexed export, the tree reduction with the compaction of a bitfield, and the
vertices of an unchanged mesh about another origin. The meshes and camera
paths are seeded stand-ins of the paper's scenes with the sizes of this
repository's configurations (a cube; a 100 x 100 height field; a cube-sphere
and a dodecahedron of Earth's size).
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2407_02215_gb300 import cbt as B

EARTH = 6.371e6
PRECISION = {"fp32": 0, "fixed": 1, "fp64": 2, "sphere": 3}


def listed():
    return [
        # One small prop or widget seen from changing sides: 24 halfedges, a few
        # thousand leaves, so the frame is launch and barrier latency.
        _frame("cube_orbit", "cube", D=16, max_depth=14, tau=4.0, path=64, at=8, span=16),
        # The main use: a terrain patch flown over, FP32, vertices for the renderer.
        _frame("grid_flythrough", "grid", n=100, D=20, max_depth=26, tau=2.0, path=120, at=36, span=24),
        # The same with a procedural relief added at every vertex (six octaves).
        _frame("terrain_relief", "grid", n=100, D=20, max_depth=26, tau=2.0, path=120, at=36, span=24, octaves=6),
        # A pool of eight million slots under a sub-pixel target: offline or
        # film-quality refinement, above what one block table of the small frames holds.
        _frame("grid_large_pool", "grid", n=100, D=23, max_depth=26, tau=0.7, path=120, at=48, span=16),
        # Landing on a planet with exact fixed-point vertices: millions of leaves.
        _frame("planet_fixed", "cubesphere", n=8, D=22, max_depth=48, tau=4.0, path=600, at=400, span=24,
               precision="fixed"),
        # The paper's planet: a projected dodecahedron in FP64, its points cached.
        _frame("dodeca_cached", "dodeca", D=17, max_depth=50, tau=14.0, path=300, at=120, span=24,
               precision="sphere", cache=True),
        # The paper's water planet (radial waves), without the optional cache.
        _frame("dodeca_waves", "dodeca", D=17, max_depth=50, tau=14.0, path=300, at=120, span=24,
               precision="sphere", octaves=4),
        # Many objects of a level updated at once: 64 meshes of 24 to 40,000 halfedges.
        {"name": "batch_64", "kind": "batch", "count": 64, "h_max": 40000, "tau": 4.0, "warm": 24, "span": 8},
        # A server's tick: four of sixteen resident objects, waited for.
        {"name": "serve_tick", "kind": "serve", "count": 16, "k": 4, "h_max": 12000, "tau": 4.0, "warm": 20,
         "span": 8},
        # A frame and its indexed triangulation for a visibility buffer.
        {**_frame("grid_indexed", "grid", n=100, D=20, max_depth=26, tau=2.0, path=120, at=36, span=24),
         "kind": "index"},
        # The tree reduction and compaction of a bitfield of 2^27 slots on their own.
        {"name": "reduce_compact", "kind": "reduce", "D": 27, "density": 0.5},
        # The vertices of a uniformly refined mesh about another origin (a second
        # view, a shadow pass): no update between.
        {"name": "second_view", "kind": "view", "n": 60, "depth": 6, "precision": "fp32"},
    ]


def draw(rng):
    kind = rng.choice(["frame"] * 6 + ["batch", "serve", "index", "reduce", "view"])
    tau = lambda lo, hi: round(_log_uniform(rng, lo, hi), 3)  # noqa: E731
    if kind == "reduce":
        return {"kind": "reduce", "D": rng.randint(18, 27), "density": round(rng.uniform(0.02, 0.98), 4)}
    if kind == "view":
        n, depth = int(_log_uniform(rng, 5, 61)), rng.randint(1, 6)
        return {"kind": "view", "n": n, "depth": depth, "precision": rng.choice(["fp32", "fp32", "fixed", "fp64"])}
    if kind in ("batch", "serve"):
        case = {"kind": kind, "count": rng.randint(8, 64), "h_max": int(_log_uniform(rng, 400, 40000)),
                "tau": tau(3.0, 8.0), "warm": rng.randint(12, 24), "span": 8}
        return {**case, "count": min(case["count"], 24), "k": rng.randint(1, 8)} if kind == "serve" else case
    scene = "grid" if kind == "index" else rng.choice(["cube", "grid", "grid", "grid", "cubesphere", "dodeca"])
    if scene == "cube":
        return _frame("", "cube", D=rng.randint(13, 18), max_depth=rng.randint(10, 20), tau=tau(2.0, 12.0), path=64,
                      at=rng.randint(0, 40), span=rng.randint(8, 20), named=False)
    if scene == "grid":
        n = int(_log_uniform(rng, 5, 130))
        D = min(22, max(rng.randint(14, 21), math.ceil(math.log2(4.2 * n * n)) + 2))
        case = _frame("", "grid", n=n, D=D, max_depth=rng.randint(16, 30), tau=tau(1.5, 8.0), path=120,
                      at=rng.randint(20, 80), span=rng.randint(8, 32), octaves=rng.choice([0, 0, 0, rng.randint(1, 8)]),
                      precision="fp32", named=False)
        if kind == "index":
            return {**case, "kind": "index", "octaves": 0, "D": min(D, 20)}
        return case
    if scene == "cubesphere":
        return _frame("", "cubesphere", n=rng.randint(2, 13), D=rng.randint(15, 21), max_depth=rng.randint(36, 48),
                      tau=tau(4.0, 14.0), path=600, at=rng.randint(200, 550), span=rng.randint(8, 32),
                      precision=rng.choice(["fixed", "fixed", "fp64"]), named=False)
    return _frame("", "dodeca", D=rng.randint(14, 19), max_depth=rng.randint(38, 50), tau=tau(8.0, 28.0), path=300,
                  at=rng.randint(60, 270), span=rng.randint(8, 32), precision="sphere",
                  cache=rng.random() < 0.5, octaves=rng.choice([0, 0, rng.randint(1, 6)]), named=False)


def prepare(case, seed):
    return {"frame": _prepare_frame, "index": _prepare_index, "batch": _prepare_batch, "serve": _prepare_serve,
            "reduce": _prepare_reduce, "view": _prepare_view}[case["kind"]](case, seed)


def run(state):
    return state.run(state)


def work(case):
    """The bytes a pass cannot do without (each input read once, each output
    written once) and its FP32/FP64 operations, from the leaf counts that the
    case's screen-space target gives (within the pool)."""
    kind = case["kind"]
    if kind == "reduce":
        bits = 1 << case["D"]
        return {"bytes": bits / 8 + 2 * bits / 8 + 4 * bits * case["density"], "flops": bits / 16}
    if kind == "view":
        leaves = 4 * case["n"] ** 2 << case["depth"]
        return {"bytes": leaves * (4 + 8 + 36.0), "flops": leaves * 54.0}
    if kind in ("batch", "serve"):
        each = [_leaves(scene, n, D, case["tau"]) for scene, n, D, _ in _population(case)]
        share = 1.0 if kind == "batch" else min(1.0, case["k"] / len(each))
        leaves, slots = share * sum(each), share * sum(2.0 ** D for _, _, D, _ in _population(case))
    else:
        leaves, slots = _leaves(case["scene"], case["n"], case["D"], case["tau"]), 2.0 ** case["D"]
    # per leaf: its heap ID and links in, its vertices out; the bitfield in and
    # out and the sum tree out
    nbytes = leaves * (8 + 16 + 36) + slots / 8 * 2 + slots / 4
    flops = leaves * 170.0 * (1 + case.get("octaves", 0))
    if kind == "index":
        nbytes += leaves * (36 + 16 + 6 + 12 + 8)
    return {"bytes": nbytes, "flops": flops}


def _leaves(scene, n, D, tau):
    roots = {"cube": 24, "grid": 4.2 * n * n, "cubesphere": 24 * n * n, "dodeca": 60}[scene]
    area = {"cube": 0.7e6, "grid": 3.7e6, "cubesphere": 37e6, "dodeca": 37e6}[scene]
    return min(0.95 * 2.0 ** D, roots + area / tau ** 2)


def exact(case, seed):
    """The second view's vertices in FP64: the uniform refinement has a closed
    form. The other cases' leaves follow from decisions taken frame after
    frame in the library's own FP32 arithmetic, which 64 bits do not give."""
    if case["kind"] != "view":
        return None
    mesh, origin = _view_inputs(case, seed)
    H, depth = mesh.H, case["depth"]
    root = np.arange(H)
    path = np.zeros(H, np.int64)  # bits of the path from the root, first split highest
    slot = np.arange(H)
    cap = 1 << _view_pool(H, depth)
    for _ in range(depth):
        # every leaf splits: leaves in slot order, each one's children together,
        # take the first free slots of the bitfield as it stands
        used = np.zeros(cap, bool)
        used[slot] = True
        order = np.argsort(slot)
        root, path = np.repeat(root[order], 2), np.repeat(path[order] * 2, 2)
        path[1::2] += 1
        slot = np.nonzero(~used)[0][:2 * H]
        H *= 2
    order = np.argsort(slot)
    root, path = root[order], path[order]
    v0, v1, c = _root_triangles(mesh)
    tri = np.stack([v0[root], v1[root], c[root]], 1)  # [N, 3, 3]
    for k in range(depth - 1, -1, -1):
        bit = (path >> k & 1).astype(bool)[:, None]
        mid = (tri[:, 0] + tri[:, 1]) * 0.5
        tri = np.stack([np.where(bit, tri[:, 2], tri[:, 0]), np.where(bit, tri[:, 1], tri[:, 2]), mid], 1)
    return torch.from_numpy(tri - np.asarray(origin))


# ------------------------------------------------------------------- frames

def _frame(name, scene, *, D, max_depth, tau, path, at, span, n=1, precision="fp32", octaves=0, cache=False,
           named=True):
    """One frame per pass: frames at .. at + span - 1 of a camera path of `path`
    frames, played back and forth, after the frames before them."""
    case = {"name": name} if named else {}
    return {**case, "kind": "frame", "scene": scene, "n": n, "D": D, "max_depth": max_depth, "tau": tau, "path": path,
            "at": at, "span": span, "precision": precision, "octaves": octaves, "cache": cache}


def _prepare_frame(case, seed):
    mesh, frames = _scene(case, seed)
    g = B.CBT(mesh, case["D"], case["max_depth"], point_cache=case["cache"])
    at, span = case["at"], case["span"]
    for fp in frames[:at]:
        g.update(fp)
    return SimpleNamespace(g=g, frames=frames[at:at + span], k=0, run=_run_frame,
                           rows=torch.zeros((1 << case["D"], 3, 3), dtype=torch.float32, device="cuda"),
                           live=torch.zeros(1, dtype=torch.int32, device="cuda"))


def _run_frame(s):
    s.g.update(_next(s), vertices_out=s.rows)
    s.g.live_count_async(s.live)
    return {"live": s.live, "vertices": s.rows}


def _prepare_index(case, seed):
    s = _prepare_frame(case, seed)
    cap = 1 << case["D"]
    s.run = _run_index
    s.workspace = s.g.index_workspace(cap)
    s.out = (torch.zeros((2 * cap, 3), dtype=torch.float32, device="cuda"),
             torch.zeros((cap, 3), dtype=torch.int32, device="cuda"),
             torch.zeros(cap, dtype=torch.int64, device="cuda"))
    return s


def _run_index(s):
    s.g.update(_next(s), vertices_out=s.rows)
    vertices, indices, _ = s.g.index(s.rows, workspace=s.workspace, out=s.out)
    return {"counts": [vertices.shape[0], indices.shape[0]], "vertices": s.out[0], "indices": s.out[1],
            "heap": s.out[2]}


def _next(s):
    """The next frame of a path played back and forth."""
    n = len(s.frames)
    cycle, pos = divmod(s.k, n)
    s.k += 1
    return s.frames[pos if cycle % 2 == 0 else n - 1 - pos]


# ------------------------------------------------------- batches and serving

def _population(case):
    """Scene, mesh size, pool and own seed of each instance: halfedge counts
    log-uniform (cubes below 100), pools of 2^14 to 2^20 slots or what the mesh needs."""
    rng = np.random.default_rng(case["count"])
    found = []
    for _ in range(case["count"]):
        H = math.exp(rng.uniform(math.log(24), math.log(case["h_max"])))
        n = max(1, round(math.sqrt(H / 4.2)))
        D = max(int(rng.integers(14, 21)), math.ceil(math.log2(6 * n * n)) + 2)
        found.append(("cube" if H < 100 else "grid", n, D, int(rng.integers(1 << 30))))
    return found


def _instances(case, seed):
    """The population's instances, the frames of each one's camera path, and
    one buffer for the vertices of all with each instance's part of it."""
    instances, paths = [], []
    for scene, n, D, own in _population(case):
        spec = {"scene": scene, "n": n, "tau": case["tau"], "path": 64, "precision": "fp32", "octaves": 0}
        mesh, path = _scene(spec, [seed, own], case["warm"] + case["span"])
        instances.append(B.CBT(mesh, D, 14 if scene == "cube" else 26))
        paths.append(path)
    at = np.cumsum([0] + [g.cap for g in instances])
    rows = torch.zeros((int(at[-1]), 3, 3), dtype=torch.float32, device="cuda")
    return instances, paths, rows, [rows[a:b] for a, b in zip(at[:-1], at[1:])]


def _prepare_batch(case, seed):
    instances, paths, rows, views = _instances(case, seed)
    batch = B.Batch(instances)
    warm, span = case["warm"], case["span"]
    for k in range(warm):
        batch.update([p[k] for p in paths])
    packed = [B.pack_frames([p[warm + k] for p in paths], "cuda", views) for k in range(span)]
    return SimpleNamespace(batch=batch, frames=packed, k=0, rows=rows, run=_run_batch)


def _run_batch(s):
    s.batch.update_packed(_next(s)[0])
    return {"vertices": s.rows}


def _prepare_serve(case, seed):
    instances, paths, rows, views = _instances(case, seed)
    server = B.Server(instances, inflight=2)
    k, warm = case["k"], case["warm"]
    for f in range(warm):
        for b, g in enumerate(instances):
            g.update(paths[b][f])
    torch.cuda.synchronize()
    return SimpleNamespace(server=server, paths=[p[warm:] for p in paths], views=views, rows=rows, tick=0, k=k,
                           run=_run_serve, stream=torch.cuda.Stream())


def _run_serve(s):
    n, span = len(s.paths), len(s.paths[0])
    ids = [(s.tick * s.k + i) % n for i in range(min(s.k, n))]
    f = s.tick * s.k // n % (2 * span)
    f = f if f < span else 2 * span - 1 - f
    s.tick += 1
    ticket = s.server.submit(ids, [s.paths[b][f] for b in ids], stream=s.stream,
                             vertices_out=[s.views[b] for b in ids])
    return {"live": s.server.poll(ticket, wait=True), "vertices": s.rows}


# ------------------------------------------- bitfields and unchanged meshes

def _prepare_reduce(case, seed):
    bits = 1 << case["D"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    words = torch.empty(bits // 32, dtype=torch.int32, device="cuda")
    weight = (1 << torch.arange(32, device="cuda", dtype=torch.int64))[None]
    step = 1 << 17
    for w in range(0, words.numel(), step):
        on = torch.rand((min(step, words.numel() - w), 32), device="cuda", generator=gen) < case["density"]
        words[w:w + step] = (on * weight).sum(1).to(torch.int32)
    return SimpleNamespace(words=words, D=case["D"], run=_run_reduce,
                           sums=torch.zeros(2 * words.numel(), dtype=torch.int32, device="cuda"),
                           live=torch.zeros(bits, dtype=torch.int32, device="cuda"))


def _run_reduce(s):
    B.sum_reduce(s.words, s.D, s.sums)
    B.compact(s.words, s.sums, s.D, s.live)
    return {"sums": s.sums[1:], "live": s.live}


def _view_pool(H, depth):
    """A pool in which the last level fits beside its parents: each split is
    charged for its partner's children too."""
    return math.ceil(math.log2(2.5 * (H << depth)))


def _view_inputs(case, seed):
    rng = np.random.default_rng(seed)
    return _grid_mesh(case["n"], 0.0, rng), rng.uniform(0.0, 1.0, 3) - [0.0, 0.0, 1.5]


def _prepare_view(case, seed):
    mesh, origin = _view_inputs(case, seed)
    D = _view_pool(mesh.H, case["depth"])
    g = B.CBT(mesh, D, case["depth"])
    grow = SimpleNamespace(eye=np.zeros(3), planes=np.zeros((5, 3), np.float32), nplanes=0, q=1.0, mode=1, seed=0,
                           precision=0, fixed_shift=20, gate=0)
    for _ in range(case["depth"]):
        g.update(grow)
    return SimpleNamespace(g=g, origin=origin, precision=PRECISION[case["precision"]], run=_run_view,
                           rows=torch.zeros((mesh.H << case["depth"], 3, 3), dtype=torch.float32, device="cuda"))


def _run_view(s):
    return s.g.vertices(s.origin, s.precision, 40 if s.precision == 1 else 20, out=s.rows)


# ----------------------------------------------------------- scenes (inputs)

def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _mesh(sizes, corners, pos):
    sizes = np.asarray(sizes, np.int32)
    return SimpleNamespace(face_sizes=sizes, face_verts=np.asarray(corners, np.int32).ravel(),
                           pos=np.ascontiguousarray(pos, np.float64), H=int(sizes.sum()))


def _root_triangles(mesh):
    """Per halfedge of an all-quad mesh its vertex, the next one's and the face's centroid."""
    quads = mesh.pos[mesh.face_verts.reshape(-1, 4)]  # [F, 4, 3]
    c = (((quads[:, 0] + quads[:, 1]) + quads[:, 2]) + quads[:, 3]) / 4.0
    return quads.reshape(-1, 3), np.roll(quads, -1, 1).reshape(-1, 3), np.repeat(c, 4, 0)


def _cube_mesh():
    p = np.array([[(i >> a & 1) - 0.5 for a in range(3)] for i in range(8)])
    return _mesh([4] * 6, [[0, 2, 3, 1], [4, 5, 7, 6], [0, 1, 5, 4], [2, 6, 7, 3], [0, 4, 6, 2], [1, 3, 7, 5]], p)


def _grid_mesh(n, tri_share, rng):
    """n x n cells of the unit square with normal heights; a share of the cells
    are two triangles."""
    a = (np.arange(n)[:, None] * (n + 1) + np.arange(n)[None, :]).ravel()
    b, c, d = a + 1, a + n + 2, a + n + 1
    X, Y = np.meshgrid(np.arange(n + 1) / n, np.arange(n + 1) / n, indexing="xy")
    pos = np.stack([X.ravel(), Y.ravel(), rng.normal(0.0, 0.05, X.size)], 1).astype(np.float32)
    split = rng.random(n * n) < tri_share
    turn = split & (rng.random(n * n) < 0.5)  # the other diagonal
    sizes = np.where(split[:, None], [3, 3], [4, 0])
    corners = np.where(split[:, None], np.where(turn[:, None], np.stack([a, b, d, b, c, d], 1),
                                                np.stack([a, b, c, a, c, d], 1)), np.stack([a, b, c, d, a, a], 1))
    used = np.arange(6) < sizes.sum(1)[:, None]
    return _mesh(sizes[sizes > 0], corners[used], pos)


def _cubesphere_mesh(n):
    index, pos, faces = {}, [], []

    def vertex(p):
        if p not in index:
            index[p] = len(pos)
            x = np.array(p) - n / 2.0
            pos.append(x / np.linalg.norm(x) * EARTH)
        return index[p]

    for axis in range(3):
        for side in (0, n):
            for i in range(n):
                for j in range(n):
                    corner = []
                    for du, dv in ((0, 0), (1, 0), (1, 1), (0, 1)):
                        p = [0, 0, 0]
                        p[axis], p[(axis + 1) % 3], p[(axis + 2) % 3] = side, i + du, j + dv
                        corner.append(vertex(tuple(p)))
                    faces.append(corner if side else corner[::-1])
    return _mesh([4] * len(faces), faces, np.array(pos))


def _dodeca_mesh():
    phi = (1.0 + 5.0 ** 0.5) / 2.0
    pos = [(x, y, z) for x in (-1, 1) for y in (-1, 1) for z in (-1, 1)]
    for s in (-1, 1):
        for t in (-1, 1):
            pos += [(0, s / phi, t * phi), (s / phi, t * phi, 0), (t * phi, 0, s / phi)]
    pos = np.array(pos, float) * (EARTH / 3.0 ** 0.5)
    faces = []
    for s in (-1, 1):
        for t in (-1, 1):
            for nrm in ((0, t * phi, s), (t * phi, s, 0), (s, 0, t * phi)):
                nrm = np.array(nrm) / np.linalg.norm(nrm)
                ring = np.argsort(-(pos @ nrm))[:5]
                mid = pos[ring].mean(0)
                e = (pos[ring[0]] - mid) / np.linalg.norm(pos[ring[0]] - mid)
                turn = np.arctan2((pos[ring] - mid) @ np.cross(nrm, e), (pos[ring] - mid) @ e)
                faces.append(ring[np.argsort(turn)])
    return _mesh([5] * 12, faces, pos)


def _look(eye, target, up, case):
    """A frame's parameters from a 1920 x 1080 camera with a 90 degree view."""
    cam = B.frame_from_camera(eye, target, up, math.pi / 2, 16 / 9, 1920, 1080, case["tau"])
    octaves = case["octaves"]
    sphere = case["scene"] == "dodeca"
    return SimpleNamespace(**cam, mode=0, seed=0, precision=PRECISION[case["precision"]], fixed_shift=20, gate=0,
                           sphere_radius=EARTH if sphere else 0.0,
                           disp_amplitude=(2.0 if sphere else 0.02) if octaves else 0.0,
                           disp_frequency=6371.0 if sphere else 4.0, disp_octaves=octaves, disp_seed=23)


def _scene(case, seed, count=None):
    """The mesh and the first `count` frames of the camera path (default: those
    up to the end of the measured span)."""
    rng = np.random.default_rng(seed)
    scene, total = case["scene"], case["path"]
    count = case["at"] + case["span"] if count is None else count
    up = np.array([0.0, 0.0, 1.0])
    frames = []
    if scene == "cube":
        mesh = _cube_mesh()
        for _ in range(count):  # from a new side each time
            eye = rng.normal(size=3)
            frames.append(_look(eye / np.linalg.norm(eye) * rng.uniform(1.5, 3.0), np.zeros(3), up, case))
    elif scene == "grid":
        mesh = _grid_mesh(case["n"], 0.1, rng)
        turns, phase = rng.uniform(0.6, 1.2, 2), rng.uniform(0.0, 1.0, 2)
        spot = lambda t: 0.5 + 0.4 * np.sin(2 * np.pi * (turns * t + phase))  # noqa: E731
        for k in range(count):  # down from 0.5 to 0.01 and up again, pitched 30 degrees down
            t = k / (total - 1)
            ahead = spot(t + 1e-3) - spot(t)
            ahead = ahead / np.linalg.norm(ahead) * math.cos(math.pi / 6)
            eye = np.array([*spot(t), 0.5 * 0.02 ** (1.0 - abs(2.0 * t - 1.0))])
            frames.append(_look(eye, eye + [*ahead, -0.5], up, case))
    else:  # a descent from 2e7 m to 2 m over a point of the surface
        if scene == "cubesphere":
            mesh = _cubesphere_mesh(case["n"])
            a, b, c = np.stack(_root_triangles(mesh), 1)[int(rng.integers(mesh.H))]
            target = rng.dirichlet(np.ones(3)) @ np.stack([a, b, c])
            nrm = np.cross(b - a, c - a)
            nrm *= np.sign(nrm @ target) / np.linalg.norm(nrm)
        else:
            mesh = _dodeca_mesh()
            face = mesh.pos[mesh.face_verts.reshape(-1, 5)[int(rng.integers(12))]]
            a, b = face[0], face[1]
            nrm = rng.dirichlet(np.ones(5)) @ face
            nrm /= np.linalg.norm(nrm)
            target = nrm * EARTH
        along = b - a
        along = along - nrm * (along @ nrm)
        along /= np.linalg.norm(along)
        for k in range(count):
            alt = 2e7 * 1e-7 ** (k / (total - 1))
            frames.append(_look(target + nrm * alt, target + along * (10.0 * alt), nrm, case))
    return mesh, frames
