"""The work a user of the framework has it do, as cases that can be timed.

A case is a dict of plain values; ``kind`` names the entry points it goes
through, the rest are sizes and options.  The sizes are those of the
framework's own configurations: a 36-triangle Cornell box, a 176k-triangle
room, a 2M-triangle building floor; six roughness levels; 16 to 256 samples
per point.  Geometry, radiance, materials and images are drawn from the seed.
"""
import math

import numpy as np
import torch

import paper_2304_05669_gb300 as F

SIGMA = {2: (0.1, 0.8), 4: (0.05, 0.25, 0.6, 1.0), 6: (0.02, 0.1, 0.25, 0.5, 0.75, 1.0),
         8: (0.02, 0.1, 0.2, 0.3, 0.45, 0.6, 0.8, 1.0)}
MOST_RAYS = 600_000_000          # of a drawn bake: well under the largest listed one


def listed():
    return [
        # the smallest scene and a small batch of points: latency, not throughput
        {"name": "bake_cornell", "kind": "bake", "scene": "cornell", "n": 4096, "spp_d": 64, "spp_s": 64, "K": 6,
         "voxel": 0, "sky": False},
        # the ordinary bake: one room's input views at the paper's diffuse sample count
        {"name": "bake_room", "kind": "bake", "scene": "room", "n": 1 << 20, "spp_d": 128, "spp_s": 128, "K": 6,
         "voxel": 0, "sky": False},
        # the largest: a building floor whose tree is larger than the L2
        {"name": "bake_floor", "kind": "bake", "scene": "floor4", "n": 1 << 21, "spp_d": 128, "spp_s": 128, "K": 6,
         "voxel": 0, "sky": False},
        # a ragged batch with the paper's voxel cache, light from outside and its 128 / 64 samples
        {"name": "bake_voxel_sky", "kind": "bake", "scene": "open_room", "n": 100_003, "spp_d": 128, "spp_s": 64,
         "K": 4, "voxel": 256, "sky": True},
        # stage 3: path-traced refinement through glossy surfaces with multiple importance sampling
        {"name": "refine_room", "kind": "refine", "scene": "room", "n": 131_072, "spp_d": 32, "spp_s": 32, "K": 6,
         "depth": 8, "mis": True},
        # a burst of bake and render requests to the serving loop, host buffers in and out
        {"name": "serve_burst", "kind": "serve", "bakes": 6, "renders": 4, "most_points": 60_000, "spp": 64,
         "most_rows": 65_536},
        # a scene's tree, built on the device for every new mesh
        {"name": "build_floor", "kind": "build", "scene": "floor4"},
        # the input views' first hits, compacted to query points
        {"name": "first_hits_room", "kind": "first_hits", "scene": "room", "views": 24, "w": 640, "h": 416},
        # one step of the BRDF optimisation over every pixel of the room's views
        {"name": "train_full", "kind": "train", "n": 24 * 640 * 416, "K": 6, "mask": True},
        # the same step on the paper's batch of 8192 pixels
        {"name": "train_batch", "kind": "train", "n": 8192, "K": 6, "mask": False},
        # per-triangle error of the floor's views, then emitter extraction at 100 points per triangle
        {"name": "emitters_floor", "kind": "emitters", "scene": "floor4", "views": 16, "w": 512, "h": 512,
         "per_tri": 100},
        # pooling the input pixels' radiance into the paper's 256^3 grid
        {"name": "pool_room", "kind": "pool", "scene": "room", "views": 16, "w": 512, "h": 512, "R": 256},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["bake", "bake", "bake", "refine", "serve", "build", "first_hits", "train", "train", "emitters",
                       "pool"])
    scene = rng.choice(["cornell", "room", "open_room", "floor1", "floor2", "floor4"])
    closed = rng.choice(["room", "floor1", "floor2", "floor4"])
    w, h = rng.randrange(64, 641), rng.randrange(48, 513)
    if kind == "bake":
        K = rng.choice([2, 4, 6, 6, 8])
        d = rng.choice([16, 64, 100, 128, 256])
        s = rng.choice([d, max(1, d // 2)])
        most = min(1 << 20, MOST_RAYS // (d + K * s))
        return {"kind": kind, "scene": scene, "n": _log_int(rng, 1000, most), "spp_d": d, "spp_s": s, "K": K,
                "voxel": rng.choice([0, 0, 64, 256]), "sky": rng.random() < 0.3}
    if kind == "refine":
        return {"kind": kind, "scene": scene, "n": _log_int(rng, 1000, 131_072), "spp_d": rng.choice([8, 16, 32]),
                "spp_s": rng.choice([8, 16, 32]), "K": rng.choice([4, 6]), "depth": rng.choice([4, 8]),
                "mis": rng.random() < 0.8}
    if kind == "serve":
        return {"kind": kind, "bakes": rng.randrange(1, 7), "renders": rng.randrange(1, 5),
                "most_points": _log_int(rng, 2000, 60_000), "spp": rng.choice([16, 64]),
                "most_rows": _log_int(rng, 8192, 65_536)}
    if kind == "build":
        return {"kind": kind, "scene": scene, "stretch": round(rng.uniform(0.5, 2.0), 3)}
    if kind == "first_hits":
        return {"kind": kind, "scene": closed, "views": rng.randrange(1, 25), "w": w, "h": h}
    if kind == "train":
        return {"kind": kind, "n": _log_int(rng, 1000, 24 * 640 * 416), "K": rng.choice([2, 4, 6, 8]),
                "mask": rng.random() < 0.5}
    if kind == "emitters":
        return {"kind": kind, "scene": closed, "views": rng.randrange(1, 17), "w": w, "h": h,
                "per_tri": rng.choice([64, 100])}
    return {"kind": kind, "scene": closed, "views": rng.randrange(1, 17), "w": w, "h": h,
            "R": rng.choice([64, 128, 256])}


# ---------------------------------------------------------------- meshes
def _sphere(level):
    p = (1 + 5 ** 0.5) / 2
    V = np.array([(-1, p, 0), (1, p, 0), (-1, -p, 0), (1, -p, 0), (0, -1, p), (0, 1, p), (0, -1, -p), (0, 1, -p),
                  (p, 0, -1), (p, 0, 1), (-p, 0, -1), (-p, 0, 1)], float)
    T = np.array([(0, 11, 5), (0, 5, 1), (0, 1, 7), (0, 7, 10), (0, 10, 11), (1, 5, 9), (5, 11, 4), (11, 10, 2),
                  (10, 7, 6), (7, 1, 8), (3, 9, 4), (3, 4, 2), (3, 2, 6), (3, 6, 8), (3, 8, 9), (4, 9, 5), (2, 4, 11),
                  (6, 2, 10), (8, 6, 7), (9, 8, 1)])
    for _ in range(level):
        e = np.sort(np.concatenate([T[:, [0, 1]], T[:, [1, 2]], T[:, [2, 0]]]), 1)
        u, at = np.unique(e, axis=0, return_inverse=True)
        ab, bc, ca = at.reshape(3, -1) + len(V)
        V = np.concatenate([V, V[u].sum(1)])
        a, b, c = T.T
        T = np.concatenate([np.stack(x, 1) for x in ((a, ab, ca), (b, bc, ab), (c, ca, bc), (ab, bc, ca))])
    return V / np.linalg.norm(V, axis=1, keepdims=True), T


class _Soup:
    def __init__(self):
        self.V, self.T, self.light, self.nv = [], [], [], 0

    def add(self, V, T, light=0.0):
        self.V.append(V)
        self.T.append(T + self.nv)
        self.light.append(np.full(len(T), light))
        self.nv += len(V)

    def sheet(self, at, du, dv, nu, nv, n, light=0.0):
        """An nu x nv grid of square cells whose faces look along n."""
        at, du, dv = (np.asarray(x, float) for x in (at, du, dv))
        s, t = np.meshgrid(np.arange(nu + 1) / nu, np.arange(nv + 1) / nv, indexing="ij")
        V = (at + s[..., None] * du + t[..., None] * dv).reshape(-1, 3)
        i = np.arange((nu + 1) * (nv + 1)).reshape(nu + 1, nv + 1)
        a, b, c, d = i[:-1, :-1].ravel(), i[1:, :-1].ravel(), i[1:, 1:].ravel(), i[:-1, 1:].ravel()
        T = np.concatenate([np.stack([a, b, c], 1), np.stack([a, c, d], 1)])
        self.add(V, T if np.dot(np.cross(du, dv), n) > 0 else T[:, ::-1], light)

    def walls(self, lo, hi, step, inward, open_front=False):
        """The six faces of a box, seen from inside (a room) or outside (furniture)."""
        lo, ex = np.asarray(lo, float), np.asarray(hi, float) - np.asarray(lo, float)
        for a in range(3):
            u, v = [k for k in range(3) if k != a]
            for side in (0, 1):
                if open_front and a == 2 and side == 0:
                    continue
                at, du, dv, n = lo.copy(), np.zeros(3), np.zeros(3), np.zeros(3)
                at[a] += side * ex[a]
                du[u], dv[v] = ex[u], ex[v]
                n[a] = (1 if side == 0 else -1) * (1 if inward else -1)
                cells = [max(1, round(ex[k] / step)) for k in (u, v)] if step else (1, 1)
                self.sheet(at, du, dv, *cells, n)


def _mesh(scene, rng, stretch=1.0):
    """V, F, Le, cache (numpy), the rooms' boxes and the balls (centre, radius)."""
    s, rooms, spheres = _Soup(), [], []
    if scene == "cornell":
        rooms = [((0, 0, 0), (1, 1, 1))]
        s.walls((0, 0, 0), (1, 1, 1), 1.0, True, open_front=True)
        s.walls((0.55, 0, 0.15), (0.85, 0.3, 0.45), 0, False)
        s.walls((0.15, 0, 0.5), (0.45, 0.6, 0.8), 0, False)
        s.sheet((0.35, 0.999, 0.35), (0.3, 0, 0), (0, 0, 0.3), 1, 1, (0, -1, 0), 1.0)
    else:
        floor = scene.startswith("floor")
        size, step, boxes, balls, level = ((5, 3, 6), 0.05, 80, 20, 5) if floor else ((4, 3, 6), 0.1, 60, 30, 4)
        U, T = _sphere(level)
        for r in range(int(scene[5:]) if floor else 1):
            lo = np.array([5.2 * r, 0.0, 0.0])
            hi = lo + size
            rooms.append((lo, hi))
            s.walls(lo, hi, step, True, open_front=scene == "open_room")
            for _ in range(boxes):
                e = rng.uniform(0.2, 1.2, 3)
                at = np.array([rng.uniform(lo[0] + 0.05, hi[0] - e[0] - 0.05), 0.0,
                               rng.uniform(lo[2] + 0.05, hi[2] - e[2] - 0.05)])
                s.walls(at, at + e, 0, False)
            for _ in range(balls):
                k = rng.uniform(0.1, 0.4)
                at = rng.uniform(lo + k, hi - k)
                s.add(at + k * U, T)
                spheres.append((*at, k))
            for _ in range(3):
                e = rng.uniform(0.5, 1.2, 2)
                at = (rng.uniform(lo[0] + 0.1, hi[0] - e[0] - 0.1), hi[1] - 0.01,
                      rng.uniform(lo[2] + 0.1, hi[2] - e[1] - 0.1))
                s.sheet(at, (e[0], 0, 0), (0, 0, e[1]), 1, 1, (0, -1, 0), math.exp(rng.uniform(math.log(5), math.log(50))))
    V = (np.concatenate(s.V) * (stretch, 1.0, 1.0)).astype(np.float32)
    T = np.ascontiguousarray(np.concatenate(s.T), np.int32)
    light = np.concatenate(s.light)[:, None]
    Le = light * (np.array([17.0, 12.0, 4.0]) if scene == "cornell" else np.ones(3))
    cache = np.full((len(T), 3), 0.5) if scene == "cornell" else rng.uniform(0, 1, (len(T), 3))
    cache = np.where(light > 0, 0.0, cache)
    return {"V": V, "F": T, "Le": Le.astype(np.float32), "cache": cache.astype(np.float32), "rooms": rooms,
            "balls": np.array(spheres).reshape(-1, 4)}


def _views(m, count, rng):
    """Pinhole cameras at eye height in the rooms in turn, clear of the balls, looking about level."""
    c = np.zeros((count, 10))
    for v in range(count):
        lo, hi = (np.asarray(x, float) for x in m["rooms"][v % len(m["rooms"])])
        while True:
            eye = lo + (hi - lo) * (rng.uniform(0.1, 0.9), rng.uniform(0.42, 0.6), rng.uniform(0.1, 0.9))
            if (np.linalg.norm(m["balls"][:, :3] - eye, axis=1) > m["balls"][:, 3] + 0.05).all():
                break
        c[v, 0:3] = eye
        yaw, pitch = rng.uniform(0, 2 * np.pi), np.deg2rad(rng.uniform(-20, 20))
        c[v, 3:6] = np.cos(pitch) * np.sin(yaw), np.sin(pitch), np.cos(pitch) * np.cos(yaw)
        c[v, 7], c[v, 9] = 1.0, np.deg2rad(60.0)
    return _cuda(c.astype(np.float32))


def _surface_points(m, n, rng):
    """Area-uniform points with cosine-weighted viewing directions (x, n, wo, tri)."""
    P = m["V"].astype(float)[m["F"]]
    cr = np.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
    area = np.linalg.norm(cr, axis=1)
    t = rng.choice(len(P), n, p=area / area.sum())
    r, w = np.sqrt(rng.random(n)), rng.random(n)
    x = (1 - r)[:, None] * P[t, 0] + (r * (1 - w))[:, None] * P[t, 1] + (r * w)[:, None] * P[t, 2]
    nn = (cr / area[:, None])[t]
    d = rng.normal(size=(n, 3))
    wo = nn + 0.95 * d / np.linalg.norm(d, axis=1, keepdims=True)
    wo /= np.linalg.norm(wo, axis=1, keepdims=True)
    return [_cuda(a.astype(np.float32)) for a in (x, nn, wo)] + [_cuda(t.astype(np.int32))]


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _scene(m):
    return F.Scene(*(_cuda(m[k]) for k in ("V", "F", "Le", "cache")))


def _queries(m, scene, name, n, rng):
    """n query points: surface points in the Cornell box, first hits of views elsewhere."""
    if name == "cornell":
        return F.pack_queries(*_surface_points(m, n, rng))
    count = 16 if name.startswith("floor") else 24
    k = math.sqrt(1.5 * n / (count * 320 * 208)) if name == "open_room" else math.sqrt(1.05 * n / (count * 320 * 208))
    w, h = int(320 * k) + 2, int(208 * k) + 2
    q, valid = scene.camera_queries(_views(m, count, rng), w, h)
    out, _, found = F.compact_queries(q, valid, n)
    return out[:int(found)]


def _tables(n, K, gen):
    base = torch.exp(torch.empty(n, 1, 3, device="cuda").uniform_(math.log(0.05), math.log(5.0), generator=gen))
    ramp = torch.linspace(1.0, 0.4, K, device="cuda")[None, :, None]
    u = lambda lo, hi, *s: torch.empty(*s, device="cuda").uniform_(lo, hi, generator=gen)  # noqa: E731
    return (base[:, 0] * u(0.5, 1.5, n, 3)).contiguous(), base * ramp * u(0.8, 1.2, n, K, 3), 0.1 * base * ramp * u(0.8, 1.2, n, K, 3)


def _materials(n, gen):
    u = lambda lo, *s: torch.empty(*s, device="cuda").uniform_(lo, 1.0, generator=gen)  # noqa: E731
    return u(0.0, n, 3), u(0.02, n), u(0.0, n)


def _target(tables, K, gen):
    """An image of other materials on the same tables, as a captured view gives it."""
    Ld, Ls0, Ls1 = tables
    a, r, m = _materials(Ld.shape[0], gen)
    k = (r * (K - 1)).long()[:, None, None].expand(-1, 1, 3)
    m = m[:, None]
    return a * (1 - m) * Ld + (0.04 * (1 - m) + a * m) * Ls0.gather(1, k)[:, 0] + Ls1.gather(1, k)[:, 0]


# ---------------------------------------------------------------- the cases' inputs
def prepare(case, seed):
    kind, rng = case["kind"], np.random.default_rng(seed)
    gen = torch.Generator("cuda").manual_seed(seed)
    s = {"case": case, "seed": seed}
    if kind == "train":
        s["sigma"], s["tables"] = SIGMA[case["K"]], _tables(case["n"], case["K"], gen)
        s["mat"] = tuple(x.requires_grad_() for x in _materials(case["n"], gen))
        s["Lgt"] = _target(s["tables"], case["K"], gen)
        s["mask"] = (torch.rand(case["n"], device="cuda", generator=gen) > 0.03).to(torch.uint8) if case["mask"] else None
        return s
    if kind == "serve":
        s["server"] = srv = F.Server(512 << 20)
        meshes = {k: _mesh(k, rng) for k in ("cornell", "room")}
        scenes = {k: _scene(m) for k, m in meshes.items()}
        ids = {k: srv.add_scene(x) for k, x in scenes.items()}
        s["jobs"] = []
        for j in range(case["bakes"]):
            k, n = ("room", "cornell")[j % 2], case["most_points"] // (1 + j)
            q = _queries(meshes[k], scenes[k], k, n, rng).cpu().pin_memory()
            s["jobs"].append(("bake", ids[k], q, (case["spp"], 16)[j % 3 == 2], j))
        s["tables"] = _tables(case["most_rows"], 6, gen)
        s["table"] = srv.add_table(*s["tables"], SIGMA[6])
        Lgt = _target(s["tables"], 6, gen)
        for j in range(case["renders"]):
            n = case["most_rows"] // (1 + j)
            ins = [x.cpu().pin_memory() for x in (*_materials(n, gen), Lgt[:n])]
            s["jobs"].append(("render", s["table"], ins, 0, j))
        torch.cuda.synchronize()
        return s
    s["mesh"] = m = _mesh(case["scene"], rng, case.get("stretch", 1.0))
    if kind == "build":
        s["arrays"] = [_cuda(m[k]) for k in ("V", "F", "Le", "cache")]
        return s
    s["scene"] = scene = _scene(m)
    if kind in ("first_hits", "emitters", "pool"):
        s["cams"] = _views(m, case["views"], rng)
        if kind == "first_hits":
            return s
        s["q"] = scene.camera_queries(s["cams"], case["w"], case["h"])[0]
        P = s["q"].shape[0]
        s["L"] = torch.exp(torch.randn(P, 3, device="cuda", generator=gen) - 1.0)
        if kind == "emitters":
            T = len(m["F"])
            light = _cuda((m["Le"] > 0).any(1))
            s["Lr"] = s["L"] * torch.empty(P, 3, device="cuda").uniform_(0.8, 1.2, generator=gen)
            # the mask field is near 1 on emitters and near 0 elsewhere
            s["alpha"] = (torch.rand(T, case["per_tri"], device="cuda", generator=gen) * 0.015 + 0.9 * light[:, None]).reshape(-1)
        return s
    s["sigma"] = SIGMA[case["K"]]
    s["q"] = _queries(m, scene, case["scene"], case["n"], rng)
    if kind == "refine":
        T = len(m["F"])
        scene.set_materials(*_materials(T, gen))
        return s
    if case["sky"]:
        scene.set_environment(torch.empty(256, 512, 3, device="cuda").uniform_(0.1, 3.0, generator=gen))
    if case["voxel"]:
        q, _ = scene.camera_queries(_views(m, 16, rng), 256, 256)
        L = torch.empty(q.shape[0], 3, device="cuda").uniform_(0.0, 1.0, generator=gen)
        scene.set_voxel_cache(scene.voxel_cache(q, L, case["voxel"]))
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "bake":
        return F.bake(s["scene"], s["q"], s["sigma"], c["spp_d"], c["spp_s"], seed=s["seed"])
    if kind == "refine":
        return F.bake_refine(s["scene"], s["q"], s["sigma"], c["spp_d"], c["spp_s"], max_depth=c["depth"], mis=c["mis"],
                             seed=s["seed"])
    if kind == "serve":
        srv = s["server"]
        tickets = [srv.submit_bake(to, x, SIGMA[6], spp, spp, seed=s["seed"], request_id=j) if what == "bake"
                   else srv.submit_render(to, 0, *x) for what, to, x, spp, j in s["jobs"]]
        out = []
        for t in tickets:
            if srv.wait(t) != 0:
                raise RuntimeError("a request failed")
            out.append(srv.result(t))
            srv.release(t)
        return out
    if kind == "build":
        return F.Scene(*s["arrays"]).export()
    if kind == "first_hits":
        q, valid = s["scene"].camera_queries(s["cams"], c["w"], c["h"])
        out, pixel, n = F.compact_queries(q, valid, (q.shape[0] + 1) // 2)
        # the triangle of a query record is an integer in a float column
        return q[:, :9], q[:, 9:].view(torch.int32), valid, out[:, :9], out[:, 9:].view(torch.int32), pixel, n
    if kind == "train":
        loss = F.factorized_render_loss(*s["mat"], s["tables"], s["Lgt"], s["sigma"], s["mask"])
        return (loss, *torch.autograd.grad(loss, s["mat"]))
    if kind == "emitters":
        T = s["scene"].T
        err, count = F.tri_error(s["q"], s["Lr"], s["L"], T)
        x = s["scene"].emitter_points(c["per_tri"], seed=s["seed"])
        flag, mean = F.emitter_classify(s["alpha"], c["per_tri"])
        return (err, count, x, flag, mean, *F.emitter_radiance(s["q"], s["L"], flag))
    return s["scene"].voxel_cache(s["q"], s["L"], c["R"])


def work(case):
    kind = case["kind"]
    tris = {"cornell": 36, "room": 176_000, "open_room": 171_000, "floor1": 511_000, "floor2": 1_023_000,
            "floor4": 2_045_000}.get(case.get("scene"), 0)
    scene = tris * 144                       # nodes, vertices and radiance, read once
    ray = 48 * math.log2(max(tris, 2)) + 80  # two boxes on each level of a balanced tree, one triangle
    pixels = case.get("views", 0) * case.get("w", 0) * case.get("h", 0)
    if kind in ("bake", "refine"):
        n, K = case["n"], case["K"]
        rays = n * (case["spp_d"] + K * case["spp_s"])
        return {"bytes": n * (52 + 24 * K) + scene, "flops": rays * ray * (2 if kind == "refine" else 1)}
    if kind == "serve":
        rows = sum(case["most_rows"] // (1 + j) for j in range(case["renders"]))
        bakes = [(case["most_points"] // (1 + j), (case["spp"], 16)[j % 3 == 2]) for j in range(case["bakes"])]
        return {"bytes": rows * 220 + sum(n for n, _ in bakes) * 196, "flops": sum(n * 7 * spp for n, spp in bakes) * 700}
    if kind == "build":
        return {"bytes": tris * (12 + 24 + 6 + 144 + 4), "flops": tris * 100}
    if kind == "first_hits":
        return {"bytes": pixels * (44 + 44 / 2) + scene, "flops": pixels * ray}
    if kind == "train":
        return {"bytes": case["n"] * (12 + 24 * case["K"] + 20 + 12 + 20 + (1 if case["mask"] else 0)), "flops": case["n"] * 300}
    if kind == "emitters":
        return {"bytes": pixels * (4 + 24 + 12) + tris * (12 + 16 * case["per_tri"] + 9 + 16), "flops": tris * case["per_tri"] * 150}
    return {"bytes": pixels * 24 + 16 * case["R"] ** 3, "flops": pixels * 30}


# ---------------------------------------------------------------- the same in 64 bits
def _philox(c0, c1, c2, c3, seed):
    """Words 0 and 1 of Philox4x32-10 on int64 tensors that hold 32-bit values."""
    lo, k0, k1 = 0xFFFFFFFF, seed & 0xFFFFFFFF, seed >> 32

    def mul(a, x):                             # a * x as (high, low) words, in 16-bit halves
        low = a * (x & 0xFFFF)
        high = a * (x >> 16) + (low >> 16)
        return high >> 16, ((high << 16) | (low & 0xFFFF)) & lo

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & lo, (k1 + 0xBB67AE85) & lo
    return c0, c1


def _exact_render(tables, sigma, mat, Lgt, mask):
    Ld, Ls0, Ls1, a, r, m, Lgt = (x.detach().double() for x in (*tables, *mat, Lgt))
    a, r, m = (x.requires_grad_() for x in (a, r, m))
    g = torch.tensor(sigma, dtype=torch.float32, device="cuda").double()
    rc = r.clamp(float(g[0]), float(g[-1]))
    i = (torch.searchsorted(g, rc.detach(), right=True) - 1).clamp(0, len(sigma) - 2)
    t = ((rc - g[i]) / (g[i + 1] - g[i]))[:, None]
    at = lambda L, k: L.gather(1, k[:, None, None].expand(-1, 1, 3))[:, 0]  # noqa: E731
    S0, S1 = ((1 - t) * at(L, i) + t * at(L, i + 1) for L in (Ls0, Ls1))
    mm = m[:, None]
    Lr = a * (1 - mm) * Ld + (0.04 * (1 - mm) + a * mm) * S0 + S1

    def tone(x):
        y = torch.log1p(x.clamp(min=0))
        return torch.where(y <= 0.0031308, 12.92 * y, 1.055 * y.clamp(min=0.0031308) ** (1 / 2.4) - 0.055)

    d = (tone(Lr) - tone(Lgt)) ** 2
    loss = (d if mask is None else d * mask[:, None]).sum()
    return Lr.detach(), loss.detach(), torch.autograd.grad(loss, (a, r, m))


def _exact_cornell(s):
    """The bake by testing every ray against every triangle."""
    c, m, seed = s["case"], s["mesh"], s["seed"]
    P = _cuda(m["V"]).double()[_cuda(m["F"]).long()]
    L_front, L_cache = _cuda(m["Le"]).double(), _cuda(m["cache"]).double()
    e1, e2 = P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]
    ng = torch.linalg.cross(e1, e2)
    eps = float(np.float32(1e-4) * np.float32((m["V"].max(0) - m["V"].min(0)).max()))
    q = s["q"]
    tri = q[:, 9:].view(torch.int32)[:, 0].long()
    unit = lambda v: v / v.norm(dim=-1, keepdim=True)  # noqa: E731
    x, n, wo = q[:, 0:3].double(), unit(q[:, 3:6].double()), unit(q[:, 6:9].double())
    o = x + eps * n
    # an orthonormal frame about n (Duff et al. 2017)
    sg = torch.where(n[:, 2] >= -1e-6, 1.0, -1.0).double()
    a = -1 / (sg + n[:, 2])
    b = n[:, 0] * n[:, 1] * a
    tx = torch.stack([1 + sg * n[:, 0] ** 2 * a, sg * b, -sg * n[:, 0]], 1)
    ty = torch.stack([b, sg + n[:, 1] ** 2 * a, -n[:, 1]], 1)
    mu_o = (n * wo).sum(1)
    N, K = len(x), c["K"]
    pid = torch.arange(N, device="cuda")
    out = [torch.zeros(N, 3, dtype=torch.float64, device="cuda")] + [torch.zeros(N, K, 3, dtype=torch.float64, device="cuda") for _ in "01"]

    def radiance(d):
        pv = torch.linalg.cross(d[:, None].expand(-1, len(P), 3), e2[None].expand(len(d), -1, 3))
        det = (e1 * pv).sum(-1)
        tv = o[:, None] - P[None, :, 0]
        u = (tv * pv).sum(-1) / det
        qv = torch.linalg.cross(tv, e1[None].expand(len(d), -1, 3))
        v = (d[:, None] * qv).sum(-1) / det
        t = (e2 * qv).sum(-1) / det
        ok = (det != 0) & (u >= 0) & (v >= 0) & (u + v <= 1) & (t > 0) & (torch.arange(len(P), device="cuda") != tri[:, None])
        best, hit = torch.where(ok, t, math.inf).min(1)
        front = (d * ng[hit]).sum(1) < 0
        return torch.where(torch.isfinite(best)[:, None], torch.where(front[:, None], L_front[hit], 0.0) + L_cache[hit], 0.0)

    for lobe in range(K + 1):
        S = c["spp_s"] if lobe else c["spp_d"]
        nx = max(k for k in range(1, S + 1) if S % k == 0 and k * k <= S)
        for k in range(S):
            z = torch.zeros_like(pid)
            w = _philox(pid, z + k, z + lobe, z, seed)
            u = []                             # the stratified uniforms are float32 by definition
            for r, cell, div in zip(w, (k % nx, k // nx), (nx, S // nx)):
                f = ((r >> 8).float() * 2.0 ** -24 + cell) / div
                u.append(f.clamp(max=1 - 2.0 ** -24).double())
            phi = 2 * math.pi * u[1]
            if lobe == 0:
                sn, cs = u[0].sqrt(), (1 - u[0]).sqrt()
                d = (sn * phi.cos())[:, None] * tx + (sn * phi.sin())[:, None] * ty + cs[:, None] * n
                out[0] += radiance(d) / S
                continue
            a2 = float(np.float32(s["sigma"][lobe - 1])) ** 4
            den = 1 - u[0] + a2 * u[0]
            ch, sh = ((1 - u[0]) / den).sqrt(), (a2 * u[0] / den).sqrt()
            hv = (sh * phi.cos())[:, None] * tx + (sh * phi.sin())[:, None] * ty + ch[:, None] * n
            oh = (wo * hv).sum(1)
            d = 2 * oh[:, None] * hv - wo
            mu_i = (n * d).sum(1)
            g1 = lambda y: 2 * y / (y + (a2 + (1 - a2) * y * y).sqrt())  # noqa: E731
            wt = torch.where((mu_i > 0) & (oh > 0) & (mu_o > 1e-2), g1(mu_i) * g1(mu_o) * oh / (mu_o * ch), 0.0)[:, None]
            F1 = ((1 - oh) ** 5)[:, None]
            L = radiance(d) / S
            zero = torch.zeros_like(L)
            out[1][:, lobe - 1] += torch.where(wt > 0, (1 - F1) * wt * L, zero)
            out[2][:, lobe - 1] += torch.where(wt > 0, F1 * wt * L, zero)
    return tuple(out)


def _exact_emitters(s):
    c, m = s["case"], s["mesh"]
    T, per = len(m["F"]), c["per_tri"]
    tri = s["q"][:, 9:].view(torch.int32)[:, 0].long()
    on = tri >= 0
    e = torch.zeros(T, dtype=torch.float64, device="cuda")
    e.index_add_(0, tri[on], ((s["Lr"].double() - s["L"].double()) ** 2).sum(1)[on])
    P = _cuda(m["V"]).double()[_cuda(m["F"]).long()]
    x = torch.empty(T, per, 3, dtype=torch.float64, device="cuda")
    for at in range(0, T, 1 << 17):
        t = torch.arange(at, min(T, at + (1 << 17)), device="cuda")[:, None].expand(-1, per)
        j = torch.arange(per, device="cuda")[None].expand(len(t), -1)
        u1, u2 = ((w >> 8).double() * 2.0 ** -24 for w in _philox(t, j, torch.full_like(t, 0x400), torch.zeros_like(t), s["seed"]))
        r = u1.sqrt()[..., None]
        w = u2[..., None]
        p = P[at:at + len(t), None]
        x[at:at + len(t)] = (1 - r) * p[:, :, 0] + r * (1 - w) * p[:, :, 1] + r * w * p[:, :, 2]
    mean = s["alpha"].double().reshape(T, per).mean(1)
    flag = mean > float(np.float32(0.01))
    keep = on & flag[tri.clamp(min=0)]
    t, rgb = tri[keep], s["L"][keep].double()
    n = torch.bincount(t, minlength=T)
    first = n.cumsum(0) - n
    Le = torch.zeros(T, 3, dtype=torch.float64, device="cuda")
    lit = (n > 0).nonzero()[:, 0]
    for k in range(3):
        v, i = rgb[:, k].sort(stable=True)
        v = v[t[i].sort(stable=True)[1]]
        Le[lit, k] = v[first[lit] + (n[lit] - 1) // 2]
    return e, None, x.reshape(-1, 3), None, mean, Le, None


def _exact_pool(s):
    R, V = s["case"]["R"], s["mesh"]["V"].astype(float)
    lo, hi = _cuda(V.min(0)), _cuda(V.max(0))
    i = ((s["q"][:, :3].double() - lo) * (R / (hi - lo))).floor().clamp(0, R - 1).long()
    cell = (i[:, 2] * R + i[:, 1]) * R + i[:, 0]
    g = torch.zeros(R ** 3, 4, dtype=torch.float64, device="cuda")
    g.index_add_(0, cell, torch.cat([s["L"].double(), torch.ones_like(s["L"][:, :1]).double()], 1))
    g[:, :3] /= g[:, 3:].clamp(min=1)
    return g.reshape(R, R, R, 4)


def exact(case, seed):
    kind = case["kind"]
    small = kind == "bake" and case["scene"] == "cornell" and not case["voxel"] and not case["sky"]
    if kind == "bake" and not (small and case["n"] * (case["spp_d"] + case["K"] * case["spp_s"]) < 4_000_000):
        return None                            # every ray against every triangle would take minutes
    if kind in ("refine", "build", "first_hits"):
        return None
    s = prepare(case, seed)
    if kind == "bake":
        return _exact_cornell(s)
    if kind == "train":
        _, loss, grads = _exact_render(s["tables"], s["sigma"], s["mat"], s["Lgt"], s["mask"])
        return (loss, *grads)
    if kind == "emitters":
        return _exact_emitters(s)
    if kind == "pool":
        return _exact_pool(s)
    out = []
    for what, _, x, _, _ in s["jobs"]:
        if what == "bake":
            out.append({"Ld": None, "Ls0": None, "Ls1": None})
            continue
        n = len(x[0])
        a, r, m, Lgt = (y.cuda() for y in x)
        Lr, loss, g = _exact_render([y[:n] for y in s["tables"]], SIGMA[6], (a, r, m), Lgt, None)
        out.append({"Lr": Lr, "loss": loss[None], "g_albedo": g[0], "g_rough": g[1], "g_metal": g[2]})
    s["server"].close()
    return out
