"""The work that a user of this framework has it do, as cases to be timed.

Four kinds of call, all through the public entry points of the package:

* ``generate``  RICI images of oriented points of a scene (``rici_generate``);
* ``search``    ranks, true distances and top-1 of needle images in a haystack (``crss_search``);
* ``batch``     images and searches of many scenes in one call (``batch_run``);
* ``clutter``   the clutter measure around the points of an object (``clutter_areas``).

Scenes follow the repository's recipes: noise-displaced icospheres and tori, fitted to the unit
sphere, at random orientations in a box, the target first.  Mesh sizes are fixed by the case;
noise, orientations and positions come from the seed.
"""
import functools
import math

import numpy as np
import torch

import paper_2007_02306_gb300 as rici

DEV = "cuda"
BOX = 1.0  # centres are uniform in [-BOX, BOX]^3
MODES = {"default": rici.SEARCH_DEFAULT, "auto": rici.SEARCH_AUTO,
         "cuda_core": rici.SEARCH_CUDA_CORE}


def listed():
    clutter = dict(level=5, meshes=9, lo=5000, hi=50000)   # the clutter scene, about 190k triangles
    large = dict(level=7, meshes=40, lo=80000, hi=180000)  # the large scene, about 5M triangles
    return [
        # one small object, every vertex: the smallest call, where launches and latency count
        dict(name="generate_tiny", kind="generate", level=2, meshes=0, lo=0, hi=0, origins=0, N=32,
             R=0.3),
        # a few objects at a resolution and counts that are no multiple of anything
        dict(name="generate_ragged", kind="generate", level=3, meshes=3, lo=1501, hi=7019,
             origins=3001, N=33, R=0.2),
        # the clutter scene, every vertex: the haystack of one ordinary experiment
        dict(name="generate_clutter", kind="generate", origins=0, N=64, R=0.3, **clutter),
        # the large scene at the smallest and largest support radius: culling, then crossings
        dict(name="generate_large_narrow", kind="generate", origins=131072, N=64, R=0.15, **large),
        dict(name="generate_large_wide", kind="generate", origins=32768, N=64, R=0.6, **large),
        # many small scenes in one call, each with its own needles
        dict(name="batch_small_scenes", kind="batch", scenes=64, lo=2000, hi=12000, needles=64,
             N=64, R=0.3),
        # every image of one small object against each other, with all distances: the smallest
        # search
        dict(name="search_tiny", kind="search", images="scene", mode="default", level=2, meshes=0,
             lo=0, hi=0, Q=162, H=162, N=32, R=0.3, matrix=True),
        # a few query images looked up in the images of a clutter scene
        dict(name="search_query", kind="search", images="scene", mode="default", Q=100, H=90001,
             N=64, R=0.3, **clutter),
        # every target vertex of the clutter scene on the default form and on CUDA cores
        dict(name="search_cuda_core", kind="search", images="scene", mode="cuda_core", Q=10242,
             H=90000, N=64, R=0.3, **clutter),
        # a large scene's search: images with wide deltas are among the haystack's
        dict(name="search_large", kind="search", images="scene", mode="default", Q=8192, H=262144,
             N=64, R=0.3, **large),
        # images of many small objects with heavy-tailed deltas and sparse needles
        dict(name="search_sparse", kind="search", images="collection", mode="auto", Q=16384,
             H=262144, N=64, R=0.3),
        # the clutter measure around every vertex of the target of the clutter scene
        dict(name="clutter_measure", kind="clutter", origins=10242, R=0.3, **clutter),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["generate", "generate", "generate", "search", "search", "batch", "clutter"])
    if kind == "batch":
        lo = _log(rng, 1000, 4000)
        return dict(kind=kind, scenes=_log(rng, 8, 96), lo=lo, hi=lo * rng.randint(2, 6),
                    needles=_log(rng, 16, 256), N=rng.choice([32, 64]),
                    R=round(rng.uniform(0.15, 0.4), 3))
    meshes = rng.randint(0, 12)
    lo = _log(rng, 500, 20000)
    scene = dict(level=rng.randint(2, 6), meshes=meshes, lo=lo, hi=lo * rng.randint(2, 10))
    R = round(rng.uniform(0.15, 0.6), 3)
    if kind == "clutter":
        scene["meshes"] = max(3, meshes)
        return dict(kind=kind, origins=_log(rng, 100, 10242), R=min(R, 0.4), **scene)
    if kind == "generate":
        N = rng.choice([16, 32, 33, 48, 64, 64, 64, 100, 128])
        c = dict(kind=kind, N=N, R=R, **scene)
        per = _image_flops(_triangles(c), N, R)  # no more work than the largest listed case
        return dict(c, origins=_log(rng, 100, max(200, min(131072, int(8e11 / per)))))
    Q, H = _log(rng, 16, 16384), _log(rng, 1000, 262144)
    if rng.random() < 0.5:
        return dict(kind=kind, images="collection", mode=rng.choice(["default", "auto"]),
                    Q=min(Q, H), H=H, N=rng.choice([32, 64]), R=0.3)
    V, T = _vertices(scene), 10 * 4 ** scene["level"] + 2
    mode = rng.choice(["default", "default", "auto", "cuda_core"])
    H = min(H, V)
    return dict(kind=kind, images="scene", mode=mode, Q=min(Q, H, T), H=H,
                N=rng.choice([16, 32, 64, 64]), R=round(rng.uniform(0.15, 0.3), 3), **scene)


# ---------------------------------------------------------------- scenes


@functools.lru_cache(maxsize=None)
def _icosphere(level):
    """Unit vertices (float64) and outward faces of an icosahedron subdivided `level` times."""
    p = (1 + 5 ** 0.5) / 2
    v = torch.tensor([(-1, p, 0), (1, p, 0), (-1, -p, 0), (1, -p, 0), (0, -1, p), (0, 1, p),
                      (0, -1, -p), (0, 1, -p), (p, 0, -1), (p, 0, 1), (-p, 0, -1), (-p, 0, 1)],
                     dtype=torch.float64, device=DEV)
    v = v / v.norm(dim=1, keepdim=True)
    f = torch.tensor([(0, 11, 5), (0, 5, 1), (0, 1, 7), (0, 7, 10), (0, 10, 11), (1, 5, 9),
                      (5, 11, 4), (11, 10, 2), (10, 7, 6), (7, 1, 8), (3, 9, 4), (3, 4, 2),
                      (3, 2, 6), (3, 6, 8), (3, 8, 9), (4, 9, 5), (2, 4, 11), (6, 2, 10),
                      (8, 6, 7), (9, 8, 1)], device=DEV)
    for _ in range(level):
        n = v.shape[0]
        e = torch.cat([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]]).sort(dim=1).values
        key, inv = torch.unique(e[:, 0] * n + e[:, 1], return_inverse=True)
        mid = v[key // n] + v[key % n]
        v = torch.cat([v, mid / mid.norm(dim=1, keepdim=True)])
        ab, bc, ca = (inv + n).view(3, -1)
        a, b, c = f.unbind(1)
        f = torch.cat([torch.stack(t, 1) for t in
                       ((a, ab, ca), (b, bc, ab), (c, ca, bc), (ab, bc, ca))])
    return v, f


@functools.lru_cache(maxsize=None)
def _torus(want):
    """A torus of about `want` triangles: minor radius 0.35, rings in proportion."""
    m = 0.35
    nu = max(6, round(math.sqrt(want / 2 / m)))
    nv = max(3, round(want / 2 / nu))
    u = 2 * math.pi * torch.arange(nu, dtype=torch.float64, device=DEV)[:, None] / nu
    w = 2 * math.pi * torch.arange(nv, dtype=torch.float64, device=DEV)[None, :] / nv
    ring = 1 + m * torch.cos(w)
    v = torch.stack([ring * torch.cos(u), ring * torch.sin(u), m * torch.sin(w).expand(nu, nv)], -1)
    i = torch.arange(nu, device=DEV)[:, None]
    j = torch.arange(nv, device=DEV)[None, :]
    i1, j1 = (i + 1) % nu, (j + 1) % nv
    p00, p10, p11, p01 = i * nv + j, i1 * nv + j, i1 * nv + j1, i * nv + j1
    f = torch.cat([torch.stack([p00, p10, p11], -1).view(-1, 3),
                   torch.stack([p00, p11, p01], -1).view(-1, 3)])
    return v.reshape(-1, 3), f


def _parts(case):
    """The meshes of a scene: ("ico", level) or ("torus", triangles), the target first."""
    parts = [("ico", case["level"])]
    n = case["meshes"]
    for j in range(n):
        want = case["lo"] * (case["hi"] / case["lo"]) ** ((j + 0.5) / n)
        if j % 2:
            parts.append(("ico", max(1, min(7, round(math.log(want / 20, 4))))))
        else:
            parts.append(("torus", int(want)))
    return parts


def _part_sizes(part):
    """(vertices, triangles) of a mesh."""
    if part[0] == "ico":
        return 10 * 4 ** part[1] + 2, 20 * 4 ** part[1]
    nu = max(6, round(math.sqrt(part[1] / 2 / 0.35)))
    nv = max(3, round(part[1] / 2 / nu))
    return nu * nv, 2 * nu * nv


def _vertices(case):
    return sum(_part_sizes(p)[0] for p in _parts(case))


def _triangles(case):
    return sum(_part_sizes(p)[1] for p in _parts(case))


def _normals(v, f):
    """Area-weighted vertex normals; sums in fixed point, so that their order does not matter."""
    fn = torch.linalg.cross(v[f[:, 1]] - v[f[:, 0]], v[f[:, 2]] - v[f[:, 0]])
    q = (fn * (2.0 ** 50 / float(fn.abs().max()) / 1024)).round().to(torch.int64)
    n = torch.zeros(v.shape, dtype=torch.int64, device=DEV)
    for k in range(3):
        n.index_add_(0, f[:, k], q)
    n = n.to(torch.float64)
    return n / n.norm(dim=1, keepdim=True).clamp(min=1.0)


def _displaced(part, g):
    """A mesh with radial noise of 10 %, fitted to the unit sphere."""
    v, f = _icosphere(part[1]) if part[0] == "ico" else _torus(part[1])
    noise = torch.rand(v.shape[0], 1, generator=g, device=DEV, dtype=torch.float64) * 0.2 + 0.9
    v = v * noise
    v = v - 0.5 * (v.min(0).values + v.max(0).values)
    return v / v.norm(dim=1).max(), f


def _scene(parts, g):
    """One scene as the framework takes it: float32 vertices and normals, int32 triangles."""
    vs, ns, fs, nv = [], [], [], 0
    for part in parts:
        v, f = _displaced(part, g)
        q = torch.randn(4, generator=g, device=DEV, dtype=torch.float64)
        w, x, y, z = (q / q.norm()).tolist()
        rot = torch.tensor([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                            [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                            [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]],
                           dtype=torch.float64, device=DEV)
        v = (v[:, None, :] * rot[None]).sum(-1)
        v = v + (torch.rand(3, generator=g, device=DEV, dtype=torch.float64) * 2 - 1) * BOX
        vs.append(v)
        ns.append(_normals(v, f))
        fs.append(f + nv)
        nv += v.shape[0]
    return dict(vertices=torch.cat(vs).float().contiguous(),
                normals=torch.cat(ns).float().contiguous(),
                triangles=torch.cat(fs).int().contiguous())


def _origins(V, count):
    """`count` vertices in runs of up to 4,096 consecutive ones, spread over the scene (0: all)."""
    if count == 0 or count >= V:
        return torch.arange(V, dtype=torch.int32, device=DEV)
    i = torch.arange(count, device=DEV)
    run = min(4096, count)
    runs = -(-count // run)
    o = (i // run) * ((V - run) // max(1, runs - 1) if runs > 1 else 0) + i % run
    return o.clamp(max=V - 1).int()


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


# ---------------------------------------------------------------- images of a search


def _plateaus(img, image_share, row_share, heights, g):
    """Adds a height to a random range of columns in some rows of some images (in place)."""
    n, N, _ = img.shape
    pick = torch.rand(n, 1, generator=g, device=DEV) < image_share
    at = ((torch.rand(n, N, generator=g, device=DEV) < row_share) & pick).nonzero()
    c1 = torch.randint(0, N - 1, (at.shape[0], 1), generator=g, device=DEV)
    c2 = c1 + 1 + (torch.rand(c1.shape, generator=g, device=DEV) * (N - c1)).long()
    cols = torch.arange(N, device=DEV)[None]
    add = ((cols >= c1) & (cols < c2)) * heights(at.shape[0])[:, None]
    img[at[:, 0], at[:, 1]] = (img[at[:, 0], at[:, 1]].long() + add).clamp(0, 32767).short()


def _collection_images(case, g):
    """Images of many small objects: heavy-tailed plateaus in 2 % of them (heights with
    P(|v| = k) ~ k^-2 up to 300); needles are copies of distinct ones, taken before clutter raises
    rows of 30 % of the haystack by 2."""
    Q, H, N = case["Q"], case["H"], case["N"]
    v0, f0 = _icosphere(2)
    n = -(-H // v0.shape[0])
    v = v0[None] * (torch.rand(n, v0.shape[0], 1, generator=g, device=DEV, dtype=torch.float64) * 0.2 + 0.9)
    v = v / v.norm(dim=2, keepdim=True).amax(1, keepdim=True)
    k = torch.arange(n, device=DEV)
    f = (f0[None] + k[:, None, None] * v0.shape[0]).view(-1, 3)
    normals = _normals(v.view(-1, 3), f)
    # objects side by side, out of each other's reach
    side = math.ceil(n ** (1 / 3))
    v = v + 4.0 * torch.stack([k % side, k // side % side, k // side ** 2], 1).double()[:, None]
    img = rici.rici_generate(v.view(-1, 3).float().contiguous(), normals.float().contiguous(),
                             f.int().contiguous(),
                             torch.arange(H, dtype=torch.int32, device=DEV), case["R"], N)
    img = img.view(torch.int16)
    p = torch.arange(1, 301, dtype=torch.float64, device=DEV) ** -2.0

    def tail(m):
        mag = torch.multinomial(p, max(m, 1), replacement=True, generator=g)[:m] + 1
        return mag * (torch.randint(0, 2, (m,), generator=g, device=DEV) * 2 - 1)

    _plateaus(img, 0.02, 0.03, tail, g)
    match = torch.randperm(H, generator=g, device=DEV)[:Q]
    needles = img[match].clone()
    _plateaus(img, 0.3, 0.1, lambda m: torch.full((m,), 2, device=DEV), g)
    return needles.view(torch.uint16), img.view(torch.uint16), match


def _scene_images(case, g):
    """Needles: vertices of the target imaged alone; haystack: the same vertices, then others of
    the scene, imaged with everything in it."""
    Q, H = case["Q"], case["H"]
    sc = _scene(_parts(case), g)
    nv, nt = _part_sizes(("ico", case["level"]))
    need = torch.randperm(nv, generator=g, device=DEV)[:Q].sort().values.int()
    left = torch.ones(sc["vertices"].shape[0], dtype=torch.bool, device=DEV)
    left[need.long()] = False
    rest = left.nonzero()[:, 0]
    hay = torch.cat([need, rest[_origins(rest.numel(), H - Q).long()].int() if H > Q else need[:0]])
    args = sc["vertices"], sc["normals"]
    needles = rici.rici_generate(*args, sc["triangles"][:nt].contiguous(), need, case["R"], case["N"])
    images = rici.rici_generate(*args, sc["triangles"], hay.contiguous(), case["R"], case["N"])
    return needles, images, torch.arange(Q, device=DEV)


# ---------------------------------------------------------------- the cases


def prepare(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    if kind == "search":
        make = _collection_images if case["images"] == "collection" else _scene_images
        needles, haystack, match = make(case, g)
        return dict(case=case, needles=needles, haystack=haystack, true_match=match)
    if kind == "batch":
        return dict(case=case, **_batch(case, g))
    sc = _scene(_parts(case), g)
    V = sc["vertices"].shape[0]
    o = _origins(V if kind == "generate" else _part_sizes(("ico", case["level"]))[0], case["origins"])
    return dict(case=case, origins=o, **sc)


def _batch_parts(case):
    """Scene s: a target icosphere and a torus whose size goes through the range."""
    n = case["scenes"]
    out = []
    for s in range(n):
        want = case["lo"] * (case["hi"] / case["lo"]) ** ((s * 7 % n + 0.5) / n)
        out.append([("ico", 3), ("torus", max(64, int(want) - 1280))])
    return out


def _batch(case, g):
    """Scenes and, as a caller that keeps its buffers has them, the outputs of all scenes in a row."""
    N, scenes = case["N"], []
    Q, H = [], []
    for parts in _batch_parts(case):
        sc = _scene(parts, g)
        V = sc["vertices"].shape[0]
        nv, nt = _part_sizes(parts[0])
        need = torch.randperm(nv, generator=g, device=DEV)[:case["needles"]].sort().values
        scenes.append(dict(sc, needle_origins=need.int(), target_triangles=nt, true_match=need,
                           haystack_origins=torch.arange(V, dtype=torch.int32, device=DEV)))
        Q.append(need.numel())
        H.append(V)
    flat = dict(needle_images=torch.empty(sum(Q), N, N, dtype=torch.uint16, device=DEV),
                haystack_images=torch.empty(sum(H), N, N, dtype=torch.uint16, device=DEV),
                rank=torch.empty(sum(Q), dtype=torch.int32, device=DEV),
                true_distance=torch.empty(sum(Q), dtype=torch.int64, device=DEV),
                top1=torch.empty(sum(Q), dtype=torch.int32, device=DEV))
    split = {k: t.split(H if k == "haystack_images" else Q) for k, t in flat.items()}
    return dict(scenes=scenes, flat=flat,
                outputs=[{k: t[s] for k, t in split.items()} for s in range(len(Q))])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "search":
        return rici.crss_search(state["needles"], state["haystack"], state["true_match"],
                                mode=MODES[case["mode"]],
                                return_distances=case.get("matrix", False))
    if kind == "batch":
        rici.batch_run(state["scenes"], case["R"], case["N"], outputs=state["outputs"])
        return {k: t.view(torch.int16) if t.dtype == torch.uint16 else t
                for k, t in state["flat"].items()}
    args = state["vertices"], state["normals"], state["triangles"], state["origins"], case["R"]
    if kind == "clutter":
        return rici.clutter_areas(*args, _part_sizes(("ico", case["level"]))[0], with_clutter=True)
    return rici.rici_generate(*args, case["N"]).view(torch.int16)


def _image_flops(triangles, N, R):
    """Operations of one image by the method's formulas: 15 for each of a triangle's vertices and
    46 for each layer that a triangle crosses within the largest circle.  How many of a scene's
    triangles and layers those are was counted on images of the large scene: 147,686 triangles and
    575,424 layers of 5.02M at N = 64, R = 0.6, and 23,937 and 154,909 at R = 0.3."""
    pairs = 0.0294 * triangles * (R / 0.6) ** 2.6
    return 45 * pairs + 46 * pairs * 3.9 * (N / 64) * (0.6 / R) ** 0.7


def work(case):
    kind = case["kind"]
    if kind == "search":
        Q, H, px = case["Q"], case["H"], case["N"] ** 2
        # the expanded distance is two products over all pixels; where pairs may stop early
        # (sparse needles, CUDA cores), a word of four pixels or a few rows decide
        per = {"default": 4 * px, "auto": 16, "cuda_core": 4 * px // 5}[case["mode"]]
        out = 16 * Q + (8 * Q * H if case.get("matrix") else 0)
        return dict(bytes=2 * px * (Q + H) + 8 * Q + out, flops=float(per) * Q * H)
    if kind == "batch":
        b = f = 0.0
        px = case["N"] ** 2
        for parts in _batch_parts(case):
            (tv, tt), (cv, ct) = (_part_sizes(p) for p in parts)
            q, h = min(case["needles"], tv), tv + cv
            b += 24 * h + 12 * (tt + ct) + 2 * px * (q + h) + 4 * h + 28 * q
            f += _image_flops(tt + ct, case["N"], case["R"]) * h + 4 * px * q * h
        return dict(bytes=b, flops=f)
    V, T = _vertices(case), _triangles(case)
    n = case["origins"]
    n = min(n or V, V if kind == "generate" else 10 * 4 ** case["level"] + 2)
    if kind == "clutter":
        pairs = 0.0294 * T * (case["R"] / 0.6) ** 2.6
        return dict(bytes=24 * V + 12 * T + 28 * n, flops=60.0 * pairs * n)
    return dict(bytes=24 * V + 12 * T + 4 * n + 2 * n * case["N"] ** 2,
                flops=_image_flops(T, case["N"], case["R"]) * n)


# ---------------------------------------------------------------- 64-bit values


def exact(case, seed):
    kind = case["kind"]
    if kind == "search":
        if float(case["Q"]) * case["H"] * case["N"] ** 2 > 2e11:
            return None
        return _exact_search(prepare(case, seed))
    if kind == "clutter":
        n = min(case["origins"], 10 * 4 ** case["level"] + 2)
        return _exact_clutter(prepare(case, seed)) if float(n) * _triangles(case) < 1e10 else None
    return None  # crossing counts are whole numbers


def _exact_search(st):
    def deltas(img):
        x = (img.view(torch.int16).long() & 0xFFFF).double()
        return (x[:, :, 1:] - x[:, :, :-1]).flatten(1)

    a = deltas(st["needles"])
    m, match = (a != 0).double(), st["true_match"]
    H, step = st["haystack"].shape[0], 8192
    d = torch.cat([(m @ (b * b).T) - 2 * (a @ b.T) for b in
                   (deltas(st["haystack"][s:s + step]) for s in range(0, H, step))], 1)
    d += (a * a).sum(1, keepdim=True)
    true = d.gather(1, match[:, None])
    j = torch.arange(H, device=DEV)
    low = torch.where(d == d.amin(1, keepdim=True), j[None], H).amin(1)
    out = dict(rank=(d < true).sum(1).int(), true_distance=true[:, 0].long(), top1=low.int())
    return dict(out, distances=d.long()) if st["case"].get("matrix") else out


def _frame(n):
    """Rows of the rotation that takes each (float64) normal to the z axis."""
    x, y, z = n.unbind(1)
    h = torch.sqrt(x * x + y * y)
    ax, ay = torch.where(h > 0, x / h, 1.0), torch.where(h > 0, y / h, 0.0)
    g = torch.sqrt(h * h + z * z)
    bx, bz = torch.where(g > 0, h / g, 0.0), torch.where(g > 0, z / g, 1.0)
    o = torch.zeros_like(x)
    return torch.stack([torch.stack([bz * ax, bz * ay, -bx], 1), torch.stack([-ay, ax, o], 1),
                        torch.stack([bx * ax, bx * ay, bz], 1)], 1)


def _wedge(p, q, R):
    """Signed area, within the disk of radius R, of the triangle (0, p, q) of plane points."""
    d = q - p
    A = (d * d).sum(-1)
    B = (p * d).sum(-1)
    disc = B * B - A * ((p * p).sum(-1) - R * R)
    root = torch.sqrt(disc.clamp(min=0.0))
    cuts = (disc > 0) & (A > 0)
    safe = torch.where(A > 0, A, 1.0)
    t0 = torch.where(cuts, ((-B - root) / safe).clamp(0, 1), 1.0)[..., None]
    t1 = torch.where(cuts, ((-B + root) / safe).clamp(0, 1), 1.0)[..., None]
    u, w = p + t0 * d, p + t1 * d

    def cross(s, t):
        return s[..., 0] * t[..., 1] - s[..., 1] * t[..., 0]

    def sector(s, t):
        c = cross(s, t)
        return torch.where(c == 0, 0.0, torch.atan2(c, (s * t).sum(-1)))

    return 0.5 * R * R * (sector(p, u) + sector(w, q)) + 0.5 * cross(u, w)


def _area_inside(T, R):
    """Area of triangles T [n, 3, 3] within the cylinder of radius R and |z| <= R / 2."""
    H = 0.5 * R
    a, b = T, T[:, [1, 2, 0]]
    n = torch.linalg.cross(T[:, 1] - T[:, 0], T[:, 2] - T[:, 0])
    d = b - a
    dz = torch.where(d[..., 2] != 0, d[..., 2], 1.0)
    t_top, t_bot = (H - a[..., 2]) / dz, (-H - a[..., 2]) / dz
    up = d[..., 2] > 0
    flat = d[..., 2] == 0
    lo = torch.where(flat, 0.0, torch.where(up, t_bot, t_top)).clamp(0, 1)
    hi = torch.where(flat, (a[..., 2].abs() <= H).double(), torch.where(up, t_top, t_bot)).clamp(0, 1)
    hi = torch.maximum(lo, hi)
    xy, dxy = a[..., :2], d[..., :2]
    area = _wedge(xy + lo[..., None] * dxy, xy + hi[..., None] * dxy, R).sum(1)
    # the cuts along z = H and z = -H close the clipped outline
    for plane, t, above in ((H, t_top, True), (-H, t_bot, False)):
        sa = a[..., 2] > plane if above else a[..., 2] < -H
        sb = b[..., 2] > plane if above else b[..., 2] < -H
        pt = xy + t[..., None] * dxy
        leaves, enters = (~sa & sb), (sa & ~sb)
        x = torch.where(leaves[..., None], pt, 0.0).sum(1)
        y = torch.where(enters[..., None], pt, 0.0).sum(1)
        area = area + torch.where(leaves.any(1), _wedge(x, y, R), 0.0)
    return area.abs() * n.norm(dim=1) / n[:, 2].abs().clamp(min=1e-300)


def _exact_clutter(st):
    case, R = st["case"], float(np.float32(st["case"]["R"]))
    v, f = st["vertices"].double(), st["triangles"].long()
    obj = f[:, 0] < _part_sizes(("ico", case["level"]))[0]
    o = st["origins"].long()
    frames = _frame(st["normals"][o].double())
    both = []
    step = max(1, int(3e7) // max(1, f.shape[0]))
    for s in range(0, o.numel(), step):
        P = torch.einsum("okj,ovj->ovk", frames[s:s + step], v[None] - v[o[s:s + step], None])
        z = P[..., 2]
        # triangles that can reach the volume: not above or below it, not beside it
        far = (P[..., 0] > R) * 1 + (P[..., 0] < -R) * 2 + (P[..., 1] > R) * 4 + \
            (P[..., 1] < -R) * 8 + (z > 0.5 * R) * 16 + (z < -0.5 * R) * 32
        far = far.to(torch.uint8)
        oi, ti = ((far[:, f[:, 0]] & far[:, f[:, 1]] & far[:, f[:, 2]]) == 0).nonzero(as_tuple=True)
        ar = _area_inside(P[oi[:, None], f[ti]], R)
        sums = torch.zeros(2, P.shape[0], dtype=torch.float64, device=DEV)
        sums[0].index_add_(0, oi, ar)
        sums[1].index_add_(0, oi, torch.where(obj[ti], ar, 0.0))
        both.append(sums)
    total, part = torch.cat(both, 1)
    return total, part, (total - part) / total
