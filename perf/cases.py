"""The work that users of this voxelizer have it do, as measurable cases.

``listed()`` holds the fixed cases and ``draw(rng)`` more of the same ranges; ``prepare`` makes a
case's inputs on the GPU (or, for the host pipeline, in pinned host memory) from a seed, ``run`` is
one pass through the public entry points, ``work`` the bytes and operations a pass cannot do
without, and ``exact`` the same outputs from plain 64-bit integer torch arithmetic.

Meshes follow the recipes of ``meshgen`` (jittered Kuhn lattices, clipped to a torus or to a union
of spheres, with or without slivers), made on the GPU because they are made many times.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2106_01326_gb300 import batch, pipeline, slabs, voxtet

PERMS = ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))
KEPT = {"cube": 1.0, "torus": 0.0853, "blobs": 0.12}  # about the share of the lattice a shape keeps


def listed():
    return [
        # a small part (about 3k tets, as the small meshes of the tests and of smoke()) into a small
        # grid, one blocking call with everything at its defaults: the latency of an interactive tool
        {"name": "call_64", "kind": "dense", "n": 18, "res": 64, "shape": "blobs", "sliver": 0.0, "sync": True},
        # an ordinary part, enqueued without waiting (the torus configuration)
        {"name": "torus_256", "kind": "dense", "n": 48, "res": 256, "shape": "torus", "sliver": 0.0, "sync": False},
        # the headline workload of bench.py: 1.3 M tets, 2 % of them slivers
        {"name": "sliver_512", "kind": "dense", "n": 60, "res": 512, "shape": "cube", "sliver": 0.02, "sync": False},
        # the same mesh on the finer grid of the second configuration
        {"name": "sliver_1024", "kind": "dense", "n": 60, "res": 1024, "shape": "cube", "sliver": 0.02, "sync": False},
        # the other end of the served stream's range: its smallest meshes (about a thousand tets)
        # on its finest grid, tets tens of voxels wide
        {"name": "coarse_512", "kind": "dense", "n": 12, "res": 512, "shape": "blobs", "sliver": 0.0, "sync": False},
        # a grid fitted to a part: unequal odd sides, an origin and a voxel size that are not round
        {"name": "ragged_grid", "kind": "grid", "n": 40, "rx": 421, "ry": 217, "rz": 333, "shape": "blobs",
         "sliver": 0.02, "z0": 0, "z1": 333},
        # one rank's eighth of the headline grid, as a z-partition across processes hands it out
        {"name": "slab_512", "kind": "grid", "n": 60, "rx": 512, "ry": 512, "rz": 512, "shape": "cube",
         "sliver": 0.02, "z0": 192, "z1": 256},
        # a structured mesh whose vertices are lattice integers, open tetrahedra: samples fall
        # exactly on shared faces, many faces are parallel to x
        {"name": "lattice_open_256", "kind": "fixed", "n": 32, "res": 256, "mode": 1},
        # the many-mesh batch of bench.py: 256 parts of 1k-100k tets on 32^3-128^3 grids
        {"name": "batch_256", "kind": "batch", "jobs": 256, "lo": 1000, "hi": 100000, "res_lo": 32, "res_hi": 128},
        # one full batch of the server: 64 requests over meshes of 1k-2M tets and 64^3-512^3 grids
        {"name": "served_64", "kind": "batch", "jobs": 64, "lo": 1000, "hi": 1000000, "res_lo": 64, "res_hi": 512},
        # brick-sparse output of a fine grid that would be 8.6 GB dense
        {"name": "sparse_4096", "kind": "sparse", "n": 73, "rx": 4096, "ry": 4096, "rz": 4096, "shape": "torus"},
        # a stream of host meshes into host grids, the copies overlapped (bench.py's end-to-end number)
        {"name": "stream_512", "kind": "stream", "n": 60, "res": 512, "shape": "cube", "sliver": 0.02, "jobs": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dense", "dense", "dense", "grid", "grid", "fixed", "batch", "sparse", "stream"])
    if kind == "dense":
        res = 1 << rng.randint(5, 10)
        shape = rng.choice(["cube", "torus", "blobs"])
        return {"kind": kind, "n": _log(rng, max(8, res // 64), 64), "res": res, "shape": shape,
                "sliver": 0.02 if shape == "cube" else rng.choice([0.0, 0.02]), "sync": rng.random() < 0.3}
    if kind == "grid":
        sides = [_log(rng, 17, 700) for _ in range(3)]
        z0 = rng.choice([0, rng.randrange(sides[2])])
        z1 = sides[2] if rng.random() < 0.5 else rng.randint(z0 + 1, sides[2])
        shape = rng.choice(["cube", "blobs"])
        return {"kind": kind, "n": _log(rng, max(8, max(sides) // 40), 64), "rx": sides[0], "ry": sides[1],
                "rz": sides[2], "shape": shape, "sliver": 0.02 if shape == "cube" else rng.choice([0.0, 0.02]),
                "z0": z0, "z1": z1}
    if kind == "fixed":
        res = 1 << rng.randint(5, 9)
        return {"kind": kind, "n": 1 << rng.randint(2, 5), "res": res, "mode": rng.randint(0, 1)}
    if kind == "batch":
        top = rng.choice([64, 128, 256])
        return {"kind": kind, "jobs": _log(rng, 6, 256 if top < 256 else 64), "lo": 1000,
                "hi": _log(rng, 4000, 120000), "res_lo": rng.choice([32, 64]), "res_hi": top}
    if kind == "sparse":
        sides = [_log(rng, 500, 3000) for _ in range(3)]
        return {"kind": kind, "n": _log(rng, 24, 73), "rx": sides[0], "ry": sides[1], "rz": sides[2],
                "shape": rng.choice(["torus", "blobs"])}
    return {"kind": kind, "n": _log(rng, 12, 56), "res": 1 << rng.randint(6, 8), "shape": "cube", "sliver": 0.02,
            "jobs": rng.randint(2, 8)}


# ---------------------------------------------------------------- inputs

def _generator(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt) % (1 << 31))
    return g


def _inside(p, shape, g):
    """Which of the points p are inside the shape (a torus, or a union of three random spheres)."""
    if shape == "torus":
        return torch.hypot(torch.hypot(p[:, 0] - 0.5, p[:, 1] - 0.5) - 0.3, p[:, 2] - 0.5) < 0.12
    c = torch.rand((3, 3), generator=g, device="cuda", dtype=torch.float64) * 0.4 + 0.3
    r = torch.rand(3, generator=g, device="cuda", dtype=torch.float64) * 0.1 + 0.15
    hit = torch.zeros(len(p), dtype=torch.bool, device="cuda")
    for k in range(3):
        hit |= (p - c[k]).norm(dim=1) < r[k]
    return hit


def _lattice(n):
    """Vertices (i, j, l) of the n^3 Kuhn lattice and its tets, x fastest, on the GPU."""
    a = torch.arange(n + 1, device="cuda")
    l, j, i = torch.meshgrid(a, a, a, indexing="ij")
    ijk = torch.stack([i.reshape(-1), j.reshape(-1), l.reshape(-1)], 1)
    corner = ijk[(ijk < n).all(dim=1)]
    off = torch.zeros((6, 4, 3), dtype=torch.int64)
    for t, perm in enumerate(PERMS):
        for k, axis in enumerate(perm):
            off[t, k + 1:, axis] += 1
    pts = corner[:, None, None, :] + off.cuda()[None]
    tets = (pts[..., 2] * (n + 1) + pts[..., 1]) * (n + 1) + pts[..., 0]
    return ijk, tets.reshape(-1, 4)


def _mesh(n, shape, sliver, seed, salt=0):
    """(verts float32 [v, 3], tets int32 [t, 4]) in the unit cube, on the GPU."""
    g = _generator(seed, salt)
    ijk, tets = _lattice(n)
    pos = ijk.to(torch.float64)
    jit = (torch.rand(pos.shape, generator=g, device="cuda", dtype=torch.float64) - 0.5) * 0.5
    interior = ((ijk > 0) & (ijk < n)).all(dim=1, keepdim=True)
    pos = (pos + jit * interior) / n
    if shape != "cube":
        tets = tets[_inside(pos[tets].mean(dim=1), shape, g)]
        used, inv = torch.unique(tets.reshape(-1), return_inverse=True)
        pos, tets = pos[used], inv.reshape(-1, 4)
    if sliver and len(tets):
        # near-flat tets: a new vertex within 1e-6 of the plane of the opposite face
        pick = torch.nonzero(torch.rand(len(tets), generator=g, device="cuda") < sliver).reshape(-1)
        which = torch.randint(0, 4, (len(pick),), generator=g, device="cuda")
        old = tets[pick]
        p = pos[old]
        rest = torch.stack([p[torch.arange(len(pick), device="cuda"), (which + k) % 4] for k in (1, 2, 3)], 1)
        x = p[torch.arange(len(pick), device="cuda"), which]
        nrm = torch.linalg.cross(rest[:, 1] - rest[:, 0], rest[:, 2] - rest[:, 0])
        nrm = nrm / nrm.norm(dim=1, keepdim=True)
        h = ((x - rest[:, 0]) * nrm).sum(dim=1, keepdim=True)
        lift = torch.rand((len(pick), 1), generator=g, device="cuda", dtype=torch.float64) * 1e-6
        new = x - h * nrm + torch.where(h >= 0, lift, -lift) * nrm
        tets = tets.clone()
        tets[pick, which] = len(pos) + torch.arange(len(pick), device="cuda")
        pos = torch.cat([pos, new])
    return pos.to(torch.float32).contiguous(), tets.to(torch.int32).contiguous()


def _structured(n, res, seed):
    """The n^3 Kuhn lattice over the whole grid in lattice integers, moved by half a voxel or not and
    by some whole voxels per axis: faces on x = y, y = z and x = z planes through sample centres."""
    ijk, tets = _lattice(n)
    g = _generator(seed, 1)
    half = (1 << 19) // res
    shift = torch.randint(0, 2, (1,), generator=g, device="cuda") * half
    shift = shift + torch.randint(-(res // 8), res // 8 + 1, (3,), generator=g, device="cuda") * 2 * half
    return (ijk * ((1 << 20) // n) + shift).to(torch.int32).contiguous(), tets.to(torch.int32).contiguous()


def _placed(case, seed):
    """A part inside a fine grid of voxel edge h, and h: the same part for every seed, mirrored and
    moved by whole bricks (its coordinates are multiples of h / 64, so both are exact), so that every
    seed's part fills as many bricks."""
    dims = (case["rx"], case["ry"], case["rz"])
    h = 2.0 ** -(max(dims) - 1).bit_length()
    v, t = _mesh(case["n"], case["shape"], 0.0, 0)
    rng = np.random.default_rng([int(seed), 11])
    cols = []
    for q, brick in enumerate((32, 8, 8)):
        span = dims[q] // brick * brick
        x = torch.round(v[:, q].to(torch.float64) * span * 64) / 64
        if rng.integers(2):
            x = span - x
        reach = int(0.04 * span / brick)  # the shapes stay 0.05 away from the lattice's sides
        cols.append((x + brick * int(rng.integers(-reach, reach + 1))) * h)
    return torch.stack(cols, 1).to(torch.float32).contiguous(), t, h


def _fit(case):
    """Origin, voxel size and per-axis scale that fit the unit cube into a general grid."""
    h = 0.0137
    origin = (-1.25, 0.4, 2.0)
    return origin, h, [case["rx"] * h, case["ry"] * h, case["rz"] * h]


def _batch_jobs(case, seed):
    """(lattice size, grid side, salt) per job: tet counts log-uniform, grid sides uniform."""
    rng = np.random.default_rng([int(seed), 7])
    sides = [r for r in (32, 64, 128, 256, 512) if case["res_lo"] <= r <= case["res_hi"]]
    jobs = []
    for k in range(case["jobs"]):
        # evenly spread over the logarithm of the range (shuffled), so that batches of different
        # seeds are about the same amount of work
        t = math.exp(math.log(case["lo"]) + math.log(case["hi"] / case["lo"]) * (k + rng.random()) / case["jobs"])
        jobs.append((max(2, round((t / (6 * KEPT["blobs"])) ** (1 / 3))), sides[k % len(sides)]))
    order = rng.permutation(len(jobs))
    sizes = [jobs[o][0] for o in order]
    return [(sizes[k], jobs[k][1], k) for k in range(len(jobs))]


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": dict(case)}
    if kind in ("dense", "grid"):
        v, t = _mesh(case["n"], case["shape"], case["sliver"], seed)
        if kind == "dense":
            s["out"] = voxtet.alloc_grid(case["res"])
            s["ws"] = voxtet.alloc_workspace(len(t), len(v), case["res"])
        else:
            origin, h, scale = _fit(case)
            dims, zr = (case["rx"], case["ry"], case["rz"]), (case["z0"], case["z1"])
            v = (v * torch.tensor(scale, device="cuda") + torch.tensor(origin, device="cuda")).contiguous()
            if zr != (0, dims[2]):  # a rank holds the tets that reach its slab
                v, t = slabs.slab_mesh(v.cpu().numpy(), t.cpu().numpy(), origin, h, *zr)
                v, t = torch.from_numpy(v).cuda(), torch.from_numpy(t).cuda()
            s["out"] = voxtet.alloc_grid_dims(dims, zr)
            s["ws"] = voxtet.alloc_workspace(len(t), len(v), max(dims))
        s["verts"], s["tets"] = v, t
    elif kind == "fixed":
        s["verts"], s["tets"] = _structured(case["n"], case["res"], seed)
        s["out"] = voxtet.alloc_grid(case["res"])
        s["ws"] = voxtet.alloc_workspace(len(s["tets"]), len(s["verts"]), case["res"])
    elif kind == "batch":
        jobs = _batch_jobs(case, seed)
        words = [voxtet.grid_words(res) for _, res, _ in jobs]
        s["out"] = torch.empty(sum(words), dtype=torch.int32, device="cuda")  # every job's grid, one after another
        s["specs"], at = [], 0
        for (n, res, salt), w in zip(jobs, words):
            mesh = batch.Mesh(*_mesh(n, "blobs", 0.0, seed, salt))
            s["specs"].append(batch.JobSpec(mesh, res, s["out"][at:at + w].view(res, res, -1)))
            at += w
        s["plan"] = batch.Plan(batch.batch_workspace_size(s["specs"]), len(jobs))
    elif kind == "sparse":
        dims = (case["rx"], case["ry"], case["rz"])
        s["verts"], s["tets"], s["h"] = _placed(case, seed)
        s["depth"] = voxtet.default_slab_depth(dims)
        s["ws"] = voxtet.alloc_workspace(len(s["tets"]), len(s["verts"]), max(dims))
        s["scratch"] = torch.empty(voxtet.sparse_scratch_size(dims, s["depth"]), dtype=torch.uint8, device="cuda")
        bricks = -(-dims[0] // 32) * -(-dims[1] // 8) * -(-dims[2] // 8)
        s["cap"] = bricks // 4 + 1024  # the shapes fill less than a quarter of the bricks
    else:
        s["host"] = []
        for k in range(case["jobs"]):
            v, t = _mesh(case["n"], case["shape"], case["sliver"], seed, k)
            s["host"].append((v.cpu().pin_memory(), t.cpu().pin_memory()))
        s["grids"] = torch.empty((case["jobs"], case["res"], case["res"], (case["res"] + 31) // 32),
                                 dtype=torch.int32).pin_memory()
        s["pipe"] = pipeline.HostPipeline(max(len(v) for v, _ in s["host"]), max(len(t) for _, t in s["host"]),
                                          case["res"], depth=4)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "dense":
        res = case["res"]
        if case["sync"]:  # the plain call: the library's buffers are allocated and its status is checked
            return voxtet.voxelize(s["verts"], s["tets"], (0.0, 0.0, 0.0), 1.0 / res, res)
        return voxtet.voxelize(s["verts"], s["tets"], (0.0, 0.0, 0.0), 1.0 / res, res, out=s["out"],
                               workspace=s["ws"], sync=False)
    if kind == "grid":
        origin, h, _ = _fit(case)
        return voxtet.voxelize_grid(s["verts"], s["tets"], origin, h, (case["rx"], case["ry"], case["rz"]),
                                    z_range=(case["z0"], case["z1"]), out=s["out"], workspace=s["ws"], sync=False)
    if kind == "fixed":
        return voxtet.voxelize_fixed(s["verts"], s["tets"], case["res"], out=s["out"], workspace=s["ws"],
                                     mode=case["mode"], sync=False)
    if kind == "batch":
        s["plan"].wait()  # the statuses of this plan's previous batch, as a server collects them
        st = s["plan"].run(s["specs"])
        if st != voxtet.OK:
            raise voxtet.VoxtetError(st)
        return s["out"]
    if kind == "sparse":
        keys, words = voxtet.voxelize_sparse(s["verts"], s["tets"], (0.0, 0.0, 0.0), s["h"],
                                             (case["rx"], case["ry"], case["rz"]), slab_depth=s["depth"],
                                             max_bricks=s["cap"], workspace=s["ws"], scratch=s["scratch"])
        return {"keys": keys, "words": words}
    for k, (v, t) in enumerate(s["host"]):
        s["pipe"].submit(v, t, s["grids"][k], (0.0, 0.0, 0.0), 1.0 / case["res"])
    s["pipe"].wait()
    return s["grids"]


# ---------------------------------------------------------------- what a pass cannot do without

def _mesh_work(n, shape, sliver, dims, z=(0.0, 1.0)):
    """(bytes, flops) of one mesh: vertices and tets read once; per tet 150 operations (box,
    orientation, four face planes), per (tet, x-row) holding a sample 25 (four face bounds and the
    interval's words).  A tet of a cell of w voxels per axis has about wy wz / 2 such rows (counted
    on the headline mesh: 36 at w = 8.5)."""
    share = KEPT[shape] * (z[1] - z[0])
    tets = 6 * n ** 3 * share
    verts = (n + 1) ** 3 * share + sliver * tets
    w = [d / n for d in dims]
    rows = tets * 0.5 * w[1] * w[2] * min(1.0, w[0])
    return 16 * tets + 12 * verts, 150 * tets + 25 * rows


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0
        for n, res, _ in _batch_jobs(case, 0):
            x, y = _mesh_work(n, "blobs", 0.0, (res,) * 3)
            b, f = b + x + 4 * voxtet.grid_words(res), f + y
        return {"bytes": b, "flops": f}
    if kind in ("grid", "sparse"):
        dims = (case["rx"], case["ry"], case["rz"])
        z = (case["z0"] / dims[2], case["z1"] / dims[2]) if kind == "grid" else (0.0, 1.0)
        b, f = _mesh_work(case["n"], case["shape"], case.get("sliver", 0.0), dims, z)
        if kind == "grid":
            b += 4 * (case["z1"] - case["z0"]) * dims[1] * -(-dims[0] // 32)
        else:
            b += KEPT[case["shape"]] * dims[0] * dims[1] * dims[2] / 2048 * 264  # 256 bytes and a key per brick
        return {"bytes": b, "flops": f}
    res = case["res"]
    b, f = _mesh_work(case["n"], case.get("shape", "cube"), case.get("sliver", 0.0), (res,) * 3)
    b, f = b + 4 * voxtet.grid_words(res), f
    return {"bytes": b * case.get("jobs", 1), "flops": f * case.get("jobs", 1)}


# ---------------------------------------------------------------- the same grids in 64-bit integers

def _snap(v, origin, h, k):
    """X = round_half_even((v - origin) / h * 2^(20-k)) in doubles, as 64-bit integers; the origin
    and the voxel size as the float32 values the C entry points take."""
    o = torch.tensor([float(np.float32(x)) for x in origin], dtype=torch.float64, device=v.device)
    return torch.round((v.to(torch.float64) - o) / float(np.float32(h)) * 2.0 ** (20 - k)).to(torch.int64)


def _exact_grid(x, tets, dims, k, zr, strict=False):
    """Bit grid of lattice vertices x (int64): the point-in-tetrahedron test on every sample of every
    tet's bounding box, in 64-bit integers."""
    rx, ry, rz = dims
    z0, z1 = zr
    grid = torch.zeros((z1 - z0) * ry * rx, dtype=torch.bool, device=x.device)
    step, half = 1 << (20 - k), 1 << (19 - k)
    p = x[tets.to(torch.int64)]
    e = p[:, 1:] - p[:, :1]
    v6 = (e[:, 0] * torch.linalg.cross(e[:, 1], e[:, 2])).sum(dim=1)
    p = torch.where((v6 < 0)[:, None, None], p[:, [0, 1, 3, 2]], p)
    lim_lo = torch.tensor([0, 0, z0], device=x.device)
    lim_hi = torch.tensor([rx - 1, ry - 1, z1 - 1], device=x.device)
    lo = torch.maximum(-torch.div(half - p.amin(dim=1), step, rounding_mode="floor"), lim_lo)
    hi = torch.minimum(torch.div(p.amax(dim=1) - half, step, rounding_mode="floor"), lim_hi)
    count = (hi - lo + 1).clamp(min=0)
    live = (v6 != 0) & (count.prod(dim=1) > 0)
    p, lo, count = p[live], lo[live], count[live]
    if not len(p):
        return _pack(grid.view(z1 - z0, ry, rx))
    ends = torch.cumsum(count.prod(dim=1), 0)
    # face m: (P - a) . n >= 0 inside, opposite vertex m
    faces = []
    for m, (a, b, c) in enumerate(((1, 3, 2), (0, 2, 3), (0, 3, 1), (0, 1, 2))):
        nrm = torch.linalg.cross(p[:, b] - p[:, a], p[:, c] - p[:, a])
        faces.append((p[:, a], nrm))
    total, chunk, done, t0 = int(ends[-1]), 1 << 24, 0, 0
    while t0 < len(p):
        t1 = max(t0 + 1, int(torch.searchsorted(ends, done + chunk, right=True)))
        cnt = count[t0:t1].prod(dim=1)
        which = torch.repeat_interleave(torch.arange(t0, t1, device=x.device), cnt)
        at = torch.arange(len(which), device=x.device) + done - (ends[which] - count[which].prod(dim=1))
        n = count[which]
        ix = lo[which, 0] + at % n[:, 0]
        iy = lo[which, 1] + torch.div(at, n[:, 0], rounding_mode="floor") % n[:, 1]
        iz = lo[which, 2] + torch.div(at, n[:, 0] * n[:, 1], rounding_mode="floor")
        inside = torch.ones(len(which), dtype=torch.bool, device=x.device)
        for a, nrm in faces:
            q, w = a[which], nrm[which]
            lam = ((ix * step + half - q[:, 0]) * w[:, 0] + (iy * step + half - q[:, 1]) * w[:, 1]
                   + (iz * step + half - q[:, 2]) * w[:, 2])
            inside &= (lam > 0) if strict else (lam >= 0)
        grid[(((iz - z0) * ry + iy) * rx + ix)[inside]] = True
        done, t0 = int(ends[t1 - 1]), t1
    return _pack(grid.view(z1 - z0, ry, rx))


def _pack(g):
    """bool [z, y, x] -> int32 words [z, y, ceil(x / 32)], lowest x in bit 0."""
    z, y, x = g.shape
    w = -(-x // 32)
    g = torch.nn.functional.pad(g, (0, 32 * w - x)).view(z, y, w, 32)
    out = torch.zeros((z, y, w), dtype=torch.int64, device=g.device)
    for b in range(32):
        out |= g[..., b].to(torch.int64) << b
    return torch.where(out >= 1 << 31, out - (1 << 32), out).to(torch.int32)


def _samples(n, shape, dims):
    """About how many samples the bounding boxes of a mesh's tets hold."""
    return 6 * n ** 3 * KEPT[shape] * math.prod(1.4 * d / n + 0.5 for d in dims)


def exact(case, seed):
    kind = case["kind"]
    if kind == "sparse":
        return None  # terabytes of samples
    if kind == "batch":
        jobs = _batch_jobs(case, seed)
        if sum(_samples(n, "blobs", (res,) * 3) for n, res, _ in jobs) > 5e9:
            return None
        grids = []
        for n, res, salt in jobs:
            v, t = _mesh(n, "blobs", 0.0, seed, salt)
            k = res.bit_length() - 1
            grids.append(_exact_grid(_snap(v, (0, 0, 0), 1.0 / res, k), t, (res,) * 3, k, (0, res)).reshape(-1))
        return torch.cat(grids)
    dims = (case["rx"], case["ry"], case["rz"]) if kind == "grid" else (case["res"],) * 3
    if case.get("jobs", 1) * _samples(case["n"], case.get("shape", "cube"), dims) > 5e9:
        return None
    k = (max(dims) - 1).bit_length()
    if kind == "fixed":
        x, t = _structured(case["n"], case["res"], seed)
        return _exact_grid(x.to(torch.int64), t, dims, k, (0, dims[2]), case["mode"] == 1)
    if kind == "stream":
        grids = []
        for j in range(case["jobs"]):
            v, t = _mesh(case["n"], case["shape"], case["sliver"], seed, j)
            grids.append(_exact_grid(_snap(v, (0, 0, 0), 1.0 / dims[0], k), t, dims, k, (0, dims[2])).cpu())
        return torch.stack(grids)
    v, t = _mesh(case["n"], case["shape"], case["sliver"], seed)
    if kind == "dense":
        return _exact_grid(_snap(v, (0, 0, 0), 1.0 / dims[0], k), t, dims, k, (0, dims[2]))
    origin, h, scale = _fit(case)
    v = v * torch.tensor(scale, device="cuda") + torch.tensor(origin, device="cuda")
    return _exact_grid(_snap(v, origin, h, k), t, dims, k, (case["z0"], case["z1"]))
