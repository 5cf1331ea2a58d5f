"""Performance cases of the Htex lookup library.

Each case is one pass of a user's program through the public entry points:
a request's lookups, a texture fit's step, a rendered frame, a displaced
mesh, a burst of served requests.  Sizes come from the benchmark's and the
tests' configurations; draw() spreads them over the same ranges.

Inputs are made from the seed: texels uniform over their range (stored
values of every level), halfedges and barycentrics uniform, footprints zero
or log-uniform over 2^-8..1 of a quad.  The mesh belongs to the case.
exact() evaluates the method's definitions (zero-bordered bilinear samples
of the three fetches, one normalisation) in 64-bit torch.
"""
import functools
import math

import numpy as np
import torch

import paper_2207_05618_gb300 as hx
from paper_2207_05618_gb300 import render, serve

ELEM = {"f32": 4, "u8": 1, "f16": 2, "bf16": 2, "e4m3": 1}
DEV = "cuda"


# ------------------------------------------------------------------- cases

def listed():
    M = 1 << 20
    return [
        # a small request against a resident asset (a picking ray fan, a probe
        # grid): launch latency
        dict(name="request_small", kind="lookup", around=48, rows=48, res_lo=6, res_hi=6, dtype="f16", channels=4,
             n=1021, footprint="loguniform", bin=False),
        # the tiny closed cube streamed with 16M level-0 queries: texels on
        # chip, queries and results through memory
        dict(name="cube_stream", kind="lookup", around=0, rows=0, res_lo=4, res_hi=4, dtype="f32", channels=4,
             n=16 * M, footprint="zero", bin=False),
        # asset scale, the benchmark's step: 5.7 GB of RGBA8, 16M trilinear
        # queries in random order, sorted by the library
        dict(name="asset_sorted", kind="lookup", around=256, rows=460, res_lo=6, res_hi=6, dtype="u8", channels=4,
             n=16 * M, footprint="loguniform", bin=True),
        # per-edge resolutions 8..128 of RGB8 albedo, queries in the order
        # they come (ray hits), an odd count
        dict(name="mixed_rgb8", kind="lookup", around=128, rows=128, res_lo=3, res_hi=7, dtype="u8", channels=3,
             n=1500001, footprint="loguniform", bin=False),
        # reduced precision: scaled FP8 texels, a memory-bound asset, sorted
        dict(name="precision_e4m3", kind="lookup", around=256, rows=115, res_lo=6, res_hi=6, dtype="e4m3", channels=4,
             n=4 * M - 21, footprint="loguniform", bin=True),
        # a training step through autograd (RGB FP32 textures, level 0):
        # texels written, looked up, loss, adjoint into a dense gradient
        dict(name="train_step", kind="train", around=160, rows=145, res_lo=5, res_hi=5, dtype="f32", channels=3,
             n=2 * M, footprint="zero", bin=False),
        # a step of the texture fit: lookup, loss, sorted adjoint, Adam
        dict(name="fit_step", kind="fit", around=160, rows=145, res_lo=5, res_hi=5, dtype="f32", channels=3,
             n=2 * M, footprint="loguniform", bin=True),
        # anisotropic lookups, 1..16 probes
        dict(name="aniso16", kind="aniso", around=256, rows=115, res_lo=6, res_hi=6, dtype="u8", channels=4,
             n=4 * M, max_aniso=16, bin=False),
        # a 1080p frame of the asset: one query per pixel, every pixel looked up
        dict(name="frame_1080p", kind="frame", around=256, rows=460, res_lo=5, res_hi=5, dtype="u8", channels=4,
             width=1920, height=1080, max_aniso=0),
        # displacement of a tessellated asset (45 lattice points a triangle)
        # by a one-channel map
        dict(name="displace_t8", kind="displace", around=256, rows=115, res_lo=5, res_hi=5, dtype="f16", channels=1,
             tess=8, channel=0),
        # end to end: queries and results in page-locked host memory
        dict(name="host_pinned", kind="host", around=256, rows=115, res_lo=6, res_hi=6, dtype="u8", channels=4,
             n=4 * M - 3, footprint="loguniform", bin=True),
        # a burst of served requests, 1k..1M queries, of three assets
        dict(name="serve_burst", kind="serve", requests=24, lo=1000, hi=1000000),
    ]


def _size(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def _edges_about(around, rows):
    return 2.25 * around * rows


def draw(rng):
    kind = rng.choice(["lookup", "lookup", "lookup", "train", "fit", "aniso", "frame", "displace", "host", "serve"])
    if kind == "serve":
        return dict(kind="serve", requests=rng.randint(4, 32), lo=rng.randint(500, 2000), hi=_size(rng, 20000, 800000))
    around = 2 * _size(rng, 12, 128)
    rows = _size(rng, 12, 400)
    c = dict(kind=kind, around=around, rows=rows)
    lo = rng.randint(2, 6)
    c["res_lo"], c["res_hi"] = lo, lo if rng.random() < 0.5 else rng.randint(lo, 7)
    c["dtype"] = "f32" if kind in ("train", "fit") else rng.choice(["f32", "u8", "u8", "f16", "bf16", "e4m3"])
    c["channels"] = rng.choice([1, 2, 3, 4, 4])
    # textures of at most 1.5 GB (0.8 GB where they are trained)
    most = 0.8e9 if kind in ("train", "fit") else 1.5e9
    texel = c["channels"] * ELEM[c["dtype"]]
    while _edges_about(c["around"], c["rows"]) * 1.34 * 4.0 ** c["res_hi"] * texel > most:
        c["rows"] = max(4, c["rows"] // 2)
        if c["rows"] == 4 and c["around"] > 24:
            c["around"] = 24
        elif c["rows"] == 4:
            c["res_hi"] -= 1
            c["res_lo"] = min(c["res_lo"], c["res_hi"])
    if kind == "frame":
        c["width"], c["height"] = _size(rng, 200, 1920), _size(rng, 150, 1080)
        c["max_aniso"] = rng.choice([0, 0, 4, 16])
        return c
    if kind == "displace":
        c["tess"], c["channel"] = rng.randint(1, 8), rng.randint(0, c["channels"] - 1)
        return c
    c["bin"] = rng.random() < 0.5
    if kind == "aniso":
        c["n"], c["max_aniso"] = _size(rng, 1000, 4 << 20), rng.choice([2, 4, 8, 16])
        return c
    most_n = {"lookup": 16 << 20, "train": 2 << 20, "fit": 2 << 20, "host": 4 << 20}[kind]
    c["n"] = _size(rng, 1000, most_n)
    c["footprint"] = rng.choice(["zero", "loguniform"])
    return c


# ------------------------------------------------------------------ meshes

@functools.lru_cache(maxsize=8)
def mesh_faces(around, rows, closed):
    """Face sizes, vertex lists, vertex count and positions: a unit cube
    (around = 0), else a band of around x rows quads, open at both ends or
    closed into a torus; 30% of the quads split into triangles, one pair of
    neighbours in ten merged into a hexagon."""
    if around == 0:
        faces = [[0, 2, 3, 1], [4, 5, 7, 6], [0, 1, 5, 4], [2, 6, 7, 3], [0, 4, 6, 2], [1, 3, 7, 5]]
        pos = np.array([[k & 1, (k >> 1) & 1, (k >> 2) & 1] for k in range(8)], np.float32)
        return np.full(6, 4, np.int32), np.array(sum(faces, []), np.int32), 8, pos
    rng = np.random.default_rng(around * 1000003 + rows)
    rings = rows if closed else rows + 1
    r, c = np.divmod(np.arange(rows * around, dtype=np.int64), around)

    def vert(row, col):
        return (row % rings) * around + col % around

    quad = np.stack([vert(r, c), vert(r, c + 1), vert(r + 1, c + 1), vert(r + 1, c)], 1)
    merged = np.repeat(rng.random(rows * around // 2) < 0.1, 2)
    split = ~merged & (rng.random(rows * around) < 0.3)
    other = rng.random(rows * around) < 0.5
    left = merged & (c % 2 == 0)
    h = np.nonzero(left)[0]
    hexa = np.stack([vert(r[h], c[h]), vert(r[h], c[h] + 1), vert(r[h], c[h] + 2), vert(r[h] + 1, c[h] + 2),
                     vert(r[h] + 1, c[h] + 1), vert(r[h] + 1, c[h])], 1)
    q = np.nonzero(~merged & ~split)[0]
    a, b = np.nonzero(split & other)[0], np.nonzero(split & ~other)[0]
    parts = [(h, hexa), (q, quad[q]), (a, quad[a][:, [0, 1, 2]]), (a, quad[a][:, [0, 2, 3]]),
             (b, quad[b][:, [0, 1, 3]]), (b, quad[b][:, [1, 2, 3]])]
    cell = np.concatenate([p[0] for p in parts])
    sizes = np.concatenate([np.full(len(p[0]), p[1].shape[1]) for p in parts])
    verts = np.concatenate([np.pad(p[1], ((0, 0), (0, 6 - p[1].shape[1])), constant_values=-1) for p in parts])
    order = np.argsort(cell, kind="stable")
    verts = verts[order]
    V = rings * around
    i, j = np.divmod(np.arange(V), around)
    th = 2 * np.pi * j / around
    if closed:
        ph = 2 * np.pi * i / rings
        pos = np.stack([(2 + np.cos(ph)) * np.cos(th), (2 + np.cos(ph)) * np.sin(th), np.sin(ph)], 1)
    else:
        pos = np.stack([np.cos(th), np.sin(th), i / around], 1)
    return sizes[order].astype(np.int32), verts[verts >= 0].astype(np.int32), V, pos.astype(np.float32)


@functools.lru_cache(maxsize=8)
def halfedges(around, rows, closed):
    """The halfedge operators of mesh_faces(...) as numpy arrays."""
    sizes, vert, V, _ = mesh_faces(around, rows, closed)
    H = len(vert)
    h = np.arange(H)
    first = np.repeat(np.cumsum(sizes) - sizes, sizes)
    size = np.repeat(sizes, sizes)
    nxt = first + (h - first + 1) % size
    prv = first + (h - first + size - 1) % size
    a, b = vert.astype(np.int64), vert[nxt].astype(np.int64)
    key, back = a * V + b, b * V + a
    order = np.argsort(key)
    at = np.minimum(np.searchsorted(key, back, sorter=order), H - 1)
    twin = np.where(key[order[at]] == back, order[at], -1)
    owner = (twin < 0) | (h < twin)
    ids = np.cumsum(owner) - 1
    edge = np.where(owner, ids, ids[np.where(owner, h, twin)])
    return dict(H=H, E=int(owner.sum()), next=nxt, prev=prv, twin=twin, edge=edge, vert=vert,
                face=np.repeat(np.arange(len(sizes)), sizes), sizes=sizes)


def _closed(case):
    return case["kind"] in ("train", "fit")


def _halfedges(case):
    return halfedges(case["around"], case["rows"], _closed(case))


def _mesh(case):
    sizes, verts, V, _ = mesh_faces(case["around"], case["rows"], _closed(case))
    return hx.Mesh(sizes, verts, V)


# ------------------------------------------------------------------ inputs

def _generator(seed, stream=0):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 64 + stream)


def resolutions(case, E):
    lo, hi = case["res_lo"], case["res_hi"]
    return np.random.default_rng(E * 31 + lo * 8 + hi).integers(lo, hi + 1, E).astype(np.int32)


def pool_offsets(log2n, channels, dtype):
    """Byte offset of every texture and the pool's size: full chains, each
    texture on a 16-byte boundary."""
    n = log2n.astype(np.int64)
    size = ((4 ** (n + 1) - 1) // 3 * channels * ELEM[dtype] + 15) // 16 * 16
    end = np.cumsum(size)
    return end - size, int(end[-1])


def random_texels(nbytes, dtype, g):
    """A pool of stored values as bytes on the GPU: U[0, 1) (the scaled
    formats: codes over their range)."""
    if dtype == "u8":
        return torch.randint(0, 256, (nbytes,), dtype=torch.uint8, device=DEV, generator=g)
    out = torch.empty(nbytes, dtype=torch.uint8, device=DEV)
    step = 1 << 28
    for at in range(0, nbytes, step):
        part = out[at:at + step]
        x = torch.rand(part.numel() // ELEM[dtype], device=DEV, generator=g)
        if dtype == "e4m3":
            x = (x * 448.0).to(torch.float8_e4m3fn)
        elif dtype != "f32":
            x = x.to(torch.float16 if dtype == "f16" else torch.bfloat16)
        part.copy_(x.view(torch.uint8))
    return out


def asset_inputs(case, seed, E, stream=0):
    g = _generator(seed, stream)
    log2n = resolutions(case, E)
    off, nbytes = pool_offsets(log2n, case["channels"], case["dtype"])
    pool = random_texels(nbytes, case["dtype"], g)
    scales = torch.rand(E, device=DEV, generator=g) + 0.5
    if case["dtype"] == "e4m3":
        scales = scales / 448.0
    return dict(log2n=log2n, off=off, pool=pool, scales=scales)


def _triangle(n, g):
    uv = torch.rand((n, 2), device=DEV, generator=g)
    return torch.where(uv.sum(1, keepdim=True) > 1, 1 - uv, uv)


def random_queries(H, n, footprint, g):
    q = torch.zeros((n, 4), dtype=torch.int32, device=DEV)
    q[:, 0] = torch.randint(0, H, (n,), dtype=torch.int32, device=DEV, generator=g)
    q[:, 1:3] = _triangle(n, g).view(torch.int32)
    if footprint == "loguniform":
        q[:, 3] = torch.exp2(torch.rand(n, device=DEV, generator=g) * 8 - 8).view(torch.int32)
    return q


def random_queries_aniso(H, n, g):
    """Major axis 2^-8..1, anisotropy 1..16 (both log-uniform), any direction."""
    q = torch.zeros((n, 8), dtype=torch.int32, device=DEV)
    q[:, 0] = torch.randint(0, H, (n,), dtype=torch.int32, device=DEV, generator=g)
    q[:, 1:3] = _triangle(n, g).view(torch.int32)
    major = torch.exp2(torch.rand(n, device=DEV, generator=g) * 8 - 8)
    minor = major * torch.exp(-torch.rand(n, device=DEV, generator=g) * math.log(16.0))
    th = torch.rand(n, device=DEV, generator=g) * (2 * math.pi)
    d = torch.stack([major * th.cos(), major * th.sin(), -minor * th.sin(), minor * th.cos()], 1)
    q[:, 4:] = d.view(torch.int32)
    return q


def view_projection(case):
    """A camera beside the cylinder that sees its height, row-major 4 x 4."""
    zc = 0.5 * case["rows"] / case["around"]
    aspect, near, far = case["width"] / case["height"], 0.2, 40.0
    t = 1.0 / math.tan(math.radians(45.0) / 2)
    proj = np.zeros((4, 4))
    proj[0, 0], proj[1, 1] = t / aspect, t
    proj[2, 2], proj[2, 3], proj[3, 2] = (far + near) / (near - far), 2 * far * near / (near - far), -1.0
    eye = np.array([1.2 + 1.6 * max(1.0, zc), 0.0, zc])
    view = np.array([[0, 1, 0, 0], [0, 0, 1, 0], [1, 0, 0, 0], [0, 0, 0, 1]], np.float64)
    view[:3, 3] = -view[:3, :3] @ eye
    return (proj @ view).astype(np.float32)


# The assets of a served burst: small meshes with large textures and the
# other way round.
SERVED = [dict(kind="asset", around=16, rows=15, res_lo=7, res_hi=7, dtype="u8", channels=4),
          dict(kind="asset", around=64, rows=60, res_lo=5, res_hi=5, dtype="f16", channels=4),
          dict(kind="asset", around=160, rows=145, res_lo=4, res_hi=4, dtype="u8", channels=4)]


def served_requests(case):
    """(asset, queries) of each request: sizes log-spaced and interleaved."""
    k = case["requests"]
    order = np.random.default_rng(k).permutation(k)
    sizes = np.exp(np.linspace(math.log(case["lo"]), math.log(case["hi"]), k))
    return [(int(i) % len(SERVED), int(sizes[i])) for i in order]


def served_queries(case, seed):
    g = _generator(seed, 5)
    meshes = [_halfedges(a) for a in SERVED]
    return [random_queries(meshes[a]["H"], n, "loguniform", g) for a, n in served_requests(case)]


# ----------------------------------------------------------------- prepare

def _upload(case, mesh, a):
    """The asset resident, its pool then filled on the device."""
    scaled = case["dtype"] in ("f16", "bf16", "e4m3")
    tex = hx.Textures.upload_pool(mesh, a["log2n"], np.zeros(a["pool"].numel(), np.uint8),
                                  a["scales"].cpu().numpy() if scaled else None, case["channels"], case["dtype"])
    tex.write_pool(a["pool"])
    return tex


def prepare(case, seed):
    if case["kind"] == "serve":
        return _prepare_server(case, seed)
    mesh = _mesh(case)
    a = asset_inputs(case, seed, mesh.E)
    s = dict(case=case, mesh=mesh, tex=_upload(case, mesh, a))
    g = _generator(seed, 1)
    kind, flags = case["kind"], hx.LOOKUP_BIN if case.get("bin") else 0
    s["flags"] = flags
    if kind in ("frame", "displace"):
        s["geometry"] = render.Geometry(mesh, mesh_faces(case["around"], case["rows"], _closed(case))[3])
    if kind == "frame":
        px = case["width"] * case["height"]
        s["camera"] = view_projection(case)
        s["q"] = torch.empty((px, 8 if case["max_aniso"] else 4), dtype=torch.int32, device=DEV)
        s["out"] = torch.empty((px, case["channels"]), device=DEV)
    elif kind == "aniso":
        s["q"] = random_queries_aniso(mesh.H, case["n"], g)
        s["out"] = torch.empty((case["n"], case["channels"]), device=DEV)
    elif kind != "displace":
        s["q"] = random_queries(mesh.H, case["n"], case["footprint"], g)
    if kind == "lookup":
        s["out"] = torch.empty((case["n"], case["channels"]), device=DEV)
    elif kind == "host":
        s["q"] = s["q"].cpu().pin_memory()
        s["out"] = torch.empty((case["n"], case["channels"]), pin_memory=True)
    elif kind in ("train", "fit"):
        s["target"] = torch.rand((case["n"], case["channels"]), device=DEV, generator=g)
        texels = a["pool"].view(torch.float32)
        if kind == "train":
            s["texels"] = texels.requires_grad_(True)
        else:
            s["master"] = texels
            s["grad"], s["m"], s["v"] = (torch.zeros_like(texels) for _ in range(3))
            s["step"] = 0
    return s


def _prepare_server(case, seed):
    meshes = [_mesh(c) for c in SERVED]
    assets = [asset_inputs(c, seed, mesh.E, 2 + k) for k, (c, mesh) in enumerate(zip(SERVED, meshes))]
    pools = [a["pool"].cpu().numpy() for a in assets]
    scales = [a["scales"].cpu().numpy() for a in assets]
    reqs = [(a, q.cpu().pin_memory(), torch.empty((q.shape[0], 4), pin_memory=True))
            for (a, _), q in zip(served_requests(case), served_queries(case, seed))]
    server = serve.Server(budget_bytes=4 << 30)
    ids = [server.add_asset(mesh, a["log2n"], pool, sc, c["channels"], c["dtype"])
           for c, mesh, a, pool, sc in zip(SERVED, meshes, assets, pools, scales)]
    # a server in use: every asset resident, every batch slot used once (a
    # batch takes at most 2^20 queries of one request)
    q, out = np.zeros((3 << 20, 4), np.int32), np.empty((3 << 20, 4), np.float32)
    for k in ids:
        server.submit(k, q.ctypes.data, len(q) if k == ids[0] else 1, out.ctypes.data)
        server.drain()
    server.poll()
    return dict(case=case, server=server, requests=[(ids[a], q, out) for a, q, out in reqs])


# --------------------------------------------------------------------- run

def run(s):
    return globals()["_run_" + s["case"]["kind"]](s)


def _run_lookup(s):
    return hx.lookup(s["tex"], s["q"], out=s["out"], flags=s["flags"])


def _run_host(s):
    return hx.lookup_host(s["tex"], s["q"], out=s["out"], flags=s["flags"])


def _run_aniso(s):
    return hx.lookup_aniso(s["tex"], s["q"], s["case"]["max_aniso"], out=s["out"], flags=s["flags"])


def _run_train(s):
    texels = s["texels"]
    texels.grad = None
    out = hx.HtexLookup.apply(texels, s["tex"], s["q"], s["flags"])
    loss = (out - s["target"]).square().mean()
    loss.backward()
    return {"out": out.detach(), "loss": loss.detach(), "grad": texels.grad}


def _run_fit(s):
    with torch.no_grad():
        out = hx.lookup(s["tex"], s["q"])
        diff = out - s["target"]
        n = diff.numel()
        loss = diff.double().square().sum() / n
        hx.lookup_backward(s["tex"], s["q"], (2.0 / n) * diff, grad_texels=s["grad"], flags=s["flags"])
        s["step"] += 1
        s["tex"].adam_step(s["master"], s["grad"], s["m"], s["v"], s["step"], 0.05)
    return {"out": out, "loss": loss, "texels": s["master"], "m": s["m"], "v": s["v"]}


def _run_frame(s):
    case, q = s["case"], s["q"]
    if case["max_aniso"]:
        s["geometry"].rasterize_aniso(s["camera"], case["width"], case["height"], queries=q)
        image = hx.lookup_aniso(s["tex"], q, case["max_aniso"], out=s["out"])
        return {"h": q[:, 0], "uv": q.view(torch.float32)[:, 1:3], "derivatives": q.view(torch.float32)[:, 4:],
                "image": image}
    s["geometry"].rasterize(s["camera"], case["width"], case["height"], queries=q)
    image = hx.lookup(s["tex"], q, out=s["out"])
    return {"h": q[:, 0], "uv": q.view(torch.float32)[:, 1:3], "footprint": q.view(torch.float32)[:, 3],
            "image": image}


def _run_displace(s):
    return s["geometry"].displace(s["tex"], s["case"]["tess"], 0.01, s["case"]["channel"])


def _run_serve(s):
    server = s["server"]
    for asset, q, out in s["requests"]:
        server.submit(asset, q.data_ptr(), q.shape[0], out.data_ptr())
    server.drain()
    server.poll()
    return [out for _, _, out in s["requests"]]


# -------------------------------------------------------------------- work

def _mean_taps(case, footprint):
    """Texels of nonzero weight per query, from a sample of 16,384."""
    rng = np.random.default_rng(3)
    n = rng.integers(case["res_lo"], case["res_hi"] + 1, (3, 16384))
    u, v = rng.random((2, 16384))
    u, v = np.where(u + v > 1, 1 - u, u), np.where(u + v > 1, 1 - v, v)
    f = 2.0 ** (rng.random(16384) * 8 - 8) if footprint == "loguniform" else np.full(16384, 2.0 ** -30)
    lam = np.maximum(np.log2(f) + n, 0.0)
    l0 = np.minimum(np.floor(lam), n)
    total = 0.0
    for level, on in ((l0, lam >= 0), (np.minimum(l0 + 1, n), (lam > 0) & (l0 < n))):
        N = 2.0 ** (n - level)

        def inside(x, k):
            i = np.floor(x * N[k] - 0.5)
            return (i >= 0).astype(int) + (i + 1 < N[k])

        total += (on[0] * inside(u, 0) * inside(v, 0)).mean()
        total += (on[1] * (u * N[1] < 0.5) * inside(v, 1)).mean()
        total += (on[2] * (v * N[2] < 0.5) * inside(u, 2)).mean()
    return total


def _asset_bytes(case):
    return pool_offsets(resolutions(case, _halfedges(case)["E"]), case["channels"], case["dtype"])[1]


def _lookup_work(case, n, footprint):
    """Queries and results once; of records and texels what the queries
    touch, at most all of them.  Per tap two operations a channel and about
    eight for its place and weight."""
    taps, pool = _mean_taps(case, footprint), _asset_bytes(case)
    texel = case["channels"] * ELEM[case["dtype"]]
    touched = min(pool, taps * texel * n) + 16 * min(n, _halfedges(case)["H"])
    return 16 * n + 4 * case["channels"] * n + touched, n * taps * (2 * case["channels"] + 8), touched


def work(case):
    kind = case["kind"]
    if kind == "serve":
        parts = [_lookup_work(SERVED[a], n, "loguniform") for a, n in served_requests(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    C = case["channels"]
    if kind in ("lookup", "host"):
        b, f, _ = _lookup_work(case, case["n"], case["footprint"])
        return {"bytes": b, "flops": f}
    if kind in ("train", "fit"):
        n, pool = case["n"], _asset_bytes(case)
        b, f, touched = _lookup_work(case, n, case["footprint"])
        # targets, and the upstream gradient written and read; the texels
        # into the pool and the dense gradient (train), or Adam's nine streams
        b += 12 * C * n + (3 if kind == "train" else 9) * pool
        return {"bytes": b, "flops": 2 * f + (0 if kind == "train" else 10 * pool / 4)}
    if kind == "aniso":
        probes = {2: 1.85, 4: 3.2, 8: 4.9, 16: 5.94}[case["max_aniso"]]
        b, f, touched = _lookup_work(case, case["n"], "loguniform")
        return {"bytes": b + 16 * case["n"], "flops": f * probes}
    if kind == "frame":
        px, he = case["width"] * case["height"], _halfedges(case)
        q = 32 if case["max_aniso"] else 16
        # the mesh once, a query written and read and a result per pixel,
        # about two texel rows a pixel
        b = px * (2 * q + 4 * C) + he["H"] * 24 + px * 4 * C * ELEM[case["dtype"]]
        return {"bytes": b, "flops": he["H"] * 100 + px * 200}
    K = (case["tess"] + 1) * (case["tess"] + 2) // 2
    he = _halfedges(case)
    points = he["H"] * K
    texel = C * ELEM[case["dtype"]]
    return {"bytes": points * 12 + he["H"] * 28 + min(_asset_bytes(case), points * 4 * texel), "flops": points * 70}


def tolerance(case):
    """FP32 arithmetic on the stored texels everywhere: against exact() the
    lookups are off by 2e-7 to 5e-7, gradients and Adam's moments by up to
    1.8e-6, and sums in another order by as much again."""
    if case["kind"] == "frame":
        # a pixel centre on the border of two triangles may go to either one
        return {"rel": 1e-3, "max": 0.9, "differ": 1e-4}
    if case["kind"] in ("train", "fit"):
        return {"rel": 6e-6, "max": 1e-4}
    return {"rel": 2e-6, "max": 2e-5}


# ------------------------------------------------------------------- exact

class Exact:
    """One asset's topology and texels for the 64-bit evaluation."""

    def __init__(self, case, a):
        he = _halfedges(case)
        self.C, self.H = case["channels"], he["H"]
        code = np.where(np.arange(self.H) < he["twin"], 1, 0)
        g = np.stack([np.arange(self.H), he["next"], he["prev"]], 1)
        self.edge = torch.from_numpy(he["edge"][g]).to(DEV)
        self.flip = torch.from_numpy(code[g]).to(DEV).bool()
        self.n = torch.from_numpy(a["log2n"].astype(np.int64)).to(DEV)
        self.off = torch.from_numpy(a["off"] // ELEM[case["dtype"]]).to(DEV)
        self.scale = a["scales"].double() if case["dtype"] in ("f16", "bf16", "e4m3") else None
        self.unit = 1.0 / 255.0 if case["dtype"] == "u8" else 1.0
        view = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}.get(case["dtype"], torch.uint8)
        self.values = a["pool"].view(view)
        self.codes = None
        if case["dtype"] == "e4m3":
            self.codes = torch.arange(256, dtype=torch.uint8).view(torch.float8_e4m3fn).float().double().to(DEV)

    def texels(self, i):
        """The C decoded channels of the texels at element indices i."""
        x = self.values[i[:, None] + torch.arange(self.C, device=DEV)]
        x = self.codes[x.long()] if self.codes is not None else x.double()
        return x * self.unit

    def taps(self, h, u, v, log2f):
        """(edge, element index, weight) of every tap: three fetches, two
        levels, zero-bordered bilinear; indices outside go to 0 with weight 0."""
        zero = torch.zeros((), dtype=torch.float64, device=DEV)
        for k, (x, y) in enumerate(((u, v), (v, -u), (-v, u))):
            e, flip = self.edge[h, k], self.flip[h, k]
            x, y = torch.where(flip, 1 - x, x), torch.where(flip, 1 - y, y)
            n = self.n[e]
            lam = log2f + n
            low = torch.minimum(lam.clamp(min=0).floor(), n.double())
            two = (lam > 0) & (low < n)
            w1 = torch.where(two, lam - low, zero)
            for level, w in ((low.long(), 1 - w1), (torch.minimum(low.long() + 1, n), w1)):
                N = 1 << (n - level)
                base = self.off[e] + ((1 << (2 * n + 2)) - (1 << (2 * (n - level) + 2))) // 3 * self.C
                i, j = (x * N - 0.5).floor(), (y * N - 0.5).floor()
                a, b = x * N - 0.5 - i, y * N - 0.5 - j
                i, j = i.clamp(-4, 1 << 20).long(), j.clamp(-4, 1 << 20).long()
                for di, dj, wt in ((0, 0, (1 - a) * (1 - b)), (1, 0, a * (1 - b)), (0, 1, (1 - a) * b), (1, 1, a * b)):
                    ok = (i + di >= 0) & (i + di < N) & (j + dj >= 0) & (j + dj < N)
                    at = torch.where(ok, base + ((j + dj) * N + i + di) * self.C, 0)
                    yield e, at, torch.where(ok, w * wt, zero)

    def sums(self, h, u, v, log2f):
        acc = torch.zeros((h.numel(), self.C), dtype=torch.float64, device=DEV)
        W = torch.zeros(h.numel(), dtype=torch.float64, device=DEV)
        for e, at, w in self.taps(h, u, v, log2f):
            acc += (w if self.scale is None else w * self.scale[e])[:, None] * self.texels(at)
            W += w
        return acc, W


def _decode(q):
    """Halfedge, barycentrics clamped onto the triangle and log2 footprint of
    int32 [n, 4] queries (NaN barycentrics for an id below zero)."""
    h = q[:, 0].long()
    f = q.view(torch.float32)
    u, v = f[:, 1].double().clamp(min=0), f[:, 2].double().clamp(min=0)
    over = (u + v).clamp(min=1)
    bad = torch.where(h < 0, math.nan, 0.0)
    return h.clamp(min=0), u / over + bad, v / over + bad, f[:, 3].double().log2()


CHUNK = 1 << 20


def exact_lookup(x, q):
    out = []
    for part in q.split(CHUNK):
        h, u, v, lf = _decode(part)
        bad = torch.isnan(u)
        acc, W = x.sums(h, u.nan_to_num(), v.nan_to_num(), lf)
        out.append(torch.where(bad[:, None], math.nan, acc / W[:, None]))
    return torch.cat(out)


def exact_gradient(x, q, g, pool):
    """Gradient of sum(g * lookup) over the pool's elements."""
    grad = torch.zeros(pool, dtype=torch.float64, device=DEV)
    for part, gp in zip(q.split(CHUNK), g.split(CHUNK)):
        h, u, v, lf = _decode(part)
        W = sum(w for _, _, w in x.taps(h, u, v, lf))
        for _, at, w in x.taps(h, u, v, lf):
            add = gp * (w / W)[:, None]
            for c in range(x.C):
                grad.index_add_(0, at + c, add[:, c])
    return grad


def exact_aniso(x, q, kmax):
    out = []
    for part in q.split(CHUNK):
        f = part.view(torch.float32)
        h, u, v, _ = _decode(part[:, :4].contiguous())
        bad = torch.isnan(u)
        u, v = u.nan_to_num(), v.nan_to_num()
        d = f[:, 4:]
        p2 = torch.stack([d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1], d[:, 2] * d[:, 2] + d[:, 3] * d[:, 3]], 1)
        big, small = p2.max(1).values, p2.min(1).values
        K = torch.where(big == 0, 1.0, (big / small).sqrt().ceil().clamp(1, kmax)).double()
        axis = torch.where((p2[:, 1] > p2[:, 0])[:, None], d[:, 2:], d[:, :2]).double()
        length = p2.max(1).values.double().sqrt()
        axis = axis * torch.where(length > K, K / length, 1.0)[:, None]
        lf = (length / K).log2()
        acc = torch.zeros((h.numel(), x.C), dtype=torch.float64, device=DEV)
        W = torch.zeros(h.numel(), dtype=torch.float64, device=DEV)
        for k in range(int(K.max())):
            on = torch.nonzero(K > k)[:, 0]
            t = ((k + 0.5) / K[on] - 0.5)[:, None] * axis[on]
            a, w = x.sums(h[on], u[on] + t[:, 0], v[on] + t[:, 1], lf[on])
            acc.index_add_(0, on, a)
            W.index_add_(0, on, w)
        out.append(torch.where(bad[:, None], math.nan, acc / W[:, None]))
    return torch.cat(out)


def _corners(case):
    """Each halfedge's intrinsic triangle: v0 = Vert(Next h), v1 = the
    face's mean vertex, v2 = Vert(h)."""
    he = _halfedges(case)
    pos = torch.from_numpy(mesh_faces(case["around"], case["rows"], _closed(case))[3]).to(DEV).double()
    vert = torch.from_numpy(he["vert"]).to(DEV).long()
    nxt, face = torch.from_numpy(he["next"]).to(DEV), torch.from_numpy(he["face"]).to(DEV)
    sizes = torch.from_numpy(he["sizes"]).to(DEV).double()
    mean = torch.zeros((len(he["sizes"]), 3), dtype=torch.float64, device=DEV).index_add_(0, face, pos[vert])
    return pos, vert, nxt, face, [pos[vert[nxt]], (mean / sizes[:, None])[face], pos[vert]]


def exact_displace(case, x):
    pos, vert, nxt, face, (v0, v1, v2) = _corners(case)
    area = torch.linalg.cross(pos[vert], pos[vert[nxt]])
    fn = torch.zeros((int(face[-1]) + 1, 3), dtype=torch.float64, device=DEV).index_add_(0, face, area)
    vn = torch.zeros_like(pos).index_add_(0, vert, fn[face])
    fn, vn = fn / fn.norm(dim=1, keepdim=True), vn / vn.norm(dim=1, keepdim=True)
    T = case["tess"]
    i, j = np.array([(i, j) for i in range(T + 1) for j in range(T + 1 - i)]).T
    u, v = torch.from_numpy(i / T).to(DEV), torch.from_numpy(j / T).to(DEV)
    out = []
    for h in torch.arange(x.H, device=DEV).split(CHUNK // len(i)):
        n, k = h.numel(), len(i)
        hh, uu, vv = h.repeat_interleave(k), u.repeat(n), v.repeat(n)
        acc, W = x.sums(hh, uu, vv, torch.full_like(uu, -math.inf))
        d = (acc / W[:, None])[:, case["channel"]]
        uu, vv = uu[:, None], vv[:, None]
        ww = 1 - uu - vv
        N = uu * vn[vert[hh]] + vv * vn[vert[nxt[hh]]] + ww * fn[face[hh]]
        p = uu * v2[hh] + vv * v0[hh] + ww * v1[hh]
        out.append((p + 0.01 * d[:, None] * N / N.norm(dim=1, keepdim=True)).view(n, k, 3))
    return torch.cat(out)


def exact_frame(case, x):
    """The nearest triangle at every pixel centre (ties to the smaller
    halfedge), its barycentrics there, one pixel right and one pixel down,
    and the image of the queries they make."""
    tri = torch.stack(_corners(case)[4], 1)
    Wd, Ht = case["width"], case["height"]
    m = torch.from_numpy(view_projection(case)).to(DEV).double()
    clip = torch.cat([tri, torch.ones_like(tri[..., :1])], -1) @ m.T
    w = clip[..., 3]
    X = (clip[..., 0] / w * 0.5 + 0.5) * Wd
    Y = (0.5 - clip[..., 1] / w * 0.5) * Ht
    Z = clip[..., 2] / w

    def bary(h, px, py):
        xx, yy = X[h], Y[h]
        dx, dy = px - xx[:, 2], py - yy[:, 2]
        a, b = yy[:, 1] - yy[:, 2], xx[:, 2] - xx[:, 1]
        den = a * (xx[:, 0] - xx[:, 2]) + b * (yy[:, 0] - yy[:, 2])
        l0 = (a * dx + b * dy) / den
        l1 = ((yy[:, 2] - yy[:, 0]) * dx + (xx[:, 0] - xx[:, 2]) * dy) / den
        return l0, l1, 1 - l0 - l1

    x0, x1 = (X.amin(1) - 0.5).ceil().clamp(min=0), (X.amax(1) - 0.5).floor().clamp(max=Wd - 1)
    y0, y1 = (Y.amin(1) - 0.5).ceil().clamp(min=0), (Y.amax(1) - 0.5).floor().clamp(max=Ht - 1)
    nx = ((x1 - x0 + 1).clamp(min=0) * (w > 0).all(1)).long()
    count = nx * (y1 - y0 + 1).clamp(min=0).long()
    hs, pix, zs = [], [], []
    for h in torch.arange(x.H, device=DEV).split(1 << 15):
        c = count[h]
        hh = h.repeat_interleave(c)
        k = torch.arange(hh.numel(), device=DEV) - (c.cumsum(0) - c).repeat_interleave(c)
        px, py = x0[hh] + k % nx[hh].clamp(min=1), y0[hh] + k // nx[hh].clamp(min=1)
        l = torch.stack(bary(hh, px + 0.5, py + 0.5), 1)
        z = (l * Z[hh]).sum(1)
        ok = (l >= 0).all(1) & (z.abs() <= 1)
        hs.append(hh[ok])
        pix.append((py * Wd + px).long()[ok])
        zs.append(z[ok])
    hs, pix, zs = torch.cat(hs), torch.cat(pix), torch.cat(zs)
    near = torch.full((Wd * Ht,), math.inf, dtype=torch.float64, device=DEV).scatter_reduce_(0, pix, zs, "amin")
    first = zs == near[pix]
    seen = torch.full((Wd * Ht,), x.H, device=DEV).scatter_reduce_(0, pix[first], hs[first], "amin")
    at = torch.nonzero(seen < x.H)[:, 0]
    h = seen[at]
    px, py = (at % Wd) + 0.5, (at // Wd) + 0.5
    ws = w[h]

    def uv(ox, oy):
        l = torch.stack(bary(h, px + ox, py + oy), 1) / ws
        return torch.stack([l[:, 2], l[:, 0]], 1) / l.sum(1, keepdim=True)

    uv0 = uv(0, 0)
    d = torch.cat([uv(1, 0) - uv0, uv(0, 1) - uv0], 1)
    fp = torch.maximum(d[:, :2].norm(dim=1), d[:, 2:].norm(dim=1))
    q = torch.zeros((Wd * Ht, 8), dtype=torch.float32, device=DEV)
    q[at] = torch.cat([torch.zeros_like(uv0[:, :1]), uv0, fp[:, None], d], 1).float()
    qi = q.view(torch.int32)
    qi[:, 0] = -1
    qi[at, 0] = h.int()
    full = torch.zeros((Wd * Ht, 7), dtype=torch.float64, device=DEV)
    full[at] = torch.cat([uv0, fp[:, None], d], 1)
    if case["max_aniso"]:
        return {"h": None, "uv": full[:, :2], "derivatives": full[:, 3:],
                "image": exact_aniso(x, qi, case["max_aniso"])}
    return {"h": None, "uv": full[:, :2], "footprint": full[:, 2],
            "image": exact_lookup(x, qi[:, :4].contiguous())}


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        assets = [Exact(c, asset_inputs(c, seed, _halfedges(c)["E"], 2 + k)) for k, c in enumerate(SERVED)]
        return [exact_lookup(assets[a], q) for (a, _), q in zip(served_requests(case), served_queries(case, seed))]
    a = asset_inputs(case, seed, _halfedges(case)["E"])
    x = Exact(case, a)
    g = _generator(seed, 1)
    if kind == "frame":
        return exact_frame(case, x)
    if kind == "displace":
        return exact_displace(case, x)
    if kind == "aniso":
        return exact_aniso(x, random_queries_aniso(x.H, case["n"], g), case["max_aniso"])
    q = random_queries(x.H, case["n"], case["footprint"], g)
    out = exact_lookup(x, q)
    if kind in ("lookup", "host"):
        return out.cpu() if kind == "host" else out
    diff = out - torch.rand((case["n"], case["channels"]), device=DEV, generator=g).double()
    texels = a["pool"].view(torch.float32)
    grad = exact_gradient(x, q, (2.0 / diff.numel()) * diff, texels.numel())
    loss = diff.square().mean()
    if kind == "train":
        return {"out": out, "loss": loss, "grad": grad}
    b1, b2, eps, lr = (float(np.float32(b)) for b in (0.9, 0.999, 1e-8, 0.05))   # as the entry point takes them
    return {"out": out, "loss": loss, "texels": texels.double() - lr * grad / (grad.abs() + eps),
            "m": (1 - b1) * grad, "v": (1 - b2) * grad * grad}
