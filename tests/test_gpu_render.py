"""GPU parity of the rendering side (htex_triangle_vertices,
htex_rasterize, htex_displace) against the FP64 oracle."""
import numpy as np
import pytest

import htex_synth as syn
import oracle
import paper_2207_05618_gb300 as hx
from paper_2207_05618_gb300 import render

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2207_05618_gb300 import build
    build.build()
    assert torch.cuda.is_available()


def _sphere():
    fs, fv, V, pos = syn.uv_sphere(slices=14, rings=10, seed=5)
    return fs, fv, V, pos


def test_triangle_vertices_match_alg1():
    for fs, fv, V, pos in (_sphere(), syn.cylinder(around=20, rows=6, seed=2)):
        mo = oracle.mesh_from_faces(fs, fv, V)
        g = render.Geometry(hx.Mesh(fs, fv, V), pos)
        got = g.triangle_vertices().cpu().numpy()
        ref = oracle.triangle_vertices(mo, pos.astype(np.float32).astype(np.float64))
        np.testing.assert_allclose(got, ref, atol=2e-6)


@pytest.mark.parametrize("around,rows", [(3, 1), (8, 7), (12, 20), (300, 260)])
def test_triangle_vertices_block_edges(around, rows):
    """Fewer halfedges than a block takes, a few blocks with a part of one,
    and more than one pass of the grid (8 blocks of 256 per SM)."""
    fs, fv, V, pos = syn.cylinder(around=around, rows=rows, seed=around)
    mo = oracle.mesh_from_faces(fs, fv, V)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert mo.H % 256 != 0 and (mo.H > 8 * 256 * sms or around < 300)
    got = render.Geometry(hx.Mesh(fs, fv, V), pos).triangle_vertices().cpu().numpy()
    np.testing.assert_allclose(got, oracle.triangle_vertices(mo, pos.astype(np.float32).astype(np.float64)), atol=2e-6)


@pytest.mark.parametrize("W,H", [(96, 64), (61, 37)])
def test_rasterizer_matches_reference(W, H):
    """Pixels whose nearest triangle is clear (barycentric margin and depth
    gap above float rounding) carry the oracle's halfedge, barycentrics and
    footprint; every other covered pixel names a triangle that covers it
    at the nearest depth up to rounding; empty pixels agree."""
    fs, fv, V, pos = _sphere()
    mo = oracle.mesh_from_faces(fs, fv, V)
    M = syn.perspective(40.0, W / H, 0.3, 10.0) @ syn.look_at([2.3, -1.1, 0.9], [0, 0, 0], [0, 0, 1])
    g = render.Geometry(hx.Mesh(fs, fv, V), pos)
    depth = torch.empty(W * H, dtype=torch.float32, device="cuda")
    q = g.rasterize(M, W, H, depth=depth).cpu().numpy()
    pos32 = pos.astype(np.float32).astype(np.float64)
    hh, u, v, f, dref, margin, gap = oracle.rasterize(mo, pos32, M.astype(np.float32).astype(np.float64), W, H)
    gh = q[:, 0].reshape(H, W)
    gu = q[:, 1].copy().view(np.float32).reshape(H, W)
    gv = q[:, 2].copy().view(np.float32).reshape(H, W)
    gf = q[:, 3].copy().view(np.float32).reshape(H, W)
    clear = (hh >= 0) & (margin > 1e-4) & (gap > 1e-4)
    assert clear.sum() > 0.5 * (hh >= 0).sum() > 0
    np.testing.assert_array_equal(gh[clear], hh[clear])
    np.testing.assert_allclose(gu[clear], u[clear], atol=2e-4)
    np.testing.assert_allclose(gv[clear], v[clear], atol=2e-4)
    np.testing.assert_allclose(gf[clear], f[clear], rtol=2e-3, atol=1e-6)
    np.testing.assert_allclose(depth.cpu().numpy().reshape(H, W)[clear], dref[clear], atol=1e-5)
    # empty pixels: far from every triangle in the reference
    empty = gh < 0
    assert np.all((hh[empty] < 0) | (margin[empty] < 1e-4))
    # the rest: the GPU's triangle covers the pixel (up to rounding)
    tri = oracle.triangle_vertices(mo, pos32)
    for y, x in np.argwhere((gh >= 0) & ~clear):
        k = gh[y, x]
        P = gu[y, x] * tri[k, 2] + gv[y, x] * tri[k, 0] + (1 - gu[y, x] - gv[y, x]) * tri[k, 1]
        c = M @ np.append(P, 1.0)
        assert abs((c[0] / c[3] * 0.5 + 0.5) * W - (x + 0.5)) < 1e-2
        assert abs((0.5 - c[1] / c[3] * 0.5) * H - (y + 0.5)) < 1e-2
        if hh[y, x] >= 0:
            assert c[2] / c[3] <= dref[y, x] + 1e-4


@pytest.mark.parametrize("W,H", [(96, 64), (61, 37)])
def test_anisotropic_rasterizer_matches_reference(W, H):
    """htex_rasterize_aniso: the same halfedges and barycentrics as
    htex_rasterize (bit for bit), and on clear pixels the oracle's screen
    derivatives of the barycentrics; empty pixels carry h = -1."""
    fs, fv, V, pos = _sphere()
    mo = oracle.mesh_from_faces(fs, fv, V)
    M = syn.perspective(40.0, W / H, 0.3, 10.0) @ syn.look_at([2.3, -1.1, 0.9], [0, 0, 0], [0, 0, 1])
    g = render.Geometry(hx.Mesh(fs, fv, V), pos)
    qi = g.rasterize(M, W, H).cpu().numpy()
    qa = g.rasterize_aniso(M, W, H).cpu().numpy()
    np.testing.assert_array_equal(qa[:, :3], qi[:, :3])
    pos32 = pos.astype(np.float32).astype(np.float64)
    r = oracle.rasterize(mo, pos32, M.astype(np.float32).astype(np.float64), W, H, derivatives=True)
    hh, margin, gap = r[0], r[5], r[6]
    clear = (hh >= 0) & (margin > 1e-4) & (gap > 1e-4)
    assert clear.sum() > 0
    for col, ref in zip(range(4, 8), r[7:11]):
        got = qa[:, col].copy().view(np.float32).reshape(H, W)
        np.testing.assert_allclose(got[clear], ref[clear], rtol=2e-3, atol=2e-6)
    empty = qa[:, 0] < 0
    assert np.all(qa[empty][:, 4:] == 0)


def test_frame_pipeline_full_hd():
    """1920x1080 frame of the closed sphere filling the view: every pixel
    inside the silhouette gets a valid query, the lookup returns finite
    values there and NaN outside."""
    fs, fv, V, pos = _sphere()
    mesh = hx.Mesh(fs, fv, V)
    log2n = np.full(mesh.E, 5, np.int32)
    tex = hx.Textures.upload(mesh, log2n, syn.texels_u8(log2n, 4, seed=1), 4, "u8", hx.BUILD_MIPS)
    g = render.Geometry(mesh, pos)
    M = syn.perspective(45.0, 1920 / 1080, 0.3, 10.0) @ syn.look_at([2.2, 0, 0], [0, 0, 0], [0, 0, 1])
    q = g.rasterize(M, 1920, 1080)
    out = hx.lookup(tex, q).cpu().numpy()
    valid = q[:, 0].cpu().numpy() >= 0
    assert 0.2 < valid.mean() < 0.9
    assert np.all(np.isfinite(out[valid])) and np.all(np.isnan(out[~valid]))


def test_displacement_matches_oracle_and_is_crack_free():
    fs, fv, V, pos = syn.uv_sphere(slices=9, rings=7, seed=2)
    mo = oracle.mesh_from_faces(fs, fv, V)
    mesh = hx.Mesh(fs, fv, V)
    log2n = np.full(mesh.E, 3, np.int32)
    flags = hx.BUILD_MIPS | hx.FIX_CORNERS
    tex_np = syn.texels_f32(log2n, 2, 3)
    tl = hx.Textures.upload(mesh, log2n, tex_np, 2, "f32", flags)
    to = oracle.prepare_textures(mo, log2n, tex_np, 2, "f32", flags)
    g = render.Geometry(mesh, pos)
    T = 4
    got = g.displace(tl, T, 0.3, channel=1).cpu().numpy()
    pos32 = pos.astype(np.float32).astype(np.float64)
    ref = oracle.displace(mo, to, pos32, T, 0.3, channel=1)
    np.testing.assert_allclose(got, ref, atol=2e-5)
    P0 = oracle.displace(mo, to, pos32, T, 0.0).reshape(-1, 3)
    key = np.round(P0 * 1e6).astype(np.int64)
    _, inv = np.unique(key, axis=0, return_inverse=True)
    flat = got.reshape(-1, 3)
    for grp in np.unique(inv):
        pts = flat[inv == grp]
        assert np.abs(pts - pts[0]).max() < 2e-5


@pytest.mark.parametrize("dtype,C,channel", [("f32", 3, 2), ("u8", 4, 0), ("u8", 3, 1), ("f16", 1, 0), ("bf16", 2, 1),
                                             ("e4m3", 4, 3)])
@pytest.mark.parametrize("T", [1, 2, 3, 8, 64])
def test_displacement_formats_and_block_edges(dtype, C, channel, T):
    """Mixed resolutions down to 1x1 and every texel format on a mesh so small
    that each block takes one halfedge, of 3 points (T = 1, most of a block
    idle) to 2145 (T = 64, several rounds).  Tolerance: the FP32 lookup's
    1e-5 and the position's few ulp, as above."""
    fs, fv, V, pos = syn.cylinder(around=16, rows=6, seed=4)
    mo = oracle.mesh_from_faces(fs, fv, V)
    mesh = hx.Mesh(fs, fv, V)
    assert mesh.H <= 6 * torch.cuda.get_device_properties(0).multi_processor_count
    log2n = np.random.default_rng(1).integers(0, 6, mesh.E).astype(np.int32)
    flags = hx.BUILD_MIPS | hx.MIRROR_BOUNDARY
    texels = (syn.texels_u8 if dtype == "u8" else syn.texels_f32)(log2n, C, 3)
    tl = hx.Textures.upload(mesh, log2n, texels, C, dtype, flags)
    to = oracle.prepare_textures(mo, log2n, texels, C, dtype, flags)
    got = render.Geometry(mesh, pos).displace(tl, T, 0.3, channel=channel).cpu().numpy()
    pos32 = pos.astype(np.float32).astype(np.float64)
    np.testing.assert_allclose(got, oracle.displace(mo, to, pos32, T, 0.3, channel=channel), atol=2e-5)


@pytest.mark.parametrize("around,rows,T", [(40, 31, 1), (40, 31, 2), (40, 31, 3), (40, 31, 8), (100, 80, 8), (100, 80, 16),
                                           (330, 190, 1), (330, 190, 3)])
@pytest.mark.parametrize("dtype,C,channel", [("f32", 3, 2), ("u8", 4, 1), ("e4m3", 1, 0)])
def test_displacement_several_halfedges_a_block(around, rows, T, dtype, C, channel):
    """Meshes of more than six halfedges per SM, so that a block takes several
    (as the launcher works out: few by the spread over the SMs, by the points
    a block aims at, and the most, one per thread), the last block not full,
    mixed resolutions.  Tolerance as above."""
    fs, fv, V, pos = syn.cylinder(around=around, rows=rows, seed=rows)
    mesh = hx.Mesh(fs, fv, V)
    sms, K = torch.cuda.get_device_properties(0).multi_processor_count, (T + 1) * (T + 2) // 2
    per_block = min(256, max(1, 2048 // K), -(-mesh.H // (6 * sms)))
    assert per_block > 1 and mesh.H % per_block != 0 and (around < 330 or per_block > 200)
    mo = oracle.mesh_from_faces(fs, fv, V)
    log2n = np.random.default_rng(1).integers(0, 3, mesh.E).astype(np.int32)
    texels = (syn.texels_u8 if dtype == "u8" else syn.texels_f32)(log2n, C, 3)
    tl = hx.Textures.upload(mesh, log2n, texels, C, dtype, hx.BUILD_MIPS)
    to = oracle.prepare_textures(mo, log2n, texels, C, dtype, hx.BUILD_MIPS)
    got = render.Geometry(mesh, pos).displace(tl, T, 0.3, channel=channel).cpu().numpy()
    pos32 = pos.astype(np.float32).astype(np.float64)
    np.testing.assert_allclose(got, oracle.displace(mo, to, pos32, T, 0.3, channel=channel), atol=2e-5)


@pytest.mark.parametrize("W,H,eye", [(33, 31, 2.6), (257, 190, 1.9), (640, 3, 2.2), (1, 200, 2.2)])
def test_rasterizer_small_and_large_boxes(W, H, eye):
    """Bounding boxes on both sides of the 1024 pixels that a warp pools
    (a cube's 24 large triangles beside a fine sphere's, one mesh), boxes
    one pixel wide or high, boxes cut by the frame, and a last warp that is
    not full: clear pixels carry the oracle's halfedge and depth."""
    fs, fv, V, pos = syn.cube()
    fs2, fv2, V2, pos2 = syn.uv_sphere(slices=40, rings=30, seed=3)
    fs, fv = np.concatenate([fs, fs2]), np.concatenate([fv, fv2 + V])
    pos = np.concatenate([pos - 0.5, pos2 * 0.3 + [0.9, 0.2, 0.1]])
    mo = oracle.mesh_from_faces(fs, fv, V + V2)
    M = syn.perspective(50.0, W / H, 0.3, 10.0) @ syn.look_at([eye, -0.4, 0.5], [0, 0, 0], [0, 0, 1])
    g = render.Geometry(hx.Mesh(fs, fv, V + V2), pos)
    assert g.H % 32 != 0 or g.H > 256
    depth = torch.empty(W * H, dtype=torch.float32, device="cuda")
    gh = g.rasterize(M, W, H, depth=depth).cpu().numpy()[:, 0].reshape(H, W)
    pos32 = pos.astype(np.float32).astype(np.float64)
    hh, _, _, _, dref, margin, gap = oracle.rasterize(mo, pos32, M.astype(np.float32).astype(np.float64), W, H)
    clear = (hh >= 0) & (margin > 1e-3) & (gap > 1e-4)
    assert clear.sum() > 0
    np.testing.assert_array_equal(gh[clear], hh[clear])
    np.testing.assert_allclose(depth.cpu().numpy().reshape(H, W)[clear], dref[clear], atol=1e-5)
    empty = gh < 0
    assert np.all((hh[empty] < 0) | (margin[empty] < 1e-3))


@pytest.mark.parametrize("aniso", [False, True])
def test_rasterizer_projected_triangles_kept_or_not(aniso):
    """A small mesh (whose projected triangles are kept between the passes),
    and the same mesh with faces behind the camera added until it has more
    than 2^18 halfedges and than the frame has pixels (projected again): the
    same queries and depths, bit for bit."""
    W, H = 96, 64
    fs, fv, V, pos = _sphere()
    M = syn.perspective(40.0, W / H, 0.3, 10.0) @ syn.look_at([2.3, -1.1, 0.9], [0, 0, 0], [0, 0, 1])
    fs2, fv2, V2, pos2 = syn.cylinder(around=300, rows=260, seed=1)
    more = (np.concatenate([fs, fs2]), np.concatenate([fv, fv2 + V]), V + V2,
            np.concatenate([pos, pos2 * 0.2 + [4.6, -2.2, 1.8]]))
    got = []
    for f, v, n, p in ((fs, fv, V, pos), more):
        g = render.Geometry(hx.Mesh(f, v, n), p)
        depth = torch.empty(W * H, dtype=torch.float32, device="cuda")
        q = (g.rasterize_aniso if aniso else g.rasterize)(M, W, H, depth=depth)
        got.append((g.H, q.cpu().numpy(), depth.cpu().numpy().view(np.int32)))
    assert got[0][0] < W * H < 1 << 18 < got[1][0]
    assert (got[0][1][:, 0] >= 0).mean() > 0.1
    np.testing.assert_array_equal(got[0][1], got[1][1])
    np.testing.assert_array_equal(got[0][2], got[1][2])
