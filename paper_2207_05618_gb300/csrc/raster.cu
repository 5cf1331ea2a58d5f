// The rendering side of Htex (paper Sections 3.1, 4.4) as CUDA kernels:
// Alg. 1 (the intrinsic triangle of each halfedge, evaluated once when the
// geometry is made) and rendering the intrinsic triangulation into a
// per-pixel query buffer (halfedge, perspective-correct barycentrics,
// footprint).
//
// Rasterisation: a warp projects 32 intrinsic triangles (one per lane), then
// tests the pixel centres of all their bounding boxes together, 32 at a
// time, so that a warp's work is the sum of its boxes and not its largest
// one; a triangle covers the pixel centres inside it (barycentrics >= 0,
// depth z/w in [-1, 1]) and the smallest 64-bit key (ordered depth << 32 |
// halfedge) is kept per pixel with atomicMin, so ties go to the smaller
// halfedge id.  A resolve pass turns each pixel's key into a query from the
// projected triangle, which the first pass left in scratch or (meshes fine
// beside the frame) is projected again: barycentrics at the pixel centre
// corrected for perspective, and the footprint max(|d(u,v)/dx|, |d(u,v)/dy|)
// from the same triangle's barycentrics one pixel right and one pixel down.
// Triangles with a vertex behind the camera (w <= 0) are not drawn.
//
// Bound by instruction issue.  522,370 halfedges at 1920x1080 (a thread a
// triangle, then the projection again per pixel: 52 and 38 us): covering
// 45 us, resolving 23 us; the covering with 5 blocks per SM (48 registers and
// 24 bytes of spills; 4 or 6: 3% of the frame slower; one block per 256
// triangles, smaller blocks: within 1%).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include <type_traits>

#include <cuda_runtime.h>

#include "geometry.h"
#include "htex_internal.h"
#include "packed.cuh"

namespace {

using namespace htex;   // packed FP32 pairs

constexpr int kThreads = 256;

__device__ __forceinline__ float3 ld3(const float* p, int32_t i) {
    return make_float3(p[3 * i], p[3 * i + 1], p[3 * i + 2]);
}

// What Alg. 1 reads; needed only while the geometry is made.
struct Operators {
    int32_t H;
    const int32_t* next;
    const int32_t* vert;
    const int32_t* face;
    const float* pos;   // [V][3]
};

// Alg. 1: v0 = Vert(Next h), v1 = the mean of the face's vertices walking
// the Next cycle from h, v2 = Vert(h).
__global__ void k_alg1(Operators g, float4* tri) {
    for (int32_t h = blockIdx.x * blockDim.x + threadIdx.x; h < g.H; h += gridDim.x * blockDim.x) {
        const int32_t nx = g.next[h];
        const float3 v2 = ld3(g.pos, g.vert[h]);
        const float3 v0 = ld3(g.pos, g.vert[nx]);
        float3 c = v2;
        int n = 1;
        for (int32_t k = nx; k != h && n <= g.H; k = g.next[k]) {
            const float3 p = ld3(g.pos, g.vert[k]);
            c.x += p.x;
            c.y += p.y;
            c.z += p.z;
            ++n;
        }
        const float inv = 1.0f / float(n);
        float4* t = tri + 3 * int64_t(h);
        t[0] = make_float4(v0.x, v0.y, v0.z, __int_as_float(g.vert[nx]));
        t[1] = make_float4(c.x * inv, c.y * inv, c.z * inv, __int_as_float(g.face[h]));
        t[2] = make_float4(v2.x, v2.y, v2.z, __int_as_float(g.vert[h]));
    }
}

// The intrinsic triangle of halfedge h.
__device__ __forceinline__ void triangle(const htex_geometry& g, int32_t h, float3& v0, float3& v1, float3& v2) {
    const float4* t = g.d_tri + 3 * int64_t(h);
    const float4 a = __ldg(t), b = __ldg(t + 1), c = __ldg(t + 2);
    v0 = make_float3(a.x, a.y, a.z);
    v1 = make_float3(b.x, b.y, b.z);
    v2 = make_float3(c.x, c.y, c.z);
}

// The corners without the ids: nine floats of the twelve, each read and
// written by the thread of its place in the output, so that a warp reads and
// writes whole lines.  Bound by its 84 bytes per halfedge: 4.7M halfedges
// 68 us, 5.8 TB/s (a thread per halfedge, 48 and 36 bytes from the next
// one's: 189 us).
__global__ void __launch_bounds__(kThreads) k_triangles(htex_geometry g, float* out) {
    for (int64_t h0 = int64_t(blockIdx.x) * kThreads; h0 < g.H; h0 += int64_t(gridDim.x) * kThreads) {
        const float* const src = reinterpret_cast<const float*>(g.d_tri + 3 * h0);
        float* const dst = out + 9 * h0;
        const unsigned n = 9u * unsigned(min(int64_t(kThreads), g.H - h0));
        float v[9];
#pragma unroll
        for (unsigned k = 0; k < 9; ++k) {
            const unsigned i = k * kThreads + threadIdx.x;
            if (i < n) v[k] = __ldg(src + 4 * (i / 3) + i % 3);
        }
#pragma unroll
        for (unsigned k = 0; k < 9; ++k) {
            const unsigned i = k * kThreads + threadIdx.x;
            if (i < n) dst[i] = v[k];
        }
    }
}

struct Camera {
    float m[16];   // row-major view-projection: clip = m * [p, 1]
    int32_t W, Ht;
};

struct Screen {
    float x[3], y[3], z[3], w[3];   // screen position, NDC depth and clip w of v0, v1, v2
    float den;
};

__device__ __forceinline__ bool project(const Camera& cam, const float3 (&v)[3], Screen& s) {
    for (int k = 0; k < 3; ++k) {
        const float* m = cam.m;
        const float cx = m[0] * v[k].x + m[1] * v[k].y + m[2] * v[k].z + m[3];
        const float cy = m[4] * v[k].x + m[5] * v[k].y + m[6] * v[k].z + m[7];
        const float cz = m[8] * v[k].x + m[9] * v[k].y + m[10] * v[k].z + m[11];
        const float cw = m[12] * v[k].x + m[13] * v[k].y + m[14] * v[k].z + m[15];
        if (!(cw > 0.0f)) return false;
        s.w[k] = cw;
        s.x[k] = (cx / cw * 0.5f + 0.5f) * float(cam.W);
        s.y[k] = (0.5f - cy / cw * 0.5f) * float(cam.Ht);
        s.z[k] = cz / cw;
    }
    s.den = (s.y[1] - s.y[2]) * (s.x[0] - s.x[2]) + (s.x[2] - s.x[1]) * (s.y[0] - s.y[2]);
    return s.den != 0.0f;
}

// Screen-space barycentrics of (px, py) with respect to (v0, v1, v2).
__device__ __forceinline__ void screen_bary(const Screen& s, float px, float py, float& l0, float& l1, float& l2) {
    l0 = ((s.y[1] - s.y[2]) * (px - s.x[2]) + (s.x[2] - s.x[1]) * (py - s.y[2])) / s.den;
    l1 = ((s.y[2] - s.y[0]) * (px - s.x[2]) + (s.x[0] - s.x[2]) * (py - s.y[2])) / s.den;
    l2 = 1.0f - l0 - l1;
}

// Perspective-correct (u, v): u weighs v2 = Vert(h), v weighs v0 = Vert(Next h).
__device__ __forceinline__ void uv_at(const Screen& s, float px, float py, float& u, float& v) {
    float l0, l1, l2;
    screen_bary(s, px, py, l0, l1, l2);
    const float a = l0 / s.w[0], b = l1 / s.w[1], c = l2 / s.w[2];
    const float inv = 1.0f / (a + b + c);
    u = c * inv;
    v = a * inv;
}

__device__ __forceinline__ uint32_t ordered(float z) {
    const uint32_t b = __float_as_uint(z);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__global__ void k_clear(ulonglong2* vis, int64_t pairs) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < pairs; i += int64_t(gridDim.x) * blockDim.x)
        vis[i] = make_ulonglong2(~0ull, ~0ull);
}

// A projected triangle in scratch, 64 bytes: (x, y, z, w) of each vertex,
// then den.
__device__ __forceinline__ void store_screen(float4* at, const Screen& s) {
#pragma unroll
    for (int k = 0; k < 3; ++k) at[k] = make_float4(s.x[k], s.y[k], s.z[k], s.w[k]);
    at[3] = make_float4(s.den, 0.0f, 0.0f, 0.0f);
}

__device__ __forceinline__ Screen load_screen(const float4* at) {
    Screen s;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float4 v = __ldg(at + k);
        s.x[k] = v.x;
        s.y[k] = v.y;
        s.z[k] = v.z;
        s.w[k] = v.w;
    }
    s.den = __ldg(&at[3].x);
    return s;
}

// A triangle being covered, 16-byte words in shared memory (read by lanes
// of which most hold the same triangle): the coefficients of screen_bary's
// two numerators as pairs, minus the vertex they are taken from, den and the
// bound below which a numerator's quotient is certainly negative, depths,
// and the bounding box.
struct __align__(16) RasterTriangle {
    float e0, e1, f0, f1;       // n0 = e0 dx + f0 dy, n1 = e1 dx + f1 dy
    float mx2, my2, den, below;
    float z0, z1, z2;
    int32_t h;
    int32_t bx, by, bw, first;  // corner, width, first item
    float inv_bw, pad[3];
};

// Boxes of at most this many pixels are pooled over the warp; a larger one
// is covered by the whole warp by itself.
constexpr int kPooledPixels = 1024;

__device__ __forceinline__ void cover(const RasterTriangle& t, int qx, int qy, int width, unsigned long long* vis) {
    const int x = t.bx + qx, y = t.by + qy;
    const uint64_t d = add2(pack2(x + 0.5f, y + 0.5f), pack2(t.mx2, t.my2));
    float dx, dy, n0, n1;
    unpack2(d, dx, dy);
    unpack2(add2(mul2(pack2(t.e0, t.e1), pack2(dx, dx)), mul2(pack2(t.f0, t.f1), pack2(dy, dy))), n0, n1);
    // outside for certain (the quotient negative and not rounded to -0): no division
    const float den = t.den;
    const uint32_t sign = __float_as_uint(den) & 0x80000000u;
    if (__uint_as_float(__float_as_uint(n0) ^ sign) < t.below || __uint_as_float(__float_as_uint(n1) ^ sign) < t.below)
        return;
    const float l0 = n0 / den, l1 = n1 / den, l2 = 1.0f - l0 - l1;
    if (!(l0 >= 0.0f && l1 >= 0.0f && l2 >= 0.0f)) return;
    const float z = l0 * t.z0 + l1 * t.z1 + l2 * t.z2;
    if (!(z >= -1.0f && z <= 1.0f)) return;
    const unsigned long long key = (static_cast<unsigned long long>(ordered(z)) << 32) | uint32_t(t.h);
    atomicMin(vis + int64_t(y) * width + x, key);
}

// KEPT: the projected triangles go to 'screens'.
template <bool KEPT>
__global__ void __launch_bounds__(kThreads, 5) k_raster(htex_geometry g, Camera cam, unsigned long long* vis,
                                                     float4* screens) {
    __shared__ RasterTriangle tris[kThreads / 32][32];
    const unsigned lane = threadIdx.x & 31u;
    RasterTriangle* const w = tris[threadIdx.x >> 5];
    const int64_t step = int64_t(gridDim.x) * kThreads;
    for (int64_t base = int64_t(blockIdx.x) * kThreads + (threadIdx.x & ~31u); base < g.H; base += step) {
        const int64_t h = base + lane;
        Screen s;
        int x0 = 0, y0 = 0, nx = 0, ny = 0;
        if (h < g.H) {
            float3 v[3];
            triangle(g, int32_t(h), v[0], v[1], v[2]);
            if (project(cam, v, s)) {
                const float xmin = fminf(s.x[0], fminf(s.x[1], s.x[2])), xmax = fmaxf(s.x[0], fmaxf(s.x[1], s.x[2]));
                const float ymin = fminf(s.y[0], fminf(s.y[1], s.y[2])), ymax = fmaxf(s.y[0], fmaxf(s.y[1], s.y[2]));
                x0 = max(0, int(ceilf(xmin - 0.5f)));
                y0 = max(0, int(ceilf(ymin - 0.5f)));
                const int x1 = min(cam.W - 1, int(floorf(xmax - 0.5f)));
                const int y1 = min(cam.Ht - 1, int(floorf(ymax - 0.5f)));
                nx = x1 >= x0 ? x1 - x0 + 1 : 0;
                ny = y1 >= y0 ? y1 - y0 + 1 : 0;
            }
        }
        const int pixels = nx * ny;   // of the frame, which has fewer than 2^31
        if (KEPT && pixels > 0) store_screen(screens + 4 * h, s);
        const auto put = [&](unsigned t, int first) {
            // below: 2^-140 |den|, so that the quotient is at least 2^-140
            w[t] = RasterTriangle{s.y[1] - s.y[2], s.y[2] - s.y[0], s.x[2] - s.x[1], s.x[0] - s.x[2],
                                  -s.x[2], -s.y[2], s.den, -fabsf(s.den) * __int_as_float(1 << 9),
                                  s.z[0], s.z[1], s.z[2], int32_t(h), x0, y0, nx, first, 1.0f / float(nx), {}};
        };

        // small boxes: the triangles with pixels packed to the front, their
        // pixels numbered on
        const int mine = pixels <= kPooledPixels ? pixels : 0;
        const unsigned some = __ballot_sync(0xffffffffu, mine > 0);
        int incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= unsigned(d)) incl += o;
        }
        const int P = __shfl_sync(0xffffffffu, incl, 31), start = incl - mine;
        if (mine > 0) put(__popc(some & ((1u << lane) - 1u)), start);
        __syncwarp();
        unsigned begun = 0;   // triangles that start before these 32 pixels
        for (int R = 0; R < P; R += 32) {
            const unsigned starts = __reduce_or_sync(0xffffffffu,
                                                     mine > 0 && unsigned(start - R) < 32u ? 1u << (start - R) : 0u);
            const unsigned t = begun + __popc(starts & (0xffffffffu >> (31u - lane))) - 1u;
            begun += __popc(starts);
            const int j = R + int(lane);
            if (j < P) {
                // the box's row by one product: exact, the quotient is below 1024 and at least 2^-11 from an integer
                const int r = j - w[t].first;
                const int qy = int((float(r) + 0.5f) * w[t].inv_bw);
                cover(w[t], r - qy * w[t].bw, qy, cam.W, vis);
            }
        }
        __syncwarp();
        for (unsigned big = __ballot_sync(0xffffffffu, pixels > kPooledPixels); big; big &= big - 1u) {
            const unsigned owner = unsigned(__ffs(int(big))) - 1u;
            if (lane == owner) put(0, 0);
            __syncwarp();
            const unsigned all = unsigned(__shfl_sync(0xffffffffu, pixels, int(owner)));
            const unsigned width = unsigned(w[0].bw);
            for (unsigned r = lane; r < all; r += 32) cover(w[0], int(r % width), int(r / width), cam.W, vis);
            __syncwarp();
        }
    }
}

// Per pixel: the visible triangle's perspective-correct barycentrics at the
// pixel centre and at the centres one pixel right and one pixel down; Q is
// htex_query (footprint = the longer of the two differences) or
// htex_query_aniso (the two differences as the screen derivatives).
// KEPT: the projected triangles are in 'screens'; otherwise projected again.
template <class Q, bool KEPT>
__global__ void k_resolve(htex_geometry g, Camera cam, const unsigned long long* vis, const float4* screens, Q* q,
                          float* depth) {
    const uint32_t n = uint32_t(cam.W) * uint32_t(cam.Ht);   // below 2^31
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const unsigned long long key = vis[i];
        int32_t h = -1;
        float u = 0.0f, vv = 0.0f, d[4] = {};   // differences, or the footprint in d[0]
        float zd = __int_as_float(0x7fc00000);
        if (key != ~0ull) {
            h = int32_t(uint32_t(key & 0xffffffffull));
            Screen s;
            if constexpr (KEPT) {
                s = load_screen(screens + 4 * int64_t(h));
            } else {
                float3 v[3];
                triangle(g, h, v[0], v[1], v[2]);
                project(cam, v, s);
            }
            const uint32_t row = i / uint32_t(cam.W);
            const float px = float(i - row * uint32_t(cam.W)) + 0.5f, py = float(row) + 0.5f;
            float ux, vx, uy, vy;
            uv_at(s, px, py, u, vv);
            uv_at(s, px + 1.0f, py, ux, vx);
            uv_at(s, px, py + 1.0f, uy, vy);
            d[0] = ux - u;
            d[1] = vx - vv;
            d[2] = uy - u;
            d[3] = vy - vv;
            if constexpr (std::is_same<Q, htex_query>::value) d[0] = fmaxf(hypotf(d[0], d[1]), hypotf(d[2], d[3]));
            float l0, l1, l2;
            screen_bary(s, px, py, l0, l1, l2);
            zd = l0 * s.z[0] + l1 * s.z[1] + l2 * s.z[2];
        }
        // 16 bytes a store (the entry point checks the alignment): word by word
        // every store of a warp touches all of its lines.  2 megapixels of 57k
        // halfedges, the whole call: anisotropic queries 101 -> 70 us, 8
        // megapixels 343 -> 233
        float4* const to = reinterpret_cast<float4*>(q + i);
        if constexpr (std::is_same<Q, htex_query>::value) {
            to[0] = make_float4(__int_as_float(h), u, vv, d[0]);
        } else {
            to[0] = make_float4(__int_as_float(h), u, vv, 0.0f);
            to[1] = make_float4(d[0], d[1], d[2], d[3]);
        }
        if (depth) depth[i] = zd;
    }
}

int grid_for(int64_t n) {
    static std::atomic<int> known[Occupancy::kDevices];
    int dev = 0;
    cudaGetDevice(&dev);
    const bool in = dev >= 0 && dev < Occupancy::kDevices;
    int sms = in ? known[dev].load(std::memory_order_relaxed) : 0;
    if (sms == 0) {
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 148;
        else if (in) known[dev].store(sms, std::memory_order_relaxed);
    }
    return int(std::min<int64_t>((n + kThreads - 1) / kThreads, int64_t(sms) * 8));
}

void free_geometry(htex_geometry* g) {
    if (!g) return;
    cudaFree(g->d_tri);
    cudaFree(g->d_vn);
    cudaFree(g->d_fn);
    delete g;
}

cudaMemPool_t work_pool(int device) {
    static std::mutex mu;
    static cudaMemPool_t pools[64] = {};
    std::lock_guard<std::mutex> lk(mu);
    if (device < 0 || device >= 64) return nullptr;
    if (!pools[device]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = device;
        if (cudaMemPoolCreate(&pools[device], &props) != cudaSuccess) return nullptr;
        uint64_t keep = ~uint64_t(0);
        cudaMemPoolSetAttribute(pools[device], cudaMemPoolAttrReleaseThreshold, &keep);
    }
    return pools[device];
}

}  // namespace

extern "C" htex_status htex_geometry_create(const htex_mesh* m, const float* positions, htex_stream stream,
                                            htex_geometry** out) {
    if (!m || !positions || !out) return HTEX_ERR_INVALID_ARG;
    *out = nullptr;
    const int32_t H = m->H, V = m->V, F = m->F;
    std::vector<float> vn(size_t(V) * 3), fn(size_t(F) * 3);
    try {
        // normals of the input mesh: per face, its area vector (Newell's
        // formula); per vertex, the normalised sum of its faces' vectors
        std::vector<double> fa(size_t(F) * 3, 0.0), va(size_t(V) * 3, 0.0);
        for (int32_t h = 0; h < H; ++h) {
            const float* a = positions + 3 * size_t(m->vert[h]);
            const float* b = positions + 3 * size_t(m->vert[m->next[h]]);
            double* f = &fa[3 * size_t(m->face[h])];
            f[0] += 0.5 * (double(a[1]) * b[2] - double(a[2]) * b[1]);
            f[1] += 0.5 * (double(a[2]) * b[0] - double(a[0]) * b[2]);
            f[2] += 0.5 * (double(a[0]) * b[1] - double(a[1]) * b[0]);
        }
        for (int32_t h = 0; h < H; ++h)
            for (int k = 0; k < 3; ++k) va[3 * size_t(m->vert[h]) + k] += fa[3 * size_t(m->face[h]) + k];
        auto unit = [](const double* x, float* y) {
            const double l = std::sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]);
            for (int k = 0; k < 3; ++k) y[k] = float(l > 0 ? x[k] / l : 0.0);
        };
        for (int32_t i = 0; i < V; ++i) unit(&va[3 * size_t(i)], &vn[3 * size_t(i)]);
        for (int32_t i = 0; i < F; ++i) unit(&fa[3 * size_t(i)], &fn[3 * size_t(i)]);
    } catch (const std::bad_alloc&) {
        return HTEX_ERR_OUT_OF_MEMORY;
    }
    htex_geometry* g = new (std::nothrow) htex_geometry;
    if (!g) return HTEX_ERR_OUT_OF_MEMORY;
    g->H = H;
    g->V = V;
    g->F = F;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const size_t hb = sizeof(int32_t) * size_t(H), vb = sizeof(float) * 3 * size_t(V);
    int32_t *next = nullptr, *vert = nullptr, *face = nullptr;
    float* pos = nullptr;
    bool ok = cudaMalloc(&next, hb) == cudaSuccess && cudaMalloc(&vert, hb) == cudaSuccess &&
              cudaMalloc(&face, hb) == cudaSuccess && cudaMalloc(&pos, vb) == cudaSuccess &&
              cudaMalloc(&g->d_tri, sizeof(float4) * 3 * size_t(H)) == cudaSuccess &&
              cudaMalloc(&g->d_vn, vb) == cudaSuccess &&
              cudaMalloc(&g->d_fn, sizeof(float) * 3 * size_t(F)) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(next, m->next.data(), hb, cudaMemcpyHostToDevice, s) == cudaSuccess &&
         cudaMemcpyAsync(vert, m->vert.data(), hb, cudaMemcpyHostToDevice, s) == cudaSuccess &&
         cudaMemcpyAsync(face, m->face.data(), hb, cudaMemcpyHostToDevice, s) == cudaSuccess &&
         cudaMemcpyAsync(pos, positions, vb, cudaMemcpyHostToDevice, s) == cudaSuccess &&
         cudaMemcpyAsync(g->d_vn, vn.data(), vb, cudaMemcpyHostToDevice, s) == cudaSuccess &&
         cudaMemcpyAsync(g->d_fn, fn.data(), sizeof(float) * 3 * size_t(F), cudaMemcpyHostToDevice, s) == cudaSuccess;
    if (ok) k_alg1<<<grid_for(H), kThreads, 0, s>>>(Operators{H, next, vert, face, pos}, g->d_tri);
    ok = ok && cudaGetLastError() == cudaSuccess && cudaStreamSynchronize(s) == cudaSuccess;
    cudaFree(next);
    cudaFree(vert);
    cudaFree(face);
    cudaFree(pos);
    if (!ok) {
        cudaGetLastError();
        free_geometry(g);
        return HTEX_ERR_CUDA;
    }
    *out = g;
    return HTEX_OK;
}

extern "C" void htex_geometry_destroy(htex_geometry* g) { free_geometry(g); }

extern "C" htex_status htex_triangle_vertices(const htex_geometry* g, float* out, htex_stream stream) {
    if (!g || !out) return HTEX_ERR_INVALID_ARG;
    k_triangles<<<grid_for(g->H), kThreads, 0, reinterpret_cast<cudaStream_t>(stream)>>>(*g, out);
    return cudaGetLastError() == cudaSuccess ? HTEX_OK : HTEX_ERR_CUDA;
}

namespace {

template <class Q>
htex_status rasterize(const htex_geometry* g, const float* view_proj, int32_t width, int32_t height, Q* queries,
                      float* depth, htex_stream stream) {
    if (!g || !view_proj || !queries || width <= 0 || height <= 0) return HTEX_ERR_INVALID_ARG;
    if (int64_t(width) * height >= (int64_t(1) << 31)) return HTEX_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(queries) & 15u) != 0) return HTEX_ERR_INVALID_ARG;
    Camera cam;
    std::memcpy(cam.m, view_proj, sizeof(cam.m));
    cam.W = width;
    cam.Ht = height;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int64_t n = int64_t(width) * height;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return HTEX_ERR_CUDA;
    cudaMemPool_t pool = work_pool(dev);
    if (!pool) return HTEX_ERR_CUDA;
    // The pixels' keys, then the projected triangles where they are kept: for
    // meshes of at most as many halfedges as the frame has pixels, or 2^18 (so
    // that this scratch stays within 64 bytes a pixel or 16 MiB), and while
    // there is memory for them.  Kept / projected again, halfedges per pixel
    // 0.06: 218 / 238 us, 0.25: 68 / 74, 0.57: 42 / 45 and 69 / 66, 1.3: 48 /
    // 45, 2.2: 129 / 127; 14,400 pixels of 57k halfedges 14.4 / 16.4.
    const size_t vis_b = (size_t(n) * 8 + 63) & ~size_t(63);
    void* vis = nullptr;
    const auto allocate = [&](size_t bytes) {
        if (cudaMallocFromPoolAsync(&vis, bytes, pool, s) == cudaSuccess) return true;
        cudaGetLastError();
        return false;
    };
    const bool kept = g->H <= std::max<int64_t>(n, int64_t(1) << 18) && allocate(vis_b + size_t(g->H) * 64);
    if (!kept && !allocate(vis_b)) return HTEX_ERR_OUT_OF_MEMORY;
    auto* v = static_cast<unsigned long long*>(vis);
    auto* screens = kept ? reinterpret_cast<float4*>(static_cast<uint8_t*>(vis) + vis_b) : nullptr;
    k_clear<<<grid_for(int64_t(vis_b / 16)), kThreads, 0, s>>>(static_cast<ulonglong2*>(vis), int64_t(vis_b / 16));
    const auto raster = kept ? k_raster<true> : k_raster<false>;
    const auto resolve = kept ? k_resolve<Q, true> : k_resolve<Q, false>;
    raster<<<grid_for(g->H), kThreads, 0, s>>>(*g, cam, v, screens);
    resolve<<<grid_for(n), kThreads, 0, s>>>(*g, cam, v, screens, queries, depth);
    const bool ok = cudaGetLastError() == cudaSuccess;
    cudaFreeAsync(vis, s);
    return ok ? HTEX_OK : HTEX_ERR_CUDA;
}

}  // namespace

extern "C" htex_status htex_rasterize(const htex_geometry* g, const float* view_proj, int32_t width, int32_t height,
                                      htex_query* queries, float* depth, htex_stream stream) {
    return rasterize(g, view_proj, width, height, queries, depth, stream);
}

extern "C" htex_status htex_rasterize_aniso(const htex_geometry* g, const float* view_proj, int32_t width,
                                            int32_t height, htex_query_aniso* queries, float* depth,
                                            htex_stream stream) {
    return rasterize(g, view_proj, width, height, queries, depth, stream);
}
