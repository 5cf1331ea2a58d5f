// Displacement of a tessellated lattice (paper Section 5.1): every lattice
// vertex of every intrinsic triangle moved along the interpolated normal by
// one channel of the level-0 lookup there.
#include <algorithm>

#include <cuda_runtime.h>

#include "geometry.h"
#include "lookup_core.cuh"

namespace htex {

// One pass: the lookup and the displacement of a point in the same thread.
// A block takes 'per_block' consecutive halfedges; what a triangle's points
// share (corners, normals, the three textures' places) is loaded once into
// shared memory by one thread per triangle, the lattice's (u, v) once per
// block.  Only the wanted channel of a texel is read.  Writes are staged per
// warp so that each store instruction covers whole 128-byte lines.
//
// Bound: the texel lines of level 0 (134 MB) and 12 B per point out.
// Measured on 130,598 halfedges, T = 8, one FP16 channel of 32x32 (5.9M
// points): 75 us a call; three kernels with a query (16 B) and a result
// per point between them, the face walk of Alg. 1 repeated for every
// point, took 236 us.
constexpr int kDisplaceThreads = 256;
// Points a block aims at (its halfedges: at least 1, at most one per thread,
// and few enough to give every SM six blocks): 512 / 1024 / 2048 points 96 /
// 80 / 75 us.
constexpr int kDisplacePoints = 2048;

struct DisplaceParams {
    const float4* tri;
    const float* vn;
    const float* fn;
    int32_t T, K;        // subdivision, points per triangle
    uint32_t magic;      // ceil(2^32 / K): x / K = umulhi(x, magic) for x (K - 1) < 2^32
    int32_t per_block;
    int32_t C, channel;
    float scale;
    float* out;
};

// A triangle's share: corners and normals, and for the own, Next and Prev
// fetch the byte offset of the wanted channel of texel (0, 0) of level 0,
// log2 of the resolution (Alg. 2's reflection in bit 31) and the code factor.
struct DisplaceTriangle {
    float v0[3], v1[3], v2[3], n0[3], n1[3], n2[3];
    uint32_t lo[3], hi[3];
    uint32_t n[3];
    float sc[3];
};

// Lattice point k: i = 0..T, j = 0..T - i in order; the points before row i
// are i (2T + 3 - i) / 2.
__device__ __forceinline__ void lattice_point(int32_t k, int32_t T, float& u, float& v) {
    const int32_t b = 2 * T + 3;
    int32_t i = int32_t((float(b) - sqrtf(float(b * b - 8 * k))) * 0.5f);
    while (i * (b - i) / 2 > k) --i;
    while ((i + 1) * (b - i - 1) / 2 <= k) ++i;
    u = float(i) / float(T);
    v = float(k - i * (b - i) / 2) / float(T);
}

// The wanted channel of one texel, decoded (zero where the weight is zero:
// nothing is read).
template <int DT>
__device__ __forceinline__ float channel_if(const GlobalSpace& pool, bool on, uint64_t o) {
    constexpr int ES = Fmt<DT>::ES;
    if constexpr (ES == 4) return __uint_as_float(pool.ld4_if(on, o));
    else if constexpr (ES == 2) return dec1<DT>(pool.ld2_if(on, o));
    else return dec1<DT>(pool.ld1_if(on, o));
}

__device__ __forceinline__ void copy3(float (&d)[3], const float* s) {
    d[0] = s[0];
    d[1] = s[1];
    d[2] = s[2];
}

template <int DT>
__global__ void __launch_bounds__(kDisplaceThreads) k_displace(Asset<GlobalSpace> A, DisplaceParams p) {
    constexpr int ES = Fmt<DT>::ES;
    extern __shared__ __align__(16) uint8_t smem[];
    float4* lat = reinterpret_cast<float4*>(smem);   // u, v, and the two clamped onto the triangle
    DisplaceTriangle* tri = reinterpret_cast<DisplaceTriangle*>(lat + p.K);
    __shared__ float stage[kDisplaceThreads / 32][96];
    const int32_t h0 = int32_t(blockIdx.x) * p.per_block;
    const int32_t nh = min(p.per_block, A.H - h0);

    for (int32_t k = threadIdx.x; k < p.K; k += kDisplaceThreads) {
        float u, v, uc, vc, f;
        int h;
        lattice_point(k, p.T, u, v);
        decode_query(make_int4(0, __float_as_int(u), __float_as_int(v), 0), 1, h, uc, vc, f);
        lat[k] = make_float4(u, v, uc, vc);
    }
    if (int32_t(threadIdx.x) < nh) {
        const int32_t h = h0 + threadIdx.x;
        DisplaceTriangle& t = tri[threadIdx.x];
        const float4 a = __ldg(p.tri + 3 * int64_t(h)), b = __ldg(p.tri + 3 * int64_t(h) + 1),
                     c = __ldg(p.tri + 3 * int64_t(h) + 2);
        const uint4 rec = A.rec.ld16(uint64_t(h) * 16u);
        t.v0[0] = a.x; t.v0[1] = a.y; t.v0[2] = a.z;
        t.v1[0] = b.x; t.v1[1] = b.y; t.v1[2] = b.z;
        t.v2[0] = c.x; t.v2[1] = c.y; t.v2[2] = c.z;
        copy3(t.n0, p.vn + 3 * int64_t(__float_as_int(a.w)));
        copy3(t.n1, p.fn + 3 * int64_t(__float_as_int(b.w)));
        copy3(t.n2, p.vn + 3 * int64_t(__float_as_int(c.w)));
        const uint32_t code[3] = {rec.x, rec.y, rec.z};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const TexRef r = tex_ref<DT>(A, code[k] & ~kFlipBit);
            const uint64_t o = r.off + uint64_t(p.channel) * ES;
            t.lo[k] = uint32_t(o);
            t.hi[k] = uint32_t(o >> 32);
            t.n[k] = uint32_t(r.n) | (code[k] & kFlipBit);
            t.sc[k] = code_factor<DT>(r);
        }
    }
    __syncthreads();

    const int32_t points = nh * p.K, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t TB = p.C * ES;
    float* const out = p.out + int64_t(h0) * p.K * 3;
    for (int32_t base = warp * 32; base < points; base += kDisplaceThreads) {
        const int32_t x = base + lane;
        if (x < points) {
            const uint32_t q = __umulhi(uint32_t(x), p.magic);
            const DisplaceTriangle& t = tri[q];
            const float4 L = lat[x - int32_t(q) * p.K];
            const float u = L.z, v = L.w;
            // the level-0 lookup: own 2x2 block, then the Next row and the
            // Prev column where the point lies within half a texel of them
            const int32_t n = int32_t(t.n[0] & ~kFlipBit);
            const bool fo = t.n[0] & kFlipBit;
            const OwnPlan o = own_plan<1>(n, 0, fo ? 1.0f - u : u, fo ? 1.0f - v : v, 1.0f);
            const uint64_t ob = (uint64_t(t.hi[0]) << 32 | t.lo[0]) + uint64_t(int64_t(o.o) * TB);
            const uint64_t orow = uint64_t(o.row) * uint32_t(TB);
            float tx[4];
            tx[0] = channel_if<DT>(A.pool, o.w[0] != 0.0f, ob);
            tx[1] = channel_if<DT>(A.pool, o.w[1] != 0.0f, ob + TB);
            tx[2] = channel_if<DT>(A.pool, o.w[2] != 0.0f, ob + orow);
            tx[3] = channel_if<DT>(A.pool, o.w[3] != 0.0f, ob + orow + TB);
            float acc = 0.0f, W = o.ws;
#pragma unroll
            for (int k = 0; k < 4; ++k) acc = fmaf(o.w[k] * t.sc[0], tx[k], acc);
#pragma unroll
            for (int e = 1; e < 3; ++e) {
                const int32_t ne = int32_t(t.n[e] & ~kFlipBit);
                const float dist = e == 1 ? u : v, along = e == 1 ? v : u;
                if (!(across_weight(dist, 1 << ne) > 0.0f)) continue;
                const EdgePlan g = edge_plan<1>(ne, 0, dist, along, (t.n[e] & kFlipBit) != 0, e == 1, 1.0f);
                const uint64_t gb = (uint64_t(t.hi[e]) << 32 | t.lo[e]) + uint64_t(int64_t(g.o) * TB);
                const float a = channel_if<DT>(A.pool, g.w[0] != 0.0f, gb);
                const float b = channel_if<DT>(A.pool, g.w[1] != 0.0f, gb + uint64_t(g.step) * uint32_t(TB));
                acc = fmaf(g.w[0] * t.sc[e], a, acc);
                acc = fmaf(g.w[1] * t.sc[e], b, acc);
                W += g.ws;
            }
            const float d = acc * (__frcp_rn(W) * Fmt<DT>::UNIT);
            const float w = 1.0f - L.x - L.y;
            float N[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) N[c] = L.x * t.n2[c] + L.y * t.n0[c] + w * t.n1[c];
            const float l = rsqrtf(N[0] * N[0] + N[1] * N[1] + N[2] * N[2]);
            const float s = p.scale * d * l;
#pragma unroll
            for (int c = 0; c < 3; ++c)
                stage[warp][3 * lane + c] = L.x * t.v2[c] + L.y * t.v0[c] + w * t.v1[c] + s * N[c];
        }
        __syncwarp();
        const int32_t words = 3 * min(32, points - base);
#pragma unroll
        for (int c = 0; c < 3; ++c)
            if (32 * c + lane < words) __stcs(out + 3 * int64_t(base) + 32 * c + lane, stage[warp][32 * c + lane]);
        __syncwarp();
    }
}

template <int DT>
htex_status launch_displace(const Asset<GlobalSpace>& A, const DisplaceParams& p, cudaStream_t s) {
    // at most 37 KiB with the stage (T = 64: 2145 points, one triangle; T = 1: 256 triangles)
    const size_t smem = size_t(p.K) * sizeof(float4) + size_t(p.per_block) * sizeof(DisplaceTriangle);
    const unsigned grid = unsigned((A.H + p.per_block - 1) / p.per_block);
    k_displace<DT><<<grid, kDisplaceThreads, smem, s>>>(A, p);
    return cudaGetLastError() == cudaSuccess ? HTEX_OK : HTEX_ERR_CUDA;
}

}  // namespace htex

using namespace htex;

extern "C" htex_status htex_displace(const htex_geometry* g, const htex_textures* t, int32_t tess, float scale,
                                     int32_t channel, float* out, htex_stream stream) {
    if (!g || !t || !out || tess < 1 || tess > 64 || channel < 0 || channel >= t->C || t->H != g->H)
        return HTEX_ERR_INVALID_ARG;
    const int32_t K = (tess + 1) * (tess + 2) / 2;
    if (int64_t(g->H) * K >= (int64_t(1) << 31)) return HTEX_ERR_INVALID_ARG;
    const int32_t spread = (g->H + 6 * t->num_sms - 1) / (6 * t->num_sms);
    const int32_t per_block = std::min({kDisplaceThreads, std::max(1, kDisplacePoints / K), std::max(1, spread)});
    const DisplaceParams p{g->d_tri, g->d_vn, g->d_fn, tess, K, uint32_t(((uint64_t(1) << 32) + K - 1) / K),
                           per_block, t->C, channel, scale, out};
    const Asset<GlobalSpace> A = global_asset(t);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    switch (t->dtype) {
    case HTEX_F32: return launch_displace<HTEX_F32>(A, p, s);
    case HTEX_U8: return launch_displace<HTEX_U8>(A, p, s);
    case HTEX_F16: return launch_displace<HTEX_F16>(A, p, s);
    case HTEX_BF16: return launch_displace<HTEX_BF16>(A, p, s);
    case HTEX_E4M3: return launch_displace<HTEX_E4M3>(A, p, s);
    }
    return HTEX_ERR_INVALID_ARG;
}
