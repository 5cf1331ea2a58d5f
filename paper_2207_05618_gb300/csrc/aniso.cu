// Anisotropic filtered lookup and the htex_lookup_aniso entry point.
//
// Section 5.1 renders Htex through the GPU's anisotropic filter, applied to
// each of Alg. 3's three texture fetches; the paper states no formula, so
// this follows one reading, the same as the FP64 oracle's:
//   - the footprint is given by the screen derivatives of the barycentrics,
//     ax = (du/dx, dv/dx) and ay = (du/dy, dv/dy), in quad-uv units;
//   - px2 = |ax|^2, py2 = |ay|^2 (each product and sum rounded to float);
//     the major axis m is ay when py2 > px2, else ax; the probe count K is 1
//     when both are zero, else min(ceil(sqrt(max / min)), kmax), computed
//     with correctly rounded float division and square root so that the
//     integer K is decided exactly as the oracle decides it;
//   - each probe is an isotropic trilinear sample with footprint Pmax / K;
//   - probe k sits at c + m * s * ((k + 1/2) / K - 1/2) with s = min(1,
//     K / Pmax) (the probes never span more than K quad widths);
//   - every probe samples all three fetches at its own (u', v'): own quad
//     at (u', v'), Next's at (v', -u'), Prev's at (-v', u'), each through
//     Alg. 2, with full 2x2 zero-bordered taps (a probe off the triangle can
//     reach any texel of the neighbouring quads); the result is the summed
//     data over the summed normalisation weight.
// Work distribution: a warp takes 32 queries and works through their items
// -- one (fetch, probe) pair whose probe can reach the fetch's quad, both
// levels -- 32 at a time, in the order of query, fetch, probe, so that
// neighbouring lanes read neighbouring texels.  Which probes reach a fetch
// is an interval of probe numbers (the probes lie on a line and the reach is
// a box), so the items are counted without visiting the probes.  Each
// query's constants are computed once by its own lane and kept in shared
// memory; each round's item sums go through shared memory to lanes that add
// them to their query's, one lane per query and channel, in item order: a
// query's result does not depend on which other queries share its warp.
#include <algorithm>

#include <cuda_runtime.h>

#include "lookup_core.cuh"
#include "aniso_launch.h"
#include "aniso_taps.h"

namespace htex {

struct AnisoParams {
    const htex_query_aniso* q;
    int64_t n;
    int32_t kmax;
    float* out;
    int32_t* status;
};

// Shared-memory words of a query: centre u, v, the probe spacing axis (major
// axis times s) mu, mv, K and 1 / (2K); then for each fetch with items
// (own, Next, Prev, those without left out) the byte offset of texel (0, 0)
// of its finer level (low and high half), the packed fields below, the
// coarser level's weight and, for the scaled formats, the code scale.
enum { kU, kV, kMu, kMv, kK, kInv2K, kFetch };
// packed: log2 sizes of the two levels (4 bits each), first probe (4), then:
// one level only, coordinates swapped, x negated, y negated, x and y offset
// by one (Alg. 2's reflection)
constexpr uint32_t kOneLevel = 1u << 12, kSwap = 1u << 13, kNegX = 1u << 14, kNegY = 1u << 15, kOffset = 1u << 16;

// The probes k = 0..K-1, at t = (2k + 1 - K) / (2K), for which lo < c + m t
// < hi, as an interval [k0, k1); it may hold a probe too many at either end
// (whose taps all have weight zero), never one too few.
__device__ __forceinline__ void cut_probes(float c, float inv_m, float lo, float hi, float Kf, float& k0, float& k1) {
    // inv_m = +-inf: m = 0 (or so small that every probe sits at c): the
    // bounds come out infinite, or NaN on the border, which min and max drop
    const float a = (lo - c) * inv_m, b = (hi - c) * inv_m;
    const float shift = 0.5f * Kf - 0.5f;
    k0 = fmaxf(k0, fmaf(fminf(a, b), Kf, shift) - 0.01f);
    k1 = fminf(k1, fmaf(fmaxf(a, b), Kf, shift) + 0.01f);
}

// First probe and one past the last of the three fetches: the own quad
// within h0 of [0, 1]^2, the Next quad (coordinates (v, -u)) within h1, the
// Prev quad ((-v, u)) within h2 (half a texel of the coarser level each,
// and 1e-6 for the coordinates' own rounding).
__device__ __forceinline__ void probe_ranges(float u, float v, float mu, float mv, int K, const float (&half)[3],
                                             int (&first)[3], int (&last)[3]) {
    const float iu = __frcp_rn(mu), iv = __frcp_rn(mv), Kf = float(K);
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const float h = half[e] + 1e-6f;
        float k0 = 0.0f, k1 = Kf - 1.0f;
        cut_probes(u, iu, e == 1 ? -1.0f - h : -h, e == 1 ? h : 1.0f + h, Kf, k0, k1);
        cut_probes(v, iv, e == 2 ? -1.0f - h : -h, e == 2 ? h : 1.0f + h, Kf, k0, k1);
        first[e] = max(0, int(ceilf(k0)));
        last[e] = max(first[e], min(K, int(floorf(k1)) + 1));
    }
}

// Probe count (see the file comment): same float operations as the oracle.
__device__ __forceinline__ int aniso_probes(float px2, float py2, int kmax) {
    const float mx = fmaxf(px2, py2), mn = fminf(px2, py2);
    if (mx == 0.0f) return 1;
    const float r = __fsqrt_rn(__fdiv_rn(mx, mn));
    if (!(r < float(kmax))) return kmax;
    return max(1, int(ceilf(r)));
}

constexpr int kAnisoThreads = 128;
constexpr int kAnisoWarps = kAnisoThreads / 32;
// Resident blocks per SM.  The kernel is bound by random 128-byte lines from
// DRAM and their latency: 4M queries of 1..16 probes on a 1.4 GB RGBA8 asset
// take 569 / 517 / 546 us at 8 / 9 / 10 blocks (2.8 GB of lines, 5.2 TB/s at
// 9; independent random lines reach 5.2 TB/s).  At 9 a thread has 56
// registers, and the one-, two- and four-channel kernels spill 4 to 20 bytes.
// FP32 RG and RGBA texels want fewer: with at most two probes a query (few
// shared lines) 385 / 323 / 340 and 497 / 417 / 390 us at 9 / 8 / 7, with 16
// probes 567 / 561 / 599 and 666 / 675 / 668.
template <int DT, int C>
constexpr int aniso_blocks() {
    return DT != HTEX_F32 ? 9 : C == 4 ? 7 : C == 2 ? 8 : 9;
}

// A decoded anisotropic query: validity, the probe count and line, and the
// footprint of one probe.
struct AnisoQuery {
    bool ok;
    int h, K;
    float u, v, mu, mv, footprint;
};

__device__ __forceinline__ AnisoQuery decode_aniso(int4 r0, int4 r1, int32_t H, int kmax) {
    AnisoQuery Q;
    const float dudx = __int_as_float(r1.x), dvdx = __int_as_float(r1.y);
    const float dudy = __int_as_float(r1.z), dvdy = __int_as_float(r1.w);
    const float px2 = __fadd_rn(__fmul_rn(dudx, dudx), __fmul_rn(dvdx, dvdx));
    const float py2 = __fadd_rn(__fmul_rn(dudy, dudy), __fmul_rn(dvdy, dvdy));
    float f;
    Q.ok = decode_query(make_int4(r0.x, r0.y, r0.z, 0), H, Q.h, Q.u, Q.v, f);
    Q.ok = Q.ok && isfinite(dudx) && isfinite(dvdx) && isfinite(dudy) && isfinite(dvdy) && isfinite(px2) &&
           isfinite(py2);
    Q.K = Q.ok ? aniso_probes(px2, py2, kmax) : 0;
    const bool major_y = py2 > px2;
    const float pmax = sqrtf(fmaxf(px2, py2));
    const float s = pmax > float(max(Q.K, 1)) ? float(Q.K) / pmax : 1.0f;
    Q.mu = (major_y ? dudy : dudx) * s;
    Q.mv = (major_y ? dvdy : dvdx) * s;
    Q.footprint = Q.ok ? pmax / float(Q.K) : 0.0f;
    return Q;
}

// SPREAD: a warp takes 'few' queries at a time instead of 32 (small batches;
// as a variant of its own, since the run-time count costs the full batches 8%).
template <int DT, int C, bool SPREAD>
__global__ void __launch_bounds__(kAnisoThreads, (aniso_blocks<DT, C>()))
k_lookup_aniso(Asset<GlobalSpace> A, AnisoParams p, int few) {
    constexpr int TB = C * Fmt<DT>::ES;
    constexpr int FW = Fmt<DT>::SCALED ? 5 : 4;      // words per fetch
    __shared__ uint32_t consts[kAnisoWarps][kFetch + 3 * FW][32];
    constexpr int SW = (C + 1) | 1;                  // words of an item's sums, odd (bank spread)
    __shared__ float part[kAnisoWarps][32][SW];      // one round's item sums: data and weight
    __shared__ float total[kAnisoWarps][32][SW];     // the queries' sums
    __shared__ uint8_t mark[kAnisoWarps][32];        // the fetch that starts at an item of the round
    const unsigned lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
    uint32_t (*const cw)[32] = consts[wib];
    const htex_query* const qq = reinterpret_cast<const htex_query*>(p.q);   // two 16-byte words a query
    const int per_warp = SPREAD ? few : 32;
    const int64_t step = int64_t(gridDim.x) * kAnisoWarps * per_warp;
    for (int64_t base = (int64_t(blockIdx.x) * kAnisoWarps + wib) * per_warp; base < p.n; base += step) {
        // ---- this lane's query: decode, probe count, the fetches with items
        const int64_t i = base + lane;
        const bool valid = (!SPREAD || int(lane) < per_warp) && i < p.n;
        const int4 r0 = valid ? ld_query(qq, 2 * i) : make_int4(-1, 0, 0, 0);
        const int4 r1 = valid ? ld_query(qq, 2 * i + 1) : make_int4(0, 0, 0, 0);
        const AnisoQuery Q = decode_aniso(r0, r1, A.H, p.kmax);
        if (valid && !Q.ok && p.status) atomicAdd(p.status, 1);
        int slots = 0, len[3] = {0, 0, 0};
        if (Q.ok) {
            const uint4 rec = A.rec.ld16(uint64_t(Q.h) * 16u);
            const uint32_t code[3] = {rec.x, rec.y, rec.z};
            const float lf = footprint_log2(Q.footprint);
            TexRef t[3];
            Lod d[3];
            float half[3];
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                t[e] = tex_ref<DT>(A, code[e] & ~kFlipBit);
                d[e] = select_lod(lf, t[e].n);
                half[e] = __int_as_float((126 - (t[e].n - coarsest(d[e]))) << 23);   // 2^-(log2 size + 1)
            }
            int first[3], last[3];
            probe_ranges(Q.u, Q.v, Q.mu, Q.mv, Q.K, half, first, last);
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                if (last[e] <= first[e]) continue;
                const bool flip = code[e] & kFlipBit, one = d[e].l1 < 0;
                // own (u, v), Next (v, -u), Prev (-v, u), each (1 - x, 1 - y) when reflected
                const uint32_t turn = (e ? kSwap : 0u) | ((e == 2) != flip ? kNegX : 0u) |
                                      ((e == 1) != flip ? kNegY : 0u) | (flip ? kOffset : 0u);
                const uint64_t o = t[e].off + uint64_t(level_texels(t[e].n, d[e].l0)) * TB;
                uint32_t (*f)[32] = cw + kFetch + slots * FW;
                f[0][lane] = uint32_t(o);
                f[1][lane] = uint32_t(o >> 32);
                f[2][lane] = uint32_t(t[e].n - d[e].l0) | uint32_t(t[e].n - coarsest(d[e])) << 4 |
                             uint32_t(first[e]) << 8 | (one ? kOneLevel : 0u) | turn;
                f[3][lane] = __float_as_uint(one ? 0.0f : d[e].w1);
                if constexpr (Fmt<DT>::SCALED) f[4][lane] = __float_as_uint(t[e].scale);
                const int l = last[e] - first[e];
                if (slots == 0) len[0] = l;
                else if (slots == 1) len[1] = l;
                else len[2] = l;
                ++slots;
            }
            cw[kU][lane] = __float_as_uint(Q.u);
            cw[kV][lane] = __float_as_uint(Q.v);
            cw[kMu][lane] = __float_as_uint(Q.mu);
            cw[kMv][lane] = __float_as_uint(Q.mv);
            cw[kK][lane] = uint32_t(Q.K);
            cw[kInv2K][lane] = __float_as_uint(1.0f / float(2 * Q.K));
        }
#pragma unroll
        for (int c = 0; c <= C; ++c) total[wib][lane][c] = 0.0f;

        // ---- the warp's items: where each query's fetches start
        const int items = len[0] + len[1] + len[2];
        int incl = items;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= unsigned(d)) incl += o;
        }
        const int P = __shfl_sync(0xffffffffu, incl, 31);
        const int start = incl - items;
        const uint32_t span = uint32_t(start) | uint32_t(incl) << 16;   // this lane's query's items
        uint32_t seg = 0;    // query and slot running on from the round before, and where it started
        int seg_start = 0;

        for (int R = 0; R < P; R += 32) {
            // each lane's item: mark where fetches start, look left for the nearest mark
            uint32_t starts = 0;
            int at = start - R;
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                if (len[s] > 0 && unsigned(at) < 32u) {
                    mark[wib][at] = uint8_t(lane | unsigned(s) << 5);
                    starts |= 1u << at;
                }
                at += len[s];
            }
            starts = __reduce_or_sync(0xffffffffu, starts);
            __syncwarp();
            const uint32_t before = starts & (0xffffffffu >> (31u - lane));
            if (before) {
                const int m = 31 - __clz(int(before));
                seg = mark[wib][m];
                seg_start = R + m;
            }
            const int j = R + int(lane);
            const bool has = j < P;
            const unsigned q = seg & 31u;
            uint32_t (*f)[32] = cw + kFetch + (seg >> 5) * FW;
            const uint32_t c2 = f[2][q];
            const uint64_t o0 = uint64_t(f[1][q]) << 32 | f[0][q];
            const int n0 = int(c2 & 15u), n1 = int(c2 >> 4 & 15u);
            const float w1 = has ? __uint_as_float(f[3][q]) : 0.0f, w0 = has ? 1.0f - w1 : 0.0f;
            float scale = 1.0f;
            if constexpr (Fmt<DT>::SCALED) scale = __uint_as_float(f[4][q]);
            const int k = int(c2 >> 8 & 15u) + j - seg_start;
            const float t = float(2 * k + 1 - int(cw[kK][q])) * __uint_as_float(cw[kInv2K][q]);
            const float pu = fmaf(__uint_as_float(cw[kMu][q]), t, __uint_as_float(cw[kU][q]));
            const float pv = fmaf(__uint_as_float(cw[kMv][q]), t, __uint_as_float(cw[kV][q]));
            const bool swap = c2 & kSwap;
            const float off = (c2 & kOffset) ? 1.0f : 0.0f;
            const float a = swap ? pv : pu, b = swap ? pu : pv;
            const float x = off + ((c2 & kNegX) ? -a : a), y = off + ((c2 & kNegY) ? -b : b);

            Sums<C> acc;
            LevelTaps<TB> L0, L1;
            // The code scale: on the sums where a weighted code keeps its 24 bits
            // (E4M3, F16: codes of at least 2^-9, 2^-24), else on each weight
            // (BF16 codes span the FP32 range).  4M E4M3 RGBA queries of 1..16
            // probes on 1.4 GB: 529 us on the sums, 578 us on the weights.
            constexpr bool scale_weights = DT == HTEX_BF16, scale_sums = Fmt<DT>::SCALED && !scale_weights;
            const auto weight = [&](const LevelTaps<TB>& L, int m) {
                return scale_weights ? L.w[m] * scale_of(L.w[m], scale) : L.w[m];
            };
            float W = L0.plan(o0, n0, x, y, w0);
            const bool two = __any_sync(0xffffffffu, w1 != 0.0f);
            // the coarser level's texels follow the finer one's (its own when there is no coarser one)
            const uint64_t o1 = o0 + (uint64_t(TB) << (2 * n0));
            if constexpr (TB <= 8 && (TB & (TB - 1)) == 0 && (DT != HTEX_F32 || C == 1)) {
                Raw<DT, C> ta[4], tb[4];   // every load before the first decode
#pragma unroll
                for (int m = 0; m < 4; ++m) ta[m].load_if(A.pool, L0.read(m), L0.at(m), l2_leave_policy());
                if (two) {
                    W += L1.plan(o1, n1, x, y, w1);
#pragma unroll
                    for (int m = 0; m < 4; ++m) tb[m].load_if(A.pool, L1.read(m), L1.at(m), l2_leave_policy());
                }
                float v[C];
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    ta[m].decode(v);
                    acc.fma(weight(L0, m), v);
                }
                if (two) {
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        tb[m].decode(v);
                        acc.fma(weight(L1, m), v);
                    }
                }
            } else {
                float v[4][C];
#pragma unroll
                for (int m = 0; m < 4; ++m) load_texel_if<DT, C>(A.pool, L0.read(m), L0.at(m), v[m]);
#pragma unroll
                for (int m = 0; m < 4; ++m) acc.fma(weight(L0, m), v[m]);
                if (two) {
                    W += L1.plan(o1, n1, x, y, w1);
#pragma unroll
                    for (int m = 0; m < 4; ++m) load_texel_if<DT, C>(A.pool, L1.read(m), L1.at(m), v[m]);
#pragma unroll
                    for (int m = 0; m < 4; ++m) acc.fma(weight(L1, m), v[m]);
                }
            }
            float sums[C];
            acc.get(sums);
            const float on_sums = scale_sums ? scale_of(W, scale) : 1.0f;
#pragma unroll
            for (int c = 0; c < C; ++c) part[wib][lane][c] = scale_sums ? sums[c] * on_sums : sums[c];
            part[wib][lane][C] = W;
            __syncwarp();

            // add them to their queries' sums: a lane per query and channel
            // (data or weight), the items in order
            const int end = min(P - R, 32);
            const int q0 = __shfl_sync(0xffffffffu, int(q), 0), q1 = __shfl_sync(0xffffffffu, int(q), end - 1);
            constexpr int PER = 32 / (C + 1);   // queries per pass
            const int qr = int(lane) / (C + 1), ch = int(lane) - qr * (C + 1);
            for (int qb = q0; qb <= q1; qb += PER) {
                const int qi = qb + qr;
                const uint32_t sp = __shfl_sync(0xffffffffu, span, qi & 31);
                if (qr < PER && qi <= q1) {
                    const int lo = max(int(sp & 0xffffu) - R, 0), hi = min(int(sp >> 16) - R, end);
                    float s = total[wib][qi][ch];
#pragma unroll 4
                    for (int m = lo; m < hi; ++m) s += part[wib][m][ch];
                    total[wib][qi][ch] = s;
                }
            }
            seg = __shfl_sync(0xffffffffu, seg, 31);
            seg_start = __shfl_sync(0xffffffffu, seg_start, 31);
            __syncwarp();
        }

        // ---- normalise and store (invalid queries: W = 0, data 0, 0 * inf = NaN)
        if (valid) {
            const float inv = __frcp_rn(total[wib][lane][C]) * Fmt<DT>::UNIT;
            float res[C];
#pragma unroll
            for (int c = 0; c < C; ++c) res[c] = total[wib][lane][c] * inv;
            store_out<C>(p.out, i, res);
        }
        __syncwarp();
    }
}

template <int DT, int C>
htex_status launch_aniso_c(const htex_textures* t, const AnisoParams& p, cudaStream_t s) {
    static Occupancy occupancy;
    const int b = occupancy.get(k_lookup_aniso<DT, C, false>, kAnisoThreads, t->device);
    // a warp works its queries' items off 32 at a time, so a batch that leaves
    // warps idle gives each warp fewer queries and so fewer rounds: 1,000 /
    // 16,384 / 65,536 RGBA8 queries of 1..16 probes 13.5 / 16.4 / 20.2 us ->
    // 6.2 / 10.3 / 16.5 us
    const int64_t resident = int64_t(t->num_sms) * b;
    int per_warp = 32;
    while (per_warp > 4 && p.n <= resident * kAnisoWarps * (per_warp / 2)) per_warp /= 2;
    const int64_t per_block = int64_t(kAnisoWarps) * per_warp;
    const int64_t grid = std::min<int64_t>((p.n + per_block - 1) / per_block, resident);
    const auto kernel = per_warp < 32 ? k_lookup_aniso<DT, C, true> : k_lookup_aniso<DT, C, false>;
    kernel<<<unsigned(grid), kAnisoThreads, 0, s>>>(global_asset(t), p, per_warp);
    return cudaGetLastError() == cudaSuccess ? HTEX_OK : HTEX_ERR_CUDA;
}

template <int DT>
htex_status launch_aniso_dt(const htex_textures* t, const AnisoParams& p, cudaStream_t s) {
    switch (t->C) {
    case 1: return launch_aniso_c<DT, 1>(t, p, s);
    case 2: return launch_aniso_c<DT, 2>(t, p, s);
    case 3: return launch_aniso_c<DT, 3>(t, p, s);
    case 4: return launch_aniso_c<DT, 4>(t, p, s);
    }
    return HTEX_ERR_INVALID_ARG;
}

}  // namespace htex

using namespace htex;

htex_status htex_launch_aniso(const htex_textures* t, const htex_query_aniso* q, int64_t n, int32_t kmax,
                              float* out, htex_stream stream, int32_t* d_status) {
    const AnisoParams p{q, n, kmax, out, d_status};
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    switch (t->dtype) {
    case HTEX_F32: return launch_aniso_dt<HTEX_F32>(t, p, s);
    case HTEX_U8: return launch_aniso_dt<HTEX_U8>(t, p, s);
    case HTEX_F16: return launch_aniso_dt<HTEX_F16>(t, p, s);
    case HTEX_BF16: return launch_aniso_dt<HTEX_BF16>(t, p, s);
    case HTEX_E4M3: return launch_aniso_dt<HTEX_E4M3>(t, p, s);
    }
    return HTEX_ERR_INVALID_ARG;
}

extern "C" htex_status htex_lookup_aniso(const htex_textures* t, const htex_query_aniso* q, int64_t n,
                                         int32_t max_aniso, uint32_t flags, float* out, htex_stream stream,
                                         int32_t* d_status) {
    if (!t || n < 0 || max_aniso < 1 || max_aniso > 16) return HTEX_ERR_INVALID_ARG;
    if (flags & ~uint32_t(HTEX_LOOKUP_BIN)) return HTEX_ERR_INVALID_ARG;
    if (n == 0) return HTEX_OK;
    if (!q || !out) return HTEX_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(q) & 15u) != 0) return HTEX_ERR_INVALID_ARG;
    const uintptr_t out_align = t->C == 4 ? 16u : (t->C == 2 ? 8u : 4u);
    if ((reinterpret_cast<uintptr_t>(out) & (out_align - 1)) != 0) return HTEX_ERR_INVALID_ARG;
    if (flags & HTEX_LOOKUP_BIN) {
        const htex_status st = htex_launch_aniso_sorted(t, q, n, max_aniso, out, stream, d_status);
        if (st != HTEX_ERR_OUT_OF_MEMORY) return st;   // no memory to sort in (nothing launched): in the given order
    }
    return htex_launch_aniso(t, q, n, max_aniso, out, stream, d_status);
}
