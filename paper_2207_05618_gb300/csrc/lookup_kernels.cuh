// Filter kernels of htex_lookup (paper Section 4.4, Alg. 3 with Alg. 2)
// and their launchers, instantiated per texel format in lookup_<format>.cu
// so that the formats compile in parallel.  See lookup.cu for the paths.
#pragma once

#include <algorithm>

#include <cuda_runtime.h>

#include "lookup_core.cuh"

namespace htex {

template <bool BINNED, class I>
__device__ __forceinline__ int64_t dst_of(const FwdParams& p, I i) {
    return BINNED ? int64_t(__ldcs(p.idx + i)) : i;
}

// Grid-stride loop for the global path, software-pipelined: the query two
// iterations ahead and the record one iteration ahead are in flight while
// the current query's texels are gathered.  I: the index type (32-bit when
// n allows); UNI: every texture has one resolution.
template <int DT, int C, bool BINNED, bool DEFER, bool UNI, class I, class S>
__device__ __forceinline__ void lookup_loop(const Asset<S>& A, const FwdParams& p) {
    const I n = I(p.n);
    const I stride = I(gridDim.x) * I(blockDim.x);
    I i0 = I(blockIdx.x) * I(blockDim.x) + I(threadIdx.x);
    if (i0 >= n) return;
    I i1 = i0 + stride;
    int4 raw0 = ld_query(p.q, i0);
    int64_t dst0 = dst_of<BINNED>(p, i0);
    int4 raw1 = make_int4(-1, 0, 0, 0);
    int64_t dst1 = 0;
    if (i1 < n) {
        raw1 = ld_query(p.q, i1);
        dst1 = dst_of<BINNED>(p, i1);
    }
    Record<S> rec0 = record_of(A, raw0);
    while (true) {
        const I i2 = i1 + stride;
        int4 raw2 = make_int4(-1, 0, 0, 0);
        int64_t dst2 = 0;
        if (i2 < n) {
            raw2 = ld_query(p.q, i2);
            dst2 = dst_of<BINNED>(p, i2);
        }
        const Record<S> rec1 = record_of(A, raw1);   // zeros past the end
        lookup_one<DT, C, DEFER, UNI>(A, p, raw0, rec0, dst0);
        if (i1 >= n) break;
        raw0 = raw1;
        dst0 = dst1;
        rec0 = rec1;
        raw1 = raw2;
        dst1 = dst2;
        i1 = i2;
    }
}

// Grid-stride loop for the shared-memory path, two queries per thread and
// iteration: both queries and both records are loaded before either is
// filtered, so their latencies overlap; the pair four strides ahead is
// prefetched into L2.  I: the index type (32-bit when n allows).
template <int DT, int C, bool BINNED, bool DEFER, bool UNI, class I, class S>
__device__ __forceinline__ void lookup_loop_pairs(const Asset<S>& A, const FwdParams& p) {
    const I n = I(p.n);
    const I stride = I(gridDim.x) * I(blockDim.x);
    for (I i = I(blockIdx.x) * I(blockDim.x) + I(threadIdx.x); i < n; i += 2 * stride) {
        const I j = i + stride;
        const int4 ra = ld_query(p.q, i);
        const int4 rb = j < n ? ld_query(p.q, j) : make_int4(-1, 0, 0, 0);
        if (i + 4 * stride < n) prefetch_query(p.q, i + 4 * stride);
        if (j + 4 * stride < n) prefetch_query(p.q, j + 4 * stride);
        const Record<S> ca = record_of(A, ra), cb = record_of(A, rb);
        lookup_one<DT, C, DEFER, UNI>(A, p, ra, ca, dst_of<BINNED>(p, i));
        if (j < n) lookup_one<DT, C, DEFER, UNI>(A, p, rb, cb, dst_of<BINNED>(p, j));
    }
}

// One resident block of 640 threads per SM (20 warps, 5 per scheduler)
// under 102 registers: each SM's threads then filter a contiguous stretch
// of the (sorted) queries, so the texels of neighbouring queries meet in
// its L1.  Measured on the sorted asset batch: 1 x 640 0.525 ms; 1 x 512,
// 1 x 768 2-3% slower (1 x 896 and 1 x 1024 spill); 2 x 320 0.558 ms,
// 2 x 256 1.6% slower than that, 2 x 384 and 3 x 256 2.5-5% slower, odd
// warp counts per SM (2 x 224 / 288 / 352) slower still.
constexpr int kGlobalThreads = 640;
#ifndef HTEX_GLOBAL_MIN_BLOCKS
#define HTEX_GLOBAL_MIN_BLOCKS 1
#endif
// one block of 1024 threads per SM (the pool staged once per SM): measured
// against 384 x 3 / 512 x 2 / 576 x 2 / 640 x 2 blocks per SM, 2.3-4.6%
// faster on the cube stream
constexpr int kStagedThreads = 1024;

// SORTED: the queries come sorted by halfedge range.  Their texels then
// mostly come from L1 and L2, and 8-byte texels too are worth loading ahead
// in two registers each: 4M sorted FP16 RGBA / FP32 RG lookups, the whole
// call, 279 / 259 -> 262 / 218 us on 130k halfedges (2.9 GB), 246 / 228 ->
// 219 / 182 us on 104k (0.56 GB); in a random order 203 -> 212 and 83 -> 85
// us (2M, 1M), so not there.  Other texel sizes: the same kernel either way.
template <int DT, int C, bool BINNED, bool UNI, bool SORTED>
__global__ void __launch_bounds__(kGlobalThreads, HTEX_GLOBAL_MIN_BLOCKS) k_lookup_global(Asset<GlobalSpace> A, FwdParams p) {
    constexpr bool DEFER = Raw<DT, C>::PACKED || (SORTED && Raw<DT, C>::DOUBLE);
    if (p.n <= int64_t(INT32_MAX) - 2 * int64_t(gridDim.x) * blockDim.x)
        lookup_loop<DT, C, BINNED, DEFER, UNI, int32_t>(A, p);
    else
        lookup_loop<DT, C, BINNED, DEFER, UNI, int64_t>(A, p);
}

// Shared-memory layout of a staged asset: records, headers, scales, pool,
// each starting on a 16-byte boundary.
struct StageLayout {
    uint32_t rec, hdr, scale, pool, total;
};

__host__ __device__ inline StageLayout stage_layout(int32_t H, int32_t E, int64_t pool_bytes) {
    StageLayout s;
    s.rec = 0;
    s.hdr = s.rec + uint32_t(H) * 16u;
    s.scale = s.hdr + uint32_t(E) * 16u;
    s.pool = s.scale + ((uint32_t(E) * 4u + 15u) & ~15u);
    s.total = s.pool + uint32_t(pool_bytes);
    return s;
}

__device__ __forceinline__ void stage16(uint8_t* dst, const void* src, uint32_t bytes) {
    const uint4* s = reinterpret_cast<const uint4*>(src);
    uint4* d = reinterpret_cast<uint4*>(dst);
    for (uint32_t k = threadIdx.x; k < bytes / 16u; k += blockDim.x) d[k] = __ldg(s + k);
}

template <int DT, int C, bool BINNED, bool UNI>
__global__ void __launch_bounds__(kStagedThreads, 1) k_lookup_staged(Asset<GlobalSpace> G, int32_t E,
                                                                  int64_t pool_bytes, FwdParams p) {
    extern __shared__ __align__(16) uint8_t smem[];
    const StageLayout L = stage_layout(G.H, E, pool_bytes);
    for (uint32_t h = threadIdx.x; h < uint32_t(G.H); h += blockDim.x) {   // the records as four arrays (Record<SharedSpace>)
        const uint4 r = G.rec.ld16(uint64_t(h) * 16u);
        uint32_t* w = reinterpret_cast<uint32_t*>(smem + L.rec) + h;
        w[0] = r.x;
        w[G.H] = r.y;
        w[2 * G.H] = r.z;
        w[3 * G.H] = r.w;
    }
    stage16(smem + L.hdr, G.hdr.base, uint32_t(E) * 16u);
    stage16(smem + L.scale, G.scale.base, (uint32_t(E) * 4u + 15u) & ~15u);
    stage16(smem + L.pool, G.pool.base, uint32_t(pool_bytes));
    __syncthreads();
    Asset<SharedSpace> A;
    A.rec.base = smem + L.rec;
    A.hdr.base = smem + L.hdr;
    A.scale.base = smem + L.scale;
    A.pool.base = smem + L.pool;
    A.H = G.H;
    A.uniform_log2n = G.uniform_log2n;
    A.uniform_stride16 = G.uniform_stride16;
    if (p.n <= int64_t(INT32_MAX) - 4 * int64_t(gridDim.x) * blockDim.x)
        lookup_loop_pairs<DT, C, BINNED, false, UNI, int32_t>(A, p);
    else
        lookup_loop_pairs<DT, C, BINNED, false, UNI, int64_t>(A, p);
}

// Internal flag of the launchers: the queries are sorted by halfedge range.
constexpr uint32_t kLookupSorted = 1u << 16;

constexpr uint32_t kMaxStageBytes = 96u * 1024u;       // largest asset staged in shared memory
constexpr int64_t kMinStagedQueries = int64_t(1) << 20;  // fewest queries worth staging for

template <class K>
int resident_blocks(K kernel, int threads, size_t smem) {
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, threads, smem) != cudaSuccess) b = 1;
    return b > 0 ? b : 1;
}

template <int DT, int C, bool BINNED>
htex_status launch_fwd(const htex_textures* t, const FwdParams& p, uint32_t flags, cudaStream_t s) {
    const Asset<GlobalSpace> A = global_asset(t);
    const StageLayout L = stage_layout(t->H, t->E, t->pool_bytes);
    // (sorted-index launches never stage: they serve pools above the sort threshold)
    const bool staged = !BINNED && !(flags & HTEX_LOOKUP_GLOBAL) && int64_t(L.total) <= int64_t(kMaxStageBytes) &&
                        p.n >= kMinStagedQueries;
    if (staged) {
        if constexpr (!BINNED) {
            auto k = t->uniform_log2n >= 0 ? k_lookup_staged<DT, C, false, true> : k_lookup_staged<DT, C, false, false>;
            if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(L.total)) != cudaSuccess)
                return HTEX_ERR_CUDA;
            const int64_t want = (p.n + kStagedThreads - 1) / kStagedThreads;
            const int64_t grid =
                std::min<int64_t>(want, int64_t(t->num_sms) * resident_blocks(k, kStagedThreads, L.total));
            k<<<unsigned(grid), kStagedThreads, L.total, s>>>(A, t->E, t->pool_bytes, p);
        }
    } else {
        const bool uniform = t->uniform_log2n >= 0;
        auto k = uniform ? k_lookup_global<DT, C, BINNED, true, false> : k_lookup_global<DT, C, BINNED, false, false>;
        bool sorted = false;
        if constexpr (!BINNED && Raw<DT, C>::DOUBLE) {
            sorted = flags & kLookupSorted;
            if (sorted) k = uniform ? k_lookup_global<DT, C, false, true, true> : k_lookup_global<DT, C, false, false, true>;
        }
        static Occupancy occupancy[4];
        const int blocks = occupancy[2 * sorted + uniform].get(k, kGlobalThreads, t->device);
        const int64_t resident = int64_t(t->num_sms) * blocks;
        // a batch that does not fill every SM, or fills them less than twice,
        // is spread evenly over all of them, in blocks of fewer warps: 4,096 /
        // 40,000 / 100,000 FP32 RGB lookups 10.1 / 12.3 / 17.4 us -> 5.0 / 8.3 /
        // 15.1 us; more rounds (300,000 and up) gain nothing from it
        const int64_t full = resident * kGlobalThreads, rounds = p.n > full && p.n <= 2 * full ? 2 : 1;
        const int64_t share = (p.n + resident * rounds - 1) / (resident * rounds);
        const int threads = int(std::min<int64_t>(kGlobalThreads, (share + 31) / 32 * 32));
        const int64_t grid = std::min<int64_t>((p.n + threads - 1) / threads, resident);
        k<<<unsigned(grid), threads, 0, s>>>(A, p);
    }
    return cudaGetLastError() == cudaSuccess ? HTEX_OK : HTEX_ERR_CUDA;
}

template <int DT, bool BINNED>
htex_status launch_fwd_c(const htex_textures* t, const FwdParams& p, uint32_t flags, cudaStream_t s) {
    switch (t->C) {
    case 1: return launch_fwd<DT, 1, BINNED>(t, p, flags, s);
    case 2: return launch_fwd<DT, 2, BINNED>(t, p, flags, s);
    case 3: return launch_fwd<DT, 3, BINNED>(t, p, flags, s);
    case 4: return launch_fwd<DT, 4, BINNED>(t, p, flags, s);
    }
    return HTEX_ERR_INVALID_ARG;
}

// One launcher per texel format (lookup_<format>.cu).
htex_status launch_fwd_f32(const htex_textures* t, const FwdParams& p, uint32_t flags, cudaStream_t s, bool binned);
htex_status launch_fwd_u8(const htex_textures* t, const FwdParams& p, uint32_t flags, cudaStream_t s, bool binned);
htex_status launch_fwd_f16(const htex_textures* t, const FwdParams& p, uint32_t flags, cudaStream_t s, bool binned);
htex_status launch_fwd_bf16(const htex_textures* t, const FwdParams& p, uint32_t flags, cudaStream_t s, bool binned);
htex_status launch_fwd_e4m3(const htex_textures* t, const FwdParams& p, uint32_t flags, cudaStream_t s, bool binned);

}  // namespace htex
