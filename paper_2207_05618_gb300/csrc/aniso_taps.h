// The taps of one level of one fetch of an anisotropic lookup, and which of
// them are read.  Plain C++ beside the kernel, so that the host can check
// that no tap outside its texture is ever read.
#pragma once

#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define HTEX_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define HTEX_HOST_DEVICE inline
#endif

namespace htex {

// Two taps along one axis for an arbitrary coordinate: index i = floor(s)
// unclamped, in-bounds weights (zero for a tap outside [0, N)).
struct TapsG {
    int i;
    float w0, w1;
};

HTEX_HOST_DEVICE TapsG taps_g(float p, int N) {
    const float s = fmaf(p, float(N), -0.5f);
    const float fi = floorf(s);
    const float a = s - fi;
    const int i = int(fi);
    return TapsG{i, (i >= 0 && i < N) ? 1.0f - a : 0.0f, (i + 1 >= 0 && i + 1 < N) ? a : 0.0f};
}

// Four taps of a level whose texels take TB bytes, their weights (level
// weight included, code scale not) and their places.
template <int TB>
struct LevelTaps {
    uint64_t o;
    uint32_t row;
    float w[4];

    // The level's texel (0, 0) at byte 'base', 2^n texels a side, quad
    // coordinates (x, y), level weight wl.  Returns the level's share of the
    // normalisation weight.
    HTEX_HOST_DEVICE float plan(uint64_t base, int n, float x, float y, float wl) {
        const int N = 1 << n;
        const TapsG tx = taps_g(x, N), ty = taps_g(y, N);
        const float y0 = ty.w0 * wl, y1 = ty.w1 * wl;
        w[0] = y0 * tx.w0;
        w[1] = y0 * tx.w1;
        w[2] = y1 * tx.w0;
        w[3] = y1 * tx.w1;
        o = base + uint64_t(int64_t(((ty.i << n) + tx.i) * TB));
        row = uint32_t(TB) << n;
        return wl * (tx.w0 + tx.w1) * (ty.w0 + ty.w1);
    }
    HTEX_HOST_DEVICE uint64_t at(int k) const { return o + (k & 1 ? TB : 0) + (k & 2 ? row : 0u); }
    // Tap k lies in the texture and counts.  Decided before the code scale:
    // a texture's scale may be any float, and 0 * inf is not zero.
    HTEX_HOST_DEVICE bool read(int k) const { return w[k] != 0.0f; }
};

// The code scale of something weighted: zero for a weight of zero, whatever
// the texture's scale.
HTEX_HOST_DEVICE float scale_of(float weight, float scale) { return weight != 0.0f ? scale : 0.0f; }

}  // namespace htex
