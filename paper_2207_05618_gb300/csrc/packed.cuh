// Two FP32 operations per instruction (Blackwell's packed f32x2 forms, each
// half rounded like the scalar operation): the kernels here are bound by
// instruction issue, not by the FP32 units, so a channel pair per
// instruction takes issue slots off.
#pragma once

#include <cstdint>

namespace htex {

__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t p, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// C channel sums; fma(w, t) adds w * t[c] to each (fused, rounded per channel).
template <int C>
struct Sums {
    static constexpr int P = C / 2;
    uint64_t pair[P > 0 ? P : 1];
    float odd;

    __device__ __forceinline__ Sums() : odd(0.0f) {
#pragma unroll
        for (int k = 0; k < (P > 0 ? P : 1); ++k) pair[k] = 0ull;
    }
    __device__ __forceinline__ void fma(float w, const float (&t)[C]) {
        const uint64_t ww = pack2(w, w);
#pragma unroll
        for (int k = 0; k < P; ++k) pair[k] = fma2(ww, pack2(t[2 * k], t[2 * k + 1]), pair[k]);
        if constexpr (C % 2 != 0) odd = fmaf(w, t[C - 1], odd);
    }
    __device__ __forceinline__ void get(float (&t)[C]) const {
#pragma unroll
        for (int k = 0; k < P; ++k) unpack2(pair[k], t[2 * k], t[2 * k + 1]);
        if constexpr (C % 2 != 0) t[C - 1] = odd;
    }
};

}  // namespace htex
