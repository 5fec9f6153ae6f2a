// Device arithmetic shared by the step kernels (k_step.cu, k_solo.cu).
#pragma once

#include "msat_internal.cuh"

namespace msat {

// Two independent single-precision operations in one instruction, each
// rounded to nearest.
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 d;
    asm("{.reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; add.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z;}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 d;
    asm("{.reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; mul.rn.f32x2 z, x, y; mov.b64 {%0, %1}, z;}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{.reg .b64 x, y, z; mov.b64 x, {%2, %3}; mov.b64 y, {%4, %5}; mov.b64 z, {%6, %7}; fma.rn.f32x2 z, x, y, z; mov.b64 {%0, %1}, z;}"
        : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}

// Dyadic tree over the first K lanes' values (lane 0 receives the result).
__device__ __forceinline__ float warp_dyadic(float v, int K, int lane) {
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
        const float o = __shfl_down_sync(0xffffffffu, v, s);
        if ((lane & (2 * s - 1)) == 0 && lane + s < K) v = v + o;
    }
    return v;
}

// --------------------------------------------------------------- update

struct AdamView {
    float a_t, r_t, b1, b2, omb1, omb2, eps;
};

__device__ __forceinline__ AdamView adam_view(const StepScalars *sc) {
    AdamView A;
    A.a_t = sc->a_t;
    A.r_t = sc->r_t;
    A.b1 = sc->b1f;
    A.b2 = sc->b2f;
    A.omb1 = sc->omb1f;
    A.omb2 = sc->omb2f;
    A.eps = sc->epsf;
    return A;
}

// One Adam update.  A variable none of whose clauses has been unsat has
// m = v = 0 (one in six on random 3-SAT near the threshold), and a zero
// operand sends the rounded square root and division to their special-case
// code, which the other lanes of the warp then wait for.  sqrt(+-0) = +-0 and
// +-0 / d = +-0 for d > 0 need neither: those lanes take the operations on
// harmless operands and keep the zero (one block per restart, n=5000: 15.3
// -> 15.0 us a step).
__device__ __forceinline__ float adam_update(const AdamView &A, float x, float &m, float &v,
                                             float g) {
    const float mq = A.b1 * m + A.omb1 * g;
    const float vq = A.b2 * v + (A.omb2 * g) * g;
    const bool vz = vq == 0.0f;
    const float root = sqrtf(vz ? 1.0f : vq);
    const float den = (vz ? vq : root) * A.r_t + A.eps;
    const float num = A.a_t * mq;
    const bool nz = num == 0.0f && den > 0.0f;
    const float quot = (nz ? den : num) / den;
    m = mq;
    v = vq;
    return x - (nz ? num : quot);
}

}  // namespace msat
