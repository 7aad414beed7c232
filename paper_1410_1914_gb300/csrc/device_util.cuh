// Device-side helpers shared by the kernels of the library: sums, pairs and triples of floats.
#pragma once

#include <cuda_runtime.h>

namespace cl {

// two floats in a register pair: one instruction for both, rounded as the single ones are
using F2 = unsigned long long;
__device__ __forceinline__ F2 f2(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 f2_get(F2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// s + e = a + b exactly (Knuth's two-sum)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// A sum of floats as a + b + c: b adds up what the roundings of a lose, c what those of b lose, so that it is good to
// 2^-70 of the terms, where a sum in FP64 loses up to 2^-53 at every addition.  13 FP32 instructions per term, which
// issue in a fifth of the time of one FP64 addition and its conversion (1/64 of the FP32 rate, for idle lanes too).
// With b as the last word (2^-46) the sums of 16 cells were off by up to 400 x 2^-53.
struct F3 {
    float a, b, c;
};
__device__ __forceinline__ void f3_add(F3& s, float x) {
    float e;
    two_sum(s.a, x, s.a, e);
    two_sum(s.b, e, s.b, e);
    s.c = __fadd_rn(s.c, e);
}
// a term that is small beside the others (the low word of one), as exact for half the instructions
__device__ __forceinline__ void f3_add_low(F3& s, float x) {
    float e;
    two_sum(s.b, x, s.b, e);
    s.c = __fadd_rn(s.c, e);
}
__device__ __forceinline__ void f3_add(F3& s, const F3& o) {
    f3_add(s, o.a);
    f3_add_low(s, o.b);
    s.c = __fadd_rn(s.c, o.c);
}
// w v, the rounding error of the product included
__device__ __forceinline__ void f3_add_product(F3& s, float w, float v) {
    const float p = __fmul_rn(w, v);
    f3_add(s, p);
    f3_add_low(s, __fmaf_rn(w, v, -p));
}
// the same for a small term v
__device__ __forceinline__ void f3_add_product_low(F3& s, float w, float v) {
    const float p = __fmul_rn(w, v);
    f3_add_low(s, p);
    s.c = __fadd_rn(s.c, __fmaf_rn(w, v, -p));
}
// the sum in FP64; past an overflow the errors are inf - inf, and the sum alone says what happened
__device__ __forceinline__ double f3_get(const F3& s) {
    const double lost = (double)s.b + (double)s.c;
    return isfinite(s.a) ? (double)s.a + lost : (double)s.a;
}

// 1 / a from the f32 reciprocal r (24 bits) and one third-order step, r (1 + e + e^2) with e = 1 - a r: what is left
// out is e^3, below 2^-69.  a is a finite positive normal number well inside the f32 range.
__device__ __forceinline__ double recip(double a) {
    const double r = (double)__frcp_rn((float)a);
    const double e = fma(-a, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

template <int NV>
__device__ __forceinline__ void warp_sum(double (&v)[NV]) {
#pragma unroll
    for (int k = 0; k < NV; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
}

// Block-wide sum of NV doubles in a fixed order; thread 0 writes out[0..NV).
// blockDim must be a multiple of 32 and at most 1024 threads.
template <int NV>
__device__ void block_sum_store(double (&v)[NV], double* out) {
    __shared__ double sh[32][NV];
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    const int nthreads = blockDim.x * blockDim.y * blockDim.z;
    const int lane = tid & 31, warp = tid >> 5, nwarps = (nthreads + 31) >> 5;
    warp_sum<NV>(v);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) sh[warp][k] = v[k];
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k] = lane < nwarps ? sh[lane][k] : 0.0;
        warp_sum<NV>(v);
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < NV; ++k) out[k] = v[k];
    }
}

}  // namespace cl
