// Packed FP32x2 arithmetic on two genotypes (A in .x, B in .y): each
// instruction gives two IEEE round-to-nearest results.
#pragma once

#include "adgb_internal.cuh"

namespace adgb {

__device__ __forceinline__ float2 bc(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// negations and differences as plain adds: 1.5% faster in the two-genotypes-a-
// warp search than as multiplications and FMAs by -1
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }

struct V2 {   // a 3-vector of both genotypes
    float2 x, y, z;
};

// a x b of both genotypes
__device__ __forceinline__ V2 cross2(const V2 &a, const V2 &b) {
    V2 c;
    c.x = fma2(a.y, b.z, neg2(mul2(a.z, b.y)));
    c.y = fma2(a.z, b.x, neg2(mul2(a.x, b.z)));
    c.z = fma2(a.x, b.y, neg2(mul2(a.y, b.x)));
    return c;
}
__device__ __forceinline__ float2 dot2(const V2 &a, const V2 &b) {
    return fma2(a.z, b.z, fma2(a.y, b.y, mul2(a.x, b.x)));
}

// Inputs and outputs of two genotypes searched together (pointers at each one).
struct PairIO {
    const float *genes_in[2];
    float *genes_out[2];
    float *energy[2];
    float *grad[2];
    float *state[2];
    int iters[2];
    int nvalid;   // 1: the second genotype is a copy of the first, not written
    int mode, resume;
    float rho, eps;
};

}  // namespace adgb
