// The intramolecular pair term of the scoring function (Sec. 2.1), two terms
// at a time in packed FP32x2 arithmetic (one instruction, two IEEE
// round-to-nearest results), shared by every scoring and local-search kernel.
#pragma once

#include "packed.cuh"

namespace adgb {

constexpr float PT_LOG2E = 1.4426950408889634f;
constexpr float PT_RMIN2 = ADGB_R_MIN * ADGB_R_MIN;
constexpr float PT_INV_SIG2 = 1.0f / (ADGB_DS_SIGMA * ADGB_DS_SIGMA);
constexpr float PT_GAUSS = -0.5f * PT_INV_SIG2 * PT_LOG2E;       // exp(-r^2 / 2 sigma^2) = 2^(PT_GAUSS r^2)
constexpr float PT_DECAY = -MS_LAMBDA * MS_B * PT_LOG2E;         // k exp(-lambda B r) = 2^(PT_DECAY r + log2 k)
constexpr float PT_LOG2K = 2.96049318f;                          // log2(MS_K), MS_K = 7.7839

// Special-function forms without the scaling that guards subnormal operands:
// every operand here is a normal number (r^2 >= 0.25 A^2, the dielectric's
// denominator between 20 and 78.4) or an exponent whose result may flush to
// zero.
__device__ __forceinline__ float ex2_ftz(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_ftz(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// sqrt(a) / sqrt(b), the ADADELTA step's scale, as a / sqrt(a b): one special
// function and no square root (its error, half an ulp of a b under the root,
// that of rsqrt.approx and one rounding, is below that of sqrtf times
// rsqrtf).  Where a b leaves the normal range, the two roots themselves.
__device__ __forceinline__ bool root_ratio_fine(float ab) { return ab > 1e-36f && ab < 1e38f; }
__device__ __forceinline__ float root_ratio(float a, float b) {
    const float ab = __fmul_rn(a, b);
    if (root_ratio_fine(ab)) return __fmul_rn(a, rsqrt_ftz(ab));
    return __fmul_rn(sqrtf(a), rsqrtf(b));
}
// Of two genotypes, each by its own range (neither's bits depend on the
// other); one branch where both are in range.
__device__ __forceinline__ float2 root_ratio2(float2 a, float2 b) {
    const float2 ab = mul2(a, b);
    if (root_ratio_fine(ab.x) && root_ratio_fine(ab.y))
        return mul2(a, make_float2(rsqrt_ftz(ab.x), rsqrt_ftz(ab.y)));
    return make_float2(root_ratio(a.x, b.x), root_ratio(a.y, b.y));
}

// Two pair terms from their squared distances r2 and constants A, B (12-6
// van der Waals A r^-12 - B r^-6, or 12-10 with hb), C = PT_CSCALE w_el 332.06
// q_i q_j and D = w_ds (S_i V_j + S_j V_i).  Returns the energies; ft =
// (dE/dr) / r, so that dE/dx_i = ft (x_i - x_j).
//
// With e = k exp(-lambda B r) the Mehler-Solmajer dielectric A0 + B0 / (1 + e)
// has 1/eps = (1 + e) q, q = 1 / (eps0 + A0 e), and d(1/eps)/dr =
// -lambda B0^2 e q^2: one reciprocal.  The reciprocal is taken of PT_CSCALE
// (eps0 + A0 e), which C undoes and which leaves the factor -lambda B0^2 in
// e q.  Van der Waals as r^-6 (u - b), u = A r^-6, b = B or B r^-4.  r is
// clamped at R_MIN in the singular terms (no force below); the desolvation
// Gaussian takes r itself.
// 26 packed operations and 14 scalar ones, 8 of them special functions, for
// the two terms together.
struct HbSel {
    bool a, b;
};
__device__ __forceinline__ float2 pair_terms2(float2 r2, float2 A, float2 B, float2 C, float2 D,
                                              HbSel hb, float2 &ft) {
    const float2 neg = bc(-1.f);
    const bool la = r2.x >= PT_RMIN2, lb = r2.y >= PT_RMIN2;
    const float2 r2c = make_float2(fmaxf(r2.x, PT_RMIN2), fmaxf(r2.y, PT_RMIN2));
    const float2 rinv = make_float2(rsqrt_ftz(r2c.x), rsqrt_ftz(r2c.y));
    const float2 rc = __fmul2_rn(r2c, rinv);
    const float2 r2i = __fmul2_rn(rinv, rinv);
    const float2 r4i = __fmul2_rn(r2i, r2i);
    const float2 r6i = __fmul2_rn(r4i, r2i);
    const float2 b10 = __fmul2_rn(B, r4i);
    const float2 b = make_float2(hb.a ? b10.x : B.x, hb.b ? b10.y : B.y);
    const float2 m = make_float2(hb.a ? 10.f : 6.f, hb.b ? 10.f : 6.f);
    const float2 u = __fmul2_rn(A, r6i);
    const float2 xe = __ffma2_rn(bc(PT_DECAY), rc, bc(PT_LOG2K));
    const float2 ke = make_float2(ex2_ftz(xe.x), ex2_ftz(xe.y));
    const float2 nden = __ffma2_rn(ke, neg, neg);
    const float2 dn = __ffma2_rn(bc(PT_CSCALE * MS_A), ke, bc(PT_CSCALE * MS_EPS0));
    const float2 q = make_float2(rcp_ftz(dn.x), rcp_ftz(dn.y));
    const float2 qr = __fmul2_rn(__fmul2_rn(C, rinv), q);
    const float2 nel = __fmul2_rn(qr, nden);                    // minus the Coulomb energy
    const float2 w = __fmul2_rn(qr, __fmul2_rn(ke, q));         // its r times d(1/eps)/dr
    const float2 xd = __fmul2_rn(r2, bc(PT_GAUSS));
    const float2 eds = __fmul2_rn(D, make_float2(ex2_ftz(xd.x), ex2_ftz(xd.y)));
    // (dE/dr) / r of the clamped terms: ((r^-6 (m b - 12 u) - eel) / r + w) / r
    const float2 s = __ffma2_rn(r6i, __ffma2_rn(m, b, __fmul2_rn(bc(-12.f), u)), nel);
    const float2 fr = __fmul2_rn(rinv, __ffma2_rn(rinv, s, w));
    ft = __ffma2_rn(eds, bc(-PT_INV_SIG2), make_float2(la ? fr.x : 0.f, lb ? fr.y : 0.f));
    return __ffma2_rn(nel, neg, __ffma2_rn(r6i, __ffma2_rn(b, neg, u), eds));
}

// One pair term: the same operations on one pair.
__device__ __forceinline__ float pair_term1(float r2, float4 pc, bool hb, float &ft) {
    const float r2c = fmaxf(r2, PT_RMIN2);
    const float rinv = rsqrt_ftz(r2c);
    const float rc = __fmul_rn(r2c, rinv);
    const float r2i = __fmul_rn(rinv, rinv);
    const float r4i = __fmul_rn(r2i, r2i);
    const float r6i = __fmul_rn(r4i, r2i);
    const float b = hb ? __fmul_rn(pc.y, r4i) : pc.y;
    const float u = __fmul_rn(pc.x, r6i);
    const float ke = ex2_ftz(__fmaf_rn(PT_DECAY, rc, PT_LOG2K));
    const float nden = __fsub_rn(-1.f, ke);
    const float q = rcp_ftz(__fmaf_rn(PT_CSCALE * MS_A, ke, PT_CSCALE * MS_EPS0));
    const float qr = __fmul_rn(__fmul_rn(pc.z, rinv), q);
    const float nel = __fmul_rn(qr, nden);
    const float w = __fmul_rn(qr, __fmul_rn(ke, q));
    const float eds = __fmul_rn(pc.w, ex2_ftz(__fmul_rn(r2, PT_GAUSS)));
    const float s = __fmaf_rn(r6i, __fmaf_rn(hb ? 10.f : 6.f, b, __fmul_rn(-12.f, u)), nel);
    const float fr = __fmul_rn(rinv, __fmaf_rn(rinv, s, w));
    ft = __fmaf_rn(eds, -PT_INV_SIG2, r2 >= PT_RMIN2 ? fr : 0.f);
    return __fsub_rn(__fmaf_rn(r6i, __fsub_rn(u, b), eds), nel);
}

}  // namespace adgb
