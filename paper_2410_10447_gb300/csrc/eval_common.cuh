// What the scoring / local-search kernels share: rotations of the torsion
// walk, the trilinear grid terms, and a block's set-up for the tcgen05
// reduction.
#pragma once

#include "adgb_internal.cuh"
#include "reduce.cuh"

namespace adgb {

constexpr float PI_F = 3.14159265358979f;
constexpr int SC_ROT = ADGB_MAX_TORS;  // sc[] slots after the torsions: phi, theta, alpha

__device__ __forceinline__ float3 cross3(float3 a, float3 b) {
    return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}

// p += s (k x v) + omc (k x (k x v)), v = p - b: rotation by the angle with
// sin = s, 1 - cos = omc about the axis k through b.  Exact at s = omc = 0.
__device__ __forceinline__ void rotate_about(float3 &p, float4 k4, float4 b4, float2 c) {
    const float3 k = make_float3(k4.x, k4.y, k4.z);
    const float3 v = make_float3(p.x - b4.x, p.y - b4.y, p.z - b4.z);
    const float3 kv = cross3(k, v);
    const float3 kkv = cross3(k, kv);
    p.x += c.x * kv.x + c.y * kkv.x;
    p.y += c.x * kv.y + c.y * kkv.y;
    p.z += c.x * kv.z + c.y * kkv.z;
}

// Grid cell of a point: clamped onto the grid, cell origin index, fractional
// position, inside flags, and the out-of-grid penalty and its gradient.
struct CellPos {
    size_t cell;
    float f[3], gout[3], pen;
    bool ins[3];
};

__device__ __forceinline__ CellPos locate(const RecDev &R, float3 x) {
    const float xs[3] = {x.x, x.y, x.z};
    const int n[3] = {R.nx, R.ny, R.nz};
    CellPos c;
    c.pen = 0.f;
    int i0[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const float xc = fminf(fmaxf(xs[d], R.lo[d]), R.hi[d]);
        c.ins[d] = xs[d] >= R.lo[d] && xs[d] <= R.hi[d];
        const float dd = xs[d] - xc;
        c.pen += dd * dd;
        c.gout[d] = 2.f * ADGB_W_OUT * dd;
        const float u = (xc - R.lo[d]) * R.inv_h;
        int k = (int)u;  // u >= 0
        k = k > n[d] - 2 ? n[d] - 2 : k;
        i0[d] = k;
        c.f[d] = u - (float)k;
    }
    c.cell = ((size_t)i0[2] * (R.ny - 1) + i0[1]) * (R.nx - 1) + i0[0];
    return c;
}

// Intermolecular term of one atom from its cell's corner values (type map
// t0/t1, e map e0/e1, d map d0/d1; corner c = cx + 2 cy + 4 cz): the type's
// map plus q times e plus |q| times d, trilinearly interpolated at the point
// clamped onto the grid; a point outside pays W_OUT times its squared
// distance to the grid.
__device__ __forceinline__ float inter_from_corners(const RecDev &R, const CellPos &c, float q,
                                                    float4 t0, float4 t1, float4 e0, float4 e1,
                                                    float4 d0, float4 d1, float3 &g) {
    const float aq = fabsf(q);
    const float w0 = t0.x + q * e0.x + aq * d0.x, w1 = t0.y + q * e0.y + aq * d0.y;
    const float w2 = t0.z + q * e0.z + aq * d0.z, w3 = t0.w + q * e0.w + aq * d0.w;
    const float w4 = t1.x + q * e1.x + aq * d1.x, w5 = t1.y + q * e1.y + aq * d1.y;
    const float w6 = t1.z + q * e1.z + aq * d1.z, w7 = t1.w + q * e1.w + aq * d1.w;
    const float fx = c.f[0], fy = c.f[1], fz = c.f[2];
    const float x00 = w1 - w0, x10 = w3 - w2, x01 = w5 - w4, x11 = w7 - w6;
    const float c00 = w0 + fx * x00, c10 = w2 + fx * x10;
    const float c01 = w4 + fx * x01, c11 = w6 + fx * x11;
    const float y0 = c10 - c00, y1 = c11 - c01;
    const float c0 = c00 + fy * y0, c1 = c01 + fy * y1;
    const float val = c0 + fz * (c1 - c0);
    const float dx0 = x00 + fy * (x10 - x00), dx1 = x01 + fy * (x11 - x01);
    const float dfx = dx0 + fz * (dx1 - dx0);
    const float dfy = y0 + fz * (y1 - y0);
    const float dfz = c1 - c0;
    g.x = (c.ins[0] ? dfx * R.inv_h : 0.f) + c.gout[0];
    g.y = (c.ins[1] ? dfy * R.inv_h : 0.f) + c.gout[1];
    g.z = (c.ins[2] ? dfz * R.inv_h : 0.f) + c.gout[2];
    return val + ADGB_W_OUT * c.pen;
}

__device__ __forceinline__ const float4 *cell_ptr(const RecDev &R, size_t cell) {
    return reinterpret_cast<const float4 *>(R.cells + cell * (size_t)R.M * 8);
}

// Grid term read straight from global memory (L2).
__device__ __forceinline__ float inter_atom(const RecDev &R, int t, float q, float3 x, float3 &g) {
    const CellPos c = locate(R, x);
    const float4 *cp = cell_ptr(R, c.cell);
    return inter_from_corners(R, c, q, __ldg(cp + 2 * t), __ldg(cp + 2 * t + 1),
                              __ldg(cp + 2 * (R.M - 2)), __ldg(cp + 2 * (R.M - 2) + 1),
                              __ldg(cp + 2 * (R.M - 1)), __ldg(cp + 2 * (R.M - 1) + 1), g);
}

// ------------------------------------------------- tcgen05 block set-up
// The tcgen05 reduction's shared-memory region sits at the front of the
// (1024-byte aligned) dynamic shared memory, before the ligand layout: one
// 2 KB B operand per warp at [0, 8192), the all-ones A operand at
// [8192, 10496), one mbarrier per warp at [10496, 10528) and the TMEM base
// address at [10528, 10532).  A block holds at most 4 warps (128 threads).
// The A operand (128 x 8 TF32) is read with 128-byte strides both ways, so
// its core matrices overlap inside 2304 bytes of ones.
constexpr int TC_B = 0, TC_A = 8192, TC_MBAR = 10496, TC_SLOT = 10528;
constexpr int TC_REGION = 10560;

template <int VAR>
__host__ __device__ constexpr int tc_front() { return VAR == ADGB_REDUCE_TCGEN05 ? TC_REGION : 0; }

__host__ __device__ constexpr int tc_ncols(int warps) {   // 16 D columns a warp
    return 16 * warps <= 32 ? 32 : (16 * warps <= 64 ? 64 : 128);
}

// Allocates the block's TMEM, writes the ones operand and fills `tw` (all
// threads; contains block barriers).  R is the front of the dynamic shared
// memory.
template <int VAR>
__device__ __forceinline__ void tc_begin(unsigned char *R, Tc05Warp &tw) {
    if constexpr (VAR == ADGB_REDUCE_TCGEN05) {
        uint64_t *mb = reinterpret_cast<uint64_t *>(R + TC_MBAR);
        uint32_t *slot = reinterpret_cast<uint32_t *>(R + TC_SLOT);
        const int w = threadIdx.x >> 5, W = blockDim.x >> 5;
        const uint32_t ncols = tc_ncols(W);
        const uint32_t rs = tc05::smem_u32(R);
        uint32_t *ones = reinterpret_cast<uint32_t *>(R + TC_A);
        for (int i = threadIdx.x; i < (TC_MBAR - TC_A) / 4; i += blockDim.x) ones[i] = 0x3F800000u;
        tc05::fence_proxy_async_smem();
        if (w == 0) {
            tc05::alloc(slot, ncols);
            tc05::relinquish();
        }
        if ((int)threadIdx.x < W) tc05::mbar_init(mb + threadIdx.x, 1);
        tc05::fence_before();
        __syncthreads();
        tc05::fence_after();
        const uint32_t taddr = *slot;
        tw.a_desc = tc05::desc_plain(rs + TC_A, 128, 128);
        tw.b_s = rs + TC_B + 2048u * w;
        tw.b = R + TC_B + 2048 * w;
        tw.mbar = mb + w;
        tw.d_col = taddr + 16u * w;
        tw.d_lane = tc05::lane_addr(taddr, w & 3, 16 * w);
        tw.taddr = taddr;
        tw.ncols = ncols;
        tw.phase = 0;
        tw.ok = (rs & 1023u) == 0;   // the swizzled B atoms need 1024-byte alignment
    }
}

// Releases the block's TMEM once every warp's MMAs have completed (all
// threads; a warp whose wait gave up first waits, bounded, once more).
template <int VAR>
__device__ __forceinline__ void tc_end(Tc05Warp &tw) {
    if constexpr (VAR == ADGB_REDUCE_TCGEN05) {
        if (!tw.ok && tw.phase > 0)
            (void)tc05::mbar_wait(tw.mbar, (tw.phase - 1) & 1, TC05_WAIT_LIMIT);
        tc05::fence_before();
        __syncthreads();
        tc05::fence_after();
        if ((threadIdx.x >> 5) == 0) tc05::dealloc(tw.taddr, tw.ncols);
    }
}

// Dynamic shared memory of a launch whose layout needs `layout_bytes` for a
// block of `warps` warps: the tcgen05 variant puts its region in front and
// pads the total so that no more blocks are resident on an SM than its 512
// TMEM columns serve at once (tcgen05.alloc would otherwise wait for a
// resident block to finish).  -1 if the device cannot be asked.
inline int tc_smem_bytes(int layout_bytes, int warps, int variant, int device) {
    if (variant != ADGB_REDUCE_TCGEN05) return layout_bytes;
    const int total = TC_REGION + layout_bytes;
    int sm_smem = 0, reserved = 0;
    if (cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, device) !=
            cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, device) !=
            cudaSuccess)
        return -1;
    const int fit = 512 / tc_ncols(warps);
    const int floor_bytes = sm_smem / (fit + 1) - reserved + 16;
    return total < floor_bytes ? floor_bytes : total;
}

}  // namespace adgb
