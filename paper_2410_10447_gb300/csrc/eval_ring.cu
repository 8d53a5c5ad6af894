// Fused scoring / ADADELTA local search of ligands of more than 32 atoms that
// list enough of their pairs (Sec. 2.1, Sec. 3; Table 1's gpu_gradient_minAD):
// one block of 4 warps searches two genotypes, packed (genotype A in .x, B in
// .y), so that the ligand's pair constants, torsion tree and addresses are read
// and computed once for both.
//
// The intramolecular pairs are swept as a ring (RingShape): a lane holds A
// consecutive atoms of both genotypes in registers, and at step s meets atom
// j = A lane + s of the ring, computing its A pairs with it.  In a step every
// lane's j is another atom, so the reaction on j is added to the warp's own
// copy of the forces in shared memory without atomics: two loads, two stores
// and a warp barrier for A pairs of two genotypes, all of them free of bank
// conflicts (ring_index).  The steps are split over the block's warps (and, for
// small ligands, over two teams of lanes in a warp); every atom's owner then
// sums the copies.  The pair constants come from a table in the order of the
// sweep (coalesced 16-byte loads), zeros for pairs that are not listed, the
// H-bond flag in the sign of A.
//
// What bounds it: from ~90 atoms on, the issue and FMA pipe of the pair terms
// (26 packed and 14 scalar instructions for a pair of two genotypes, 15 more
// for distances, sums and the reaction; 256 atoms: FMA pipe 52%, issue 47%,
// LSU data pipe 37% busy, the rest fixed latencies at 10-15 warps an SM); below
// that, the latency of an evaluation's five barriers, gene threads, torsion walk
// and grid loads (45 atoms, one block an SM: ring 2300 of 6500 cycles, gene
// threads 1000, walk 700, grid 700, torsions 950, atoms' sums 650).  The kernel
// it took over from for these ligands (one genotype a 64- or 128-thread group,
// forces through per-pair slots in shared memory) had its LSU data pipe 73%
// busy at 256 atoms, 46% of the shared-memory wavefronts bank-conflict replays,
// at 107K warp instructions an evaluation; this one issues 40K.  Local search,
// M evaluations/s before -> with the sweep:
// 45 atoms x 1000 genotypes 95 -> 157, 64 x 8000 58 -> 121, 90 x 1500
// 31 -> 87, 128 x 8000 17 -> 53, 160 x 6000 12 -> 38, 256 x 2048 6.2 -> 16.0
// (with 3 or 5 atoms a lane only, no 4, and then 4: 64 x 8000 113 -> 121, 128 x
// 8000 43 -> 52, 256 x 2048 12.1 -> 13.4: idle lanes).  Two steps' pairs
// computed before both reactions are stored, to overlap their chains: 2-5%
// slower (registers).
//
// Per evaluation (block barriers between the steps):
//   1. genes and sin / (1 - cos) of every angle are there (step 6, or the
//      kernel's start, published them);
//   2. a thread an atom and genotype: torsion walk, grid terms, and the sums
//      of (E, g, torque) of the grid terms: pair forces are central and
//      cancel in the rigid-body sums exactly, so they take no part in them;
//   3. ring sweep; 4. atoms' total gradients;
//   5. torsions' moving-set sums (8 lanes a torsion) and the reduction;
//   6. gene gradient, best tracking, ADADELTA and the next angles' sines by
//      the gene threads, a gene and genotype each.
#include <math.h>

#include <algorithm>

#include "adgb_internal.cuh"
#include "eval_common.cuh"
#include "packed.cuh"
#include "pair_term.cuh"
#include "reduce.cuh"

namespace adgb {

namespace {

constexpr unsigned FULL = 0xffffffffu;

// Shared-memory layout of one block: the ligand's constants, then the two
// genotypes' working arrays.  Offsets in bytes, 16-byte aligned.
struct RingSmem {
    int ref, type, frag, tparent, tatoms, taxis, tbref;
    int pxy, pz;        // positions [pos_len]: (xA, xB, yA, yB) and (zA, zB)
    int cxy, cz;        // force copies [copies][copy_len], as the positions
    int gxy, gz;        // atoms' gradients [N], as the positions
    int genes, sc, ggrad, red, stage;
    int ada;            // gene threads' state [MAX_GENES][genotype]: E[g^2], E[d^2], best, Omega
    int total;
    RingShape r;

    __host__ __device__ inline void make(int N, int T, bool mma_stage) {
        r = ring_shape(N);
        auto al16 = [](int x) { return (x + 15) & ~15; };
        const int Tn = T > 0 ? T : 1;
        int o = 0;
        ref = o;     o = al16(o + 16 * N);
        type = o;    o = al16(o + 4 * N);
        frag = o;    o = al16(o + 4 * N);
        tparent = o; o = al16(o + 4 * Tn);
        tatoms = o;  o = al16(o + 16 * Tn);
        taxis = o;   o = al16(o + 16 * Tn);
        tbref = o;   o = al16(o + 16 * Tn);
        const int pe = ring_entries(r.pos_len, r.pos_res), ce = ring_entries(r.copy_len, r.copy_res);
        pxy = o;     o = al16(o + 16 * pe);
        pz = o;      o = al16(o + 8 * pe);
        cxy = o;     o = al16(o + 16 * r.copies * ce);
        cz = o;      o = al16(o + 8 * r.copies * ce);
        gxy = o;     o = al16(o + 16 * N);
        gz = o;      o = al16(o + 8 * N);
        genes = o;   o = al16(o + 8 * MAX_GENES);
        sc = o;      o = al16(o + 16 * (ADGB_MAX_TORS + 4));
        ggrad = o;   o = al16(o + 8 * MAX_GENES);
        red = o;     o = al16(o + 4 * 16 * r.warps);
        ada = o;     o = al16(o + 32 * MAX_GENES);
        stage = o;   o = al16(o + (mma_stage ? 4 * 32 * 12 * r.warps : 0));
        total = o;
    }
};

struct RingArgs {
    RecDev rec;
    LigDev lig;
    RingSmem L;
    const float *genes_in;
    float *genes_out;
    float *energy;
    float *grad;
    float *state;
    const int *iters_pp;
    int n, iters, resume, mode;
    float rho, eps;
};

__device__ __forceinline__ void stage_ring_ligand(unsigned char *sm, const RingSmem &L,
                                                  const LigDev &lig) {
    const int N = lig.n_atoms, T = lig.n_tors;
    float4 *s_ref = reinterpret_cast<float4 *>(sm + L.ref);
    int *s_type = reinterpret_cast<int *>(sm + L.type);
    int *s_frag = reinterpret_cast<int *>(sm + L.frag);
    int *s_tpar = reinterpret_cast<int *>(sm + L.tparent);
    int4 *s_tat = reinterpret_cast<int4 *>(sm + L.tatoms);
    float4 *s_tax = reinterpret_cast<float4 *>(sm + L.taxis);
    float4 *s_tb = reinterpret_cast<float4 *>(sm + L.tbref);
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        s_ref[i] = lig.ref[i];
        s_type[i] = lig.type[i];
        s_frag[i] = lig.frag[i];
    }
    for (int k = threadIdx.x; k < T; k += blockDim.x) {
        s_tpar[k] = lig.tparent[k];
        s_tat[k] = lig.tatoms[k];
        s_tax[k] = lig.taxis[k];
        s_tb[k] = lig.tbref[k];
    }
}

__device__ __forceinline__ V2 load_v2(const float4 *xy, const float2 *z, int i) {
    const float4 a = xy[i];
    return {make_float2(a.x, a.y), make_float2(a.z, a.w), z[i]};
}

// Sums a warp's 8 values of the lane's own genotype (its parity) over the
// lanes of the same parity: reduce-scatter over lane bits 4..2, a butterfly
// over bit 1; lane (c2 c1 c0 0 g) ends with component c of genotype g.
__device__ __forceinline__ float reduce_parity8(float v[8]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int lv = 0; lv < 3; lv++) {
        const int h = 4 >> lv, m = 16 >> lv;
        const bool up = lane & m;
#pragma unroll
        for (int k = 0; k < h; k++) {
            const float send = up ? v[k] : v[k + h];
            const float keep = up ? v[k + h] : v[k];
            v[k] = keep + __shfl_xor_sync(FULL, send, m);
        }
    }
    return v[0] + __shfl_xor_sync(FULL, v[0], 2);
}

// Whole evaluation loop of a block's two genotypes (all threads).
template <int A, int VAR, bool AHEAD>
__device__ __forceinline__ void search_ring(unsigned char *sm, const RingSmem &L, const LigDev &lig,
                                            const RecDev &rec, const PairIO &io, Tc05Warp &tw) {
    const int t = threadIdx.x, TH = blockDim.x, lane = t & 31, warp = t >> 5;
    const int N = lig.n_atoms, T = lig.n_tors, G = 6 + T;
    const RingShape &rs = L.r;
    const float4 *s_ref = reinterpret_cast<const float4 *>(sm + L.ref);
    const int *s_type = reinterpret_cast<const int *>(sm + L.type);
    const int *s_frag = reinterpret_cast<const int *>(sm + L.frag);
    const int *s_tpar = reinterpret_cast<const int *>(sm + L.tparent);
    const int4 *s_tat = reinterpret_cast<const int4 *>(sm + L.tatoms);
    const float4 *s_tax = reinterpret_cast<const float4 *>(sm + L.taxis);
    const float4 *s_tb = reinterpret_cast<const float4 *>(sm + L.tbref);
    float4 *pxy = reinterpret_cast<float4 *>(sm + L.pxy);
    float2 *pz = reinterpret_cast<float2 *>(sm + L.pz);
    float4 *cxy = reinterpret_cast<float4 *>(sm + L.cxy);
    float2 *cz = reinterpret_cast<float2 *>(sm + L.cz);
    float4 *gxy = reinterpret_cast<float4 *>(sm + L.gxy);
    float2 *gz = reinterpret_cast<float2 *>(sm + L.gz);
    float2 *genes_s = reinterpret_cast<float2 *>(sm + L.genes);
    float4 *sc = reinterpret_cast<float4 *>(sm + L.sc);
    float2 *ggrad = reinterpret_cast<float2 *>(sm + L.ggrad);
    float *red = reinterpret_cast<float *>(sm + L.red);   // [warp][genotype][8]
    float *stage = reinterpret_cast<float *>(sm + L.stage) + warp * 32 * 12;

    // Thread t < 2 G: gene jj of genotype gen and its ADADELTA state, kept in
    // shared memory between evaluations (the ring sweep needs the registers).
    // The thread that steps a gene also takes the sine and cosine of its angle
    // and publishes them: one barrier an evaluation less than with a thread a
    // gene for both genotypes, and with the sums over the warps unrolled
    // (step 6) the gene threads' chain is 1450 -> 1000 of an evaluation's 7400
    // cycles (45 atoms, one block an SM).
    const int gen = t & 1;
    const bool gene_thread = t < 2 * G;
    const int jj = min(t >> 1, MAX_GENES - 1);
    float4 *ada = reinterpret_cast<float4 *>(sm + L.ada) + 2 * jj + gen;   // E[g^2], E[d^2], best, Omega
    // publishes the gene and sin / (1 - cos) of its angle (half-angle form:
    // exact zero at a zero angle; phi and theta as (sin, cos) of the angle)
    auto publish = [&](float om) {
        const bool full = jj == 3 || jj == 4;
        float sn, cs;
        sincosf(full ? om : 0.5f * om, &sn, &cs);
        reinterpret_cast<float *>(genes_s)[2 * jj + gen] = om;
        const float2 w = full ? make_float2(sn, cs) : make_float2(2.f * sn * cs, 2.f * sn * sn);
        float2 *sc2 = reinterpret_cast<float2 *>(sc) + gen;
        if (jj >= 6) sc2[2 * (jj - 6)] = w;
        else if (jj >= 3) sc2[2 * (SC_ROT + jj - 3)] = w;
    };
    if (gene_thread) {
        float o, a = 0.f, b = 0.f;
        if (io.resume) {
            const float *st = io.state[gen];
            o = st[jj];
            a = st[G + jj];
            b = st[2 * G + jj];
        } else {
            o = io.genes_in[gen][jj];
        }
        *ada = make_float4(a, b, o, o);
        publish(o);
    }
    float best_e = INFINITY;
    // the lane's place in the ring sweep
    const RingLane rl = ring_lane(rs, warp, lane);
    const int copy_ent = ring_entries(rs.copy_len, rs.copy_res);
    const int copy0 = rl.copy * copy_ent;   // the lane's copy
    auto pos_at = [&](int q) { return ring_index<A>(q, rs.pos_res); };
    auto copy_at = [&](int q) { return ring_index<A>(q, rs.copy_res); };
    const float4 *table = lig.ring + (size_t)warp * rs.steps * A * 32 + lane;
    const int iters = max(io.iters[0], io.iters[1]);

    for (int it = 0; it < iters; it++) {
        __syncthreads();   // 1. the genes and angles are published

        // 2. coordinates and grid terms of the thread's atoms in its genotype
        float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        {
            const float *gs = reinterpret_cast<const float *>(genes_s) + gen;
            const float2 *sc2 = reinterpret_cast<const float2 *>(sc) + gen;   // [2 k + genotype]
            const float3 tr = make_float3(gs[0], gs[2], gs[4]);
            const float2 sphi = sc2[2 * SC_ROT], sth = sc2[2 * SC_ROT + 2], sal = sc2[2 * SC_ROT + 4];
            const float3 u = make_float3(sth.x * sphi.y, sth.x * sphi.x, sth.y);
            // R - I = sin(a) [u]x + (1 - cos(a)) (u u^T - I)
            const float s = sal.x, o = sal.y;
            const float m00 = o * (u.x * u.x - 1.f), m11 = o * (u.y * u.y - 1.f),
                        m22 = o * (u.z * u.z - 1.f);
            const float m01 = o * u.x * u.y - s * u.z, m10 = o * u.x * u.y + s * u.z;
            const float m02 = o * u.x * u.z + s * u.y, m20 = o * u.x * u.z - s * u.y;
            const float m12 = o * u.y * u.z - s * u.x, m21 = o * u.y * u.z + s * u.x;
            for (int i = t >> 1; i < N; i += TH >> 1) {
                const float4 r4 = s_ref[i];
                float3 p = make_float3(r4.x, r4.y, r4.z);
                for (int k = s_frag[i]; k >= 0;) {
                    const int up = s_tpar[k];   // read ahead of the rotation's chain
                    rotate_about(p, s_tax[k], s_tb[k], sc2[2 * k]);
                    k = up;
                }
                float3 x, g;
                x.x = p.x + (m00 * p.x + m01 * p.y + m02 * p.z) + tr.x;
                x.y = p.y + (m10 * p.x + m11 * p.y + m12 * p.z) + tr.y;
                x.z = p.z + (m20 * p.x + m21 * p.y + m22 * p.z) + tr.z;
                float *xyf = reinterpret_cast<float *>(pxy), *zf = reinterpret_cast<float *>(pz);
                auto put = [&](int e) {
                    const int q = pos_at(e);
                    xyf[4 * q + gen] = x.x;
                    xyf[4 * q + 2 + gen] = x.y;
                    zf[2 * q + gen] = x.z;
                };
                for (int q = i; q < rs.pos_len; q += rs.np) put(q);
                if (i == 0)   // the ring's ghosts past the last atom (no listed pairs)
                    for (int a = N; a < rs.np; a++)
                        for (int q = a; q < rs.pos_len; q += rs.np) put(q);
                v[0] += inter_atom(rec, s_type[i], r4.w, x, g);
                float *gxf = reinterpret_cast<float *>(gxy), *gzf = reinterpret_cast<float *>(gz);
                gxf[4 * i + gen] = g.x;
                gxf[4 * i + 2 + gen] = g.y;
                gzf[2 * i + gen] = g.z;
                const float3 d = make_float3(x.x - tr.x, x.y - tr.y, x.z - tr.z);
                v[1] += g.x;
                v[2] += g.y;
                v[3] += g.z;
                v[4] += d.y * g.z - d.z * g.y;
                v[5] += d.z * g.x - d.x * g.z;
                v[6] += d.x * g.y - d.y * g.x;
            }
        }
        // sums of the grid terms (shuffle form: over the warp right away)
        if constexpr (VAR == ADGB_REDUCE_SHFL) {
            const float mine = reduce_parity8(v);
            if ((lane & 2) == 0) red[16 * warp + 8 * gen + (lane >> 2)] = mine;
        }
        // the warp's copies of the forces start from zero
        for (int q = lane; q < rs.teams * copy_ent; q += 32) {
            const int c = warp * rs.teams * copy_ent + q;
            cxy[c] = make_float4(0.f, 0.f, 0.f, 0.f);
            cz[c] = bc(0.f);
        }
        __syncthreads();

        // 3. ring sweep
        float2 e_pair = bc(0.f);
        if (lig.n_pairs > 0) {
            V2 xi[A], fi[A];
#pragma unroll
            for (int a = 0; a < A; a++) {
                xi[a] = load_v2(pxy, pz, pos_at(A * rl.l + a));
                fi[a] = {bc(0.f), bc(0.f), bc(0.f)};
            }
            // AHEAD: the constants of the next step are loaded before this one's
            // terms.  Taken where a block has 254 registers a thread (launches of
            // up to two blocks an SM; 300 genotypes of 256 atoms 9.9 -> 10.6M
            // evaluations/s, of 128 atoms 26.4 -> 27.8); with 168 or 128 the other
            // resident blocks hide the loads (2048 x 256 atoms 15.8 -> 15.7, 6000
            // x 160 37.2 -> 36.4).
            const float4 *tp = table;
            float4 nc[A];
            if constexpr (AHEAD) {
#pragma unroll
                for (int a = 0; a < A; a++) nc[a] = __ldg(tp + 32 * a);
            }
            // atom a l + s0 + st of the ring and its place in the copy
            int pj = pos_at(A * rl.l + rl.s0), cj = copy0 + copy_at(A * rl.l);
#pragma unroll 2
            for (int st = 0; st < rs.steps; st++, tp += A * 32) {
                const V2 xj = load_v2(pxy, pz, A == 4 ? pj : pj + st);
                if constexpr (A == 4) pj += ring_next<A>(rl.s0 + st, rs.pos_res);
                V2 fj = {bc(0.f), bc(0.f), bc(0.f)};
                float4 cc[A];
#pragma unroll
                for (int a = 0; a < A; a++) cc[a] = AHEAD ? nc[a] : __ldg(tp + 32 * a);
                if constexpr (AHEAD) {
                    const float4 *tn = st + 1 < rs.steps ? tp + A * 32 : tp;
#pragma unroll
                    for (int a = 0; a < A; a++) nc[a] = __ldg(tn + 32 * a);
                }
#pragma unroll
                for (int a = 0; a < A; a++) {
                    const float4 pc = cc[a];
                    const bool hb = __float_as_int(pc.x) < 0;
                    // x_i - x_j, exact; as FMAs 0.8% faster here than as adds
                    const float2 m1 = bc(-1.f);
                    const V2 d = {fma2(xj.x, m1, xi[a].x), fma2(xj.y, m1, xi[a].y),
                                  fma2(xj.z, m1, xi[a].z)};
                    const float2 r2 = fma2(d.z, d.z, fma2(d.y, d.y, mul2(d.x, d.x)));
                    float2 ft;
                    const float2 e = pair_terms2(r2, bc(fabsf(pc.x)), bc(pc.y), bc(pc.z), bc(pc.w),
                                                 {hb, hb}, ft);
                    e_pair = add2(e_pair, e);
                    fi[a] = {fma2(ft, d.x, fi[a].x), fma2(ft, d.y, fi[a].y), fma2(ft, d.z, fi[a].z)};
                    fj = {fma2(ft, d.x, fj.x), fma2(ft, d.y, fj.y), fma2(ft, d.z, fj.z)};
                }
                const int ce = A == 4 ? cj : cj + st;
                const V2 c = load_v2(cxy, cz, ce);
                if (rl.active) {
                    const V2 n = {sub2(c.x, fj.x), sub2(c.y, fj.y), sub2(c.z, fj.z)};
                    cxy[ce] = make_float4(n.x.x, n.x.y, n.y.x, n.y.y);
                    cz[ce] = n.z;
                }
                if constexpr (A == 4) cj += ring_next<A>(st, rs.copy_res);
                __syncwarp();   // the next step's slots were other lanes' in this one
            }
            // the lane's own atoms: slot of atom i is i - s0 around the ring
#pragma unroll
            for (int a = 0; a < A; a++) {
                int q = A * rl.l + a - rl.s0;
                if (q < 0) q += rs.np;
                q = copy0 + copy_at(q);
                if (rl.active) {
                    const V2 c = load_v2(cxy, cz, q);
                    const V2 n = {add2(c.x, fi[a].x), add2(c.y, fi[a].y), add2(c.z, fi[a].z)};
                    cxy[q] = make_float4(n.x.x, n.x.y, n.y.x, n.y.y);
                    cz[q] = n.z;
                }
            }
        }
        __syncthreads();

        // 4. atoms' total gradients: grid terms and every copy's pair forces
        if (lig.n_pairs > 0 && T > 0) {
            for (int i = t; i < N; i += TH) {
                V2 g = load_v2(gxy, gz, i);
                for (int c0 = 0; c0 < rs.copies; c0 += RING_WARPS) {
#pragma unroll
                    for (int c = c0; c < c0 + RING_WARPS; c++) {
                        int q = i - 1 - ring_slice(rs, c) * rs.steps;
                        if (q < 0) q += rs.np;
                        const V2 f = load_v2(cxy, cz, c * copy_ent + copy_at(q));
                        g = {add2(g.x, f.x), add2(g.y, f.y), add2(g.z, f.z)};
                        if (q + rs.np < rs.copy_len) {   // at most one more turn (copy_len < 2 np)
                            const V2 h = load_v2(cxy, cz, c * copy_ent + copy_at(q + rs.np));
                            g = {add2(g.x, h.x), add2(g.y, h.y), add2(g.z, h.z)};
                        }
                    }
                }
                gxy[i] = make_float4(g.x.x, g.x.y, g.y.x, g.y.y);
                gz[i] = g.z;
            }
            __syncthreads();
        }

        // 5. torsion gradients, 8 lanes a torsion: a . sum (x - x_b) x g over
        //    the moving atoms (one contiguous range), both genotypes
        for (int k0 = 0; k0 < T; k0 += TH >> 3) {
            const int k = k0 + (t >> 3);
            V2 acc = {bc(0.f), bc(0.f), bc(0.f)};
            int4 ta = make_int4(0, 0, 0, 0);
            V2 xb = acc;
            if (k < T) {
                ta = s_tat[k];
                xb = load_v2(pxy, pz, pos_at(ta.y));
#pragma unroll 1   // (unrolled 2 and 4 times: 1-3% slower)
                for (int i = ta.z + (t & 7); i < ta.w; i += 8) {
                    const V2 g = load_v2(gxy, gz, i), x = load_v2(pxy, pz, pos_at(i));
                    const V2 d = {sub2(x.x, xb.x), sub2(x.y, xb.y), sub2(x.z, xb.z)};
                    const V2 c = cross2(d, g);
                    acc = {add2(acc.x, c.x), add2(acc.y, c.y), add2(acc.z, c.z)};
                }
            }
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) {
                acc.x.x += __shfl_xor_sync(FULL, acc.x.x, off);
                acc.x.y += __shfl_xor_sync(FULL, acc.x.y, off);
                acc.y.x += __shfl_xor_sync(FULL, acc.y.x, off);
                acc.y.y += __shfl_xor_sync(FULL, acc.y.y, off);
                acc.z.x += __shfl_xor_sync(FULL, acc.z.x, off);
                acc.z.y += __shfl_xor_sync(FULL, acc.z.y, off);
            }
            if (k < T && (t & 7) == 0) {
                float2 gk = bc(0.f);
                if (ta.w > ta.z) {
                    const V2 xa = load_v2(pxy, pz, pos_at(ta.x));
                    const V2 ax = {sub2(xb.x, xa.x), sub2(xb.y, xa.y), sub2(xb.z, xa.z)};
                    const float2 l2 = dot2(ax, ax);
                    gk = mul2(dot2(ax, acc), make_float2(rsqrtf(l2.x), rsqrtf(l2.y)));
                }
                ggrad[6 + k] = gk;
            }
        }
        // the pair energies of the lane's own genotype: its own and its
        // partner lane's; in the shuffle form summed over the warp and added to
        // the grid energy, else reduced with the grid sums on the tensor cores
        float ep = gen ? e_pair.y : e_pair.x;
        ep += __shfl_xor_sync(FULL, gen ? e_pair.x : e_pair.y, 1);
        if constexpr (VAR == ADGB_REDUCE_SHFL) {
#pragma unroll
            for (int off = 16; off > 1; off >>= 1) ep += __shfl_xor_sync(FULL, ep, off);
            if (lane < 2) red[16 * warp + 8 * gen] += ep;
        } else {
            v[0] += ep;
#pragma unroll
            for (int g = 0; g < 2; g++) {
                float w[8];
#pragma unroll
                for (int c = 0; c < 8; c++) w[c] = gen == g ? v[c] : 0.f;
                if constexpr (VAR == ADGB_REDUCE_TCGEN05) warp_sum8_tc05(w, tw);
                else warp_sum8<VAR>(w, stage);
                if (lane == 0) {
#pragma unroll
                    for (int c = 0; c < 8; c++) red[16 * warp + 8 * g + c] = w[c];
                }
            }
        }
        // what the gene formulas take from this evaluation's genes, read
        // before the barrier after which they may be rewritten
        const float2 *sc_rot = reinterpret_cast<const float2 *>(sc) + 2 * SC_ROT + gen;
        const float2 c_phi = sc_rot[0], c_th = sc_rot[2], c_al = sc_rot[4];
        __syncthreads();

        // 6. gene gradient, best tracking, ADADELTA; the next evaluation's genes
        if (gene_thread) {
            auto total = [&](int c) {
                float s = red[8 * gen + c];
#pragma unroll
                for (int w = 1; w < RING_WARPS; w++) s = __fadd_rn(s, red[16 * w + 8 * gen + c]);
                return s;
            };
            const float E = total(0);
            float gj;
            if (jj < 6) {
                // d u / d phi or d theta; angular velocity sin(a) du + (1-cos a) u x du
                const float3 u = make_float3(c_th.x * c_phi.y, c_th.x * c_phi.x, c_th.y);
                const bool th = jj == 4;
                const float3 du = make_float3(th ? c_th.y * c_phi.y : -c_th.x * c_phi.x,
                                              th ? c_th.y * c_phi.x : c_th.x * c_phi.y,
                                              th ? -c_th.x : 0.f);
                auto det = [](float p, float q, float r, float s) {   // p q - r s
                    return __fmaf_rn(p, q, -__fmul_rn(r, s));
                };
                const float3 uxd = make_float3(det(u.y, du.z, u.z, du.y), det(u.z, du.x, u.x, du.z),
                                               det(u.x, du.y, u.y, du.x));
                const float3 w = make_float3(__fmaf_rn(c_al.x, du.x, __fmul_rn(c_al.y, uxd.x)),
                                             __fmaf_rn(c_al.x, du.y, __fmul_rn(c_al.y, uxd.y)),
                                             __fmaf_rn(c_al.x, du.z, __fmul_rn(c_al.y, uxd.z)));
                const float3 d = jj == 5 ? u : w;
                const float t0 = total(jj < 3 ? 1 + jj : 4);
                gj = jj < 3 ? t0 : __fmaf_rn(total(6), d.z, __fmaf_rn(total(5), d.y, __fmul_rn(t0, d.x)));
            } else {
                gj = reinterpret_cast<const float *>(ggrad)[2 * jj + gen];
            }
            if (io.mode == MODE_SCORE) {
                if (gen < io.nvalid) {
                    if (jj == 0) io.energy[gen][0] = E;
                    if (io.grad[gen]) io.grad[gen][jj] = gj;
                }
            } else {
                float4 a = *ada;
                if (it < io.iters[gen]) {
                    if (E < best_e) {
                        best_e = E;
                        a.z = a.w;
                    }
                    const float omr = 1.f - io.rho;
                    a.x = __fmaf_rn(io.rho, a.x, __fmul_rn(omr, __fmul_rn(gj, gj)));
                    const float d = __fmul_rn(
                        root_ratio(__fadd_rn(a.y, io.eps), __fadd_rn(a.x, io.eps)), -gj);
                    a.y = __fmaf_rn(io.rho, a.y, __fmul_rn(omr, __fmul_rn(d, d)));
                    float w = __fadd_rn(a.w, d);
                    if (jj >= 6) w -= 2.f * PI_F * floorf((w + PI_F) * (0.5f / PI_F));
                    a.w = w;
                    *ada = a;
                    publish(w);
                }
            }
        }
        if (io.mode == MODE_SCORE) return;
    }
    if (io.mode == MODE_SCORE || !gene_thread || gen >= io.nvalid) return;
    const float4 a = *ada;
    io.genes_out[gen][jj] = a.z;
    if (io.state[gen]) {
        float *st = io.state[gen];
        st[jj] = a.w;
        st[G + jj] = a.x;
        st[2 * G + jj] = a.y;
    }
    if (jj == 0) io.energy[gen][0] = best_e;
}

// Resident blocks of 128 threads an SM the kernels are built for (MB), i.e.
// registers a thread: 2 (254), 3 (168), 4 (128) or, for a = 3, 5 (96, a little
// spilled outside the sweep).  All give the same bits.  A launch that needs no
// more blocks an SM takes the kernel with more registers, whose loads and pair
// chains overlap better (M evaluations/s, shuffle form, 4 -> 3 -> 2 blocks;
// 300 genotypes, one block an SM: 45 atoms 70 -> 73 -> 74, 90 36 -> 40 -> 41,
// 160 16 -> 18 -> 22, 256 7.0 -> 9.0 -> 10.7; 900 genotypes, three, 4 -> 3: 45
// atoms 160 -> 166, 160 32 -> 34).  Larger launches: 5 for a = 3 up to 96 atoms
// (12 000 genotypes of 45 atoms 206 -> 214, of 90 atoms 91.8 -> 92.4), 3 above
// 192 atoms (four atoms a lane over two windows, the most registers a thread:
// times with 4 blocks over those with 3 for 4000 and 8192 genotypes, 64^3 grid
// 1.01 at 193 atoms, 1.02 at 220, 1.03 at 240 and 256, 128^3 grid 1.00-1.02,
// 1.05, 1.07, 1.08; 1500 genotypes 1.12-1.20), else 4 (161 to 192 atoms, as much
// shared memory a block but three atoms a lane: 0.95-0.97; 128 atoms, 8000
// genotypes, 3 -> 4: 52.5 -> 53.2).  Four blocks an SM that do not fit also run
// as 3 (256 atoms, 40 torsions, 1000 genotypes 10.6 -> 12.5).
template <int A, int VAR, int MB>
__global__ void __launch_bounds__(128, MB) eval_ring_kernel(const RingArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *sm = smem_raw + tc_front<VAR>();
    stage_ring_ligand(sm, a.L, a.lig);
    Tc05Warp tw;
    tc_begin<VAR>(smem_raw, tw);
    if constexpr (VAR != ADGB_REDUCE_TCGEN05) wait_for_predecessor();
    __syncthreads();
    const int G = 6 + a.lig.n_tors, p0 = 2 * blockIdx.x;
    PairIO io;
    io.nvalid = min(2, a.n - p0);
#pragma unroll
    for (int g = 0; g < 2; g++) {
        const size_t p = p0 + (g < io.nvalid ? g : 0);
        io.genes_in[g] = a.genes_in ? a.genes_in + p * G : nullptr;
        io.genes_out[g] = a.genes_out ? a.genes_out + p * G : nullptr;
        io.energy[g] = a.energy + p;
        io.grad[g] = a.grad ? a.grad + p * G : nullptr;
        io.state[g] = a.state ? a.state + p * 3 * G : nullptr;
        io.iters[g] = a.mode == MODE_SCORE ? 1 : (a.iters_pp ? a.iters_pp[p] : a.iters);
    }
    io.mode = a.mode;
    io.resume = a.resume;
    io.rho = a.rho;
    io.eps = a.eps;
    search_ring<A, VAR, MB == 2>(sm, a.L, a.lig, a.rec, io, tw);
    tc_end<VAR>(tw);
    if constexpr (VAR != ADGB_REDUCE_TCGEN05) dependents_may_start();
}

// Multi-ligand form (batches): block b searches work item b (up to two
// genotypes of one ligand); the host orders the items longest first and every
// ligand of the launch has this a and number of warps.
template <int A, int VAR>
__global__ void __launch_bounds__(128, 4) eval_ring_items_kernel(const WorkItem *items,
                                                                 const LigDev *ligs,
                                                                 const RecDev *recs) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ RingSmem L;
    unsigned char *sm = smem_raw + tc_front<VAR>();
    const WorkItem w = items[blockIdx.x];
    const LigDev &lig = ligs[w.lig];
    if (threadIdx.x == 0) L.make(lig.n_atoms, lig.n_tors, uses_mma_stage(VAR));
    __syncthreads();
    stage_ring_ligand(sm, L, lig);
    Tc05Warp tw;
    tc_begin<VAR>(smem_raw, tw);
    __syncthreads();
    PairIO io;
    io.nvalid = w.count;
#pragma unroll
    for (int g = 0; g < 2; g++) {
        const int k = g < io.nvalid ? g : 0;
        io.genes_in[g] = w.genes + (size_t)k * w.gstride;
        io.genes_out[g] = w.genes + (size_t)k * w.gstride;
        io.energy[g] = w.energy + k;
        io.grad[g] = nullptr;
        io.state[g] = nullptr;
        io.iters[g] = w.iters ? w.iters[k] : w.iters_all;
    }
    io.mode = MODE_LS;
    io.resume = 0;
    io.rho = w.rho;
    io.eps = w.eps;
    search_ring<A, VAR, false>(sm, L, lig, recs[w.rec], io, tw);
    tc_end<VAR>(tw);
}

template <int A, int VAR, int MB>
cudaError_t launch_ring_t(const RingArgs &a, int threads, int smem, cudaStream_t s) {
    auto k = eval_ring_kernel<A, VAR, MB>;
    const cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    if constexpr (VAR != ADGB_REDUCE_TCGEN05)
        return launch_dependent(k, (a.n + 1) / 2, threads, smem, s, a);
    k<<<(a.n + 1) / 2, threads, smem, s>>>(a);
    return cudaGetLastError();
}

// need: blocks an SM that hold the whole launch at once; fit: blocks whose
// shared memory an SM holds.
template <int A, int VAR>
cudaError_t launch_ring_mb(const RingArgs &a, int need, int fit, int threads, int smem,
                           cudaStream_t s) {
    if constexpr (VAR == ADGB_REDUCE_SHFL) {
        if (need <= 2) return launch_ring_t<A, VAR, 2>(a, threads, smem, s);
        if (need <= 3 || fit <= 3 || (A == 4 && need > 4 && a.L.r.windows > 1))
            return launch_ring_t<A, VAR, 3>(a, threads, smem, s);
    }
    if constexpr (A == 3)
        if (need > 4 && a.lig.n_atoms <= 96) return launch_ring_t<A, VAR, 5>(a, threads, smem, s);
    return launch_ring_t<A, VAR, 4>(a, threads, smem, s);
}

template <int A>
cudaError_t launch_ring_v(const RingArgs &a, int variant, int need, int fit, int threads, int smem,
                          cudaStream_t s) {
    switch (variant) {
        case ADGB_REDUCE_SHFL: return launch_ring_mb<A, ADGB_REDUCE_SHFL>(a, need, fit, threads, smem, s);
        case ADGB_REDUCE_MMA_TF32X2:
            return launch_ring_mb<A, ADGB_REDUCE_MMA_TF32X2>(a, need, fit, threads, smem, s);
        case ADGB_REDUCE_MMA_BF16X3:
            return launch_ring_mb<A, ADGB_REDUCE_MMA_BF16X3>(a, need, fit, threads, smem, s);
        case ADGB_REDUCE_TCGEN05:
            return launch_ring_mb<A, ADGB_REDUCE_TCGEN05>(a, need, fit, threads, smem, s);
    }
    return cudaErrorInvalidValue;
}

template <int A, int VAR>
cudaError_t launch_ring_items_t(const WorkItem *items, int n_items, const LigDev *ligs,
                                const RecDev *recs, int threads, int smem, cudaStream_t s) {
    auto k = eval_ring_items_kernel<A, VAR>;
    const cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    k<<<n_items, threads, smem, s>>>(items, ligs, recs);
    return cudaGetLastError();
}

template <int A>
cudaError_t launch_ring_items_v(const WorkItem *items, int n_items, const LigDev *ligs,
                                const RecDev *recs, int variant, int threads, int smem,
                                cudaStream_t s) {
    switch (variant) {
        case ADGB_REDUCE_SHFL:
            return launch_ring_items_t<A, ADGB_REDUCE_SHFL>(items, n_items, ligs, recs, threads, smem, s);
        case ADGB_REDUCE_MMA_TF32X2:
            return launch_ring_items_t<A, ADGB_REDUCE_MMA_TF32X2>(items, n_items, ligs, recs, threads, smem, s);
        case ADGB_REDUCE_MMA_BF16X3:
            return launch_ring_items_t<A, ADGB_REDUCE_MMA_BF16X3>(items, n_items, ligs, recs, threads, smem, s);
        case ADGB_REDUCE_TCGEN05:
            return launch_ring_items_t<A, ADGB_REDUCE_TCGEN05>(items, n_items, ligs, recs, threads, smem, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

int ring_layout_bytes(int n_atoms, int n_tors, int variant) {
    RingSmem L;
    L.make(n_atoms, n_tors, uses_mma_stage(variant));
    return L.total;
}

cudaError_t launch_eval_ring_items(const WorkItem *items, int n_items, const LigDev *ligs,
                                   const RecDev *recs, int a, int warps, int layout_bytes,
                                   int variant, cudaStream_t s) {
    if (n_items == 0) return cudaSuccess;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const int smem = tc_smem_bytes(layout_bytes, warps, variant, dev);
    if (smem < 0) return cudaErrorInvalidValue;
    if (a == 3) return launch_ring_items_v<3>(items, n_items, ligs, recs, variant, 32 * warps, smem, s);
    if (a == 4) return launch_ring_items_v<4>(items, n_items, ligs, recs, variant, 32 * warps, smem, s);
    return launch_ring_items_v<5>(items, n_items, ligs, recs, variant, 32 * warps, smem, s);
}

cudaError_t launch_eval_ring(const RecDev &rec, const LigDev &lig, const EvalCfg &cfg, int mode,
                             const float *genes_in, float *genes_out, int n, int iters, float rho,
                             float eps, int resume, float *energy, float *grad, float *state,
                             cudaStream_t s, const int *iters_per_pose) {
    if (n == 0) return cudaSuccess;
    RingArgs a;
    a.rec = rec;
    a.lig = lig;
    a.L.make(lig.n_atoms, lig.n_tors, uses_mma_stage(cfg.variant));
    const RingShape &rs = a.L.r;
    a.genes_in = genes_in;
    a.genes_out = genes_out;
    a.energy = energy;
    a.grad = grad;
    a.state = state;
    a.iters_pp = iters_per_pose;
    a.n = n;
    a.iters = iters;
    a.resume = resume;
    a.mode = mode;
    a.rho = rho;
    a.eps = eps;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const int smem = tc_smem_bytes(a.L.total, rs.warps, cfg.variant, dev);
    if (smem < 0) return cudaErrorInvalidValue;
    int sms = 0, per_sm = 0, reserved = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    if (e != cudaSuccess) return e;
    const int fit = per_sm / (smem + reserved);
    const int need = ((n + 1) / 2 + sms - 1) / sms;
    if (rs.a == 3) return launch_ring_v<3>(a, cfg.variant, need, fit, 32 * rs.warps, smem, s);
    if (rs.a == 4) return launch_ring_v<4>(a, cfg.variant, need, fit, 32 * rs.warps, smem, s);
    return launch_ring_v<5>(a, cfg.variant, need, fit, 32 * rs.warps, smem, s);
}

cudaError_t ring_tc_gave_up_async(unsigned int *dst, cudaStream_t s) {
    return cudaMemcpyFromSymbolAsync(dst, g_tc_gave_up, sizeof(unsigned int), 0,
                                     cudaMemcpyDeviceToHost, s);
}

}  // namespace adgb
