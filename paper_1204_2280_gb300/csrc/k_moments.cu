// k_moments.cu -- multipole moments of every cell (paper Sect. 2,
// "computation of the multipole moments") and the opening radius of the MAC.
//
// Per cell: mass M, centre of mass com and traceless quadrupole
//   Q_ij = sum m (3 y_i y_j - |y|^2 delta_ij),  y = x - com.
// Leaves are summed from their bodies in cell-relative coordinates (offsets
// from the first body, then from the com).  Parents combine their children
// by the parallel-axis theorem,
//   Q_p = sum_k [ Q_k + M_k (3 d_k d_k^T - |d_k|^2 I) ],  d_k = com_k - com_p,
// in a second launch: each thread finishing a cell counts down its parent's
// arrival word and the last internal child to arrive combines the parent
// (no waiting).
// The root of each system (level 0) combines in FP64 about the root cube's
// centre O and shifts to its own com:
//   with e = com_k - O:  M = sum m_k,  com = O + (sum m_k e) / M,
//   Q = sum [Q_k + m_k (3 e e^T - |e|^2 I)] - M (3 s s^T - |s|^2 I),  s = com - O.
// FP64 instructions are few per cycle here (one thread's some 180 took 6 us
// at the end of every combine pass), so the whole warp of the thread that
// completes a root works on it (root_cell).
#include "common.cuh"

namespace bonsai {

__device__ __forceinline__ unsigned compact3(unsigned long long x) {
    x &= 0x1249249249249249ull;
    x = (x ^ (x >> 2)) & 0x10c30c30c30c30c3ull;
    x = (x ^ (x >> 4)) & 0x100f00f00f00f00full;
    x = (x ^ (x >> 8)) & 0x001f0000ff0000ffull;
    x = (x ^ (x >> 16)) & 0x001f00000000ffffull;
    x = (x ^ (x >> 32)) & 0x00000000001fffffull;
    return (unsigned)x;
}

// Geometric centre and side of a cell at `level` of system `sys` whose
// first body has key k.
__device__ __forceinline__ float cell_cube(unsigned long long k, int level, int sys, const DevState *st, float3 &c) {
    unsigned long long pre = key_prefix(k, level);
    float l = ldexpf(st->side[sys], -level);
    const float *mn = st->mn + 3 * sys;
    c.x = fmaf((float)compact3(pre) + 0.5f, l, mn[0]);
    c.y = fmaf((float)compact3(pre >> 1) + 0.5f, l, mn[1]);
    c.z = fmaf((float)compact3(pre >> 2) + 0.5f, l, mn[2]);
    return l;
}

__device__ __forceinline__ float com_offset(float3 com, float3 c) {
    float dx = com.x - c.x, dy = com.y - c.y, dz = com.z - c.z;
    return sqrtf(dx * dx + dy * dy + dz * dz);
}

// (|com - geometric centre|, side) of a cell at `level` of system `sys`
// whose first body has key k.
__device__ float2 cell_delta(unsigned long long k, int level, int sys, float3 com, const DevState *st) {
    float3 c;
    const float l = cell_cube(k, level, sys, st, c);
    return make_float2(com_offset(com, c), l);
}

__device__ __forceinline__ float dist_inf(float3 a, float3 b) {
    return fmaxf(fabsf(a.x - b.x), fmaxf(fabsf(a.y - b.y), fabsf(a.z - b.z)));
}

struct Mom32 { float M, x, y, z, q[6]; };

#ifndef MOM_MINB
#define MOM_MINB 4            // resident 256-thread blocks per SM the launch bounds ask for (5 spills)
#endif
#ifndef MOM_CTHREADS
#define MOM_CTHREADS 128      // combine pass: threads per block
#endif
#ifndef MOM_MINB2
#define MOM_MINB2 6           // combine pass: resident blocks per SM the launch bounds ask for
#endif
#ifndef MOM_CPASYNC
#define MOM_CPASYNC 1         // combine: children's data through asynchronous copies to shared memory
#endif                        // (0: register loads in two round trips, 5-11% slower at 2^20..2^22)
#ifndef MOM_CBLOCKS
#define MOM_CBLOCKS 6         // combine pass: blocks per SM of its persistent grid (32 KB of staging each)
#endif
#ifndef MOM_LB
#define MOM_LB 8              // leaf bodies loaded per round trip (4: 3% slower at 2^22, 16 spills)
#endif

__device__ __forceinline__ unsigned atom_add_acq_rel_gpu(unsigned *p, unsigned v) {
    unsigned old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// The quadrupole arrays hold -Q (negation is exact): the walk consumes it in
// that form, parents and the export negate it back.
__device__ __forceinline__ void store32(int c, const Mom32 &m, float4 *mono, float4 *qa, float2 *qb) {
    mono[c] = make_float4(m.x, m.y, m.z, m.M);
    qa[c] = make_float4(-m.q[0], -m.q[1], -m.q[2], -m.q[3]);
    qb[c] = make_float2(-m.q[4], -m.q[5]);
}

// REFIT (block time steps, between rebuilds): the bodies may have left the
// cells they were sorted into.  Each cell also gets ext = half side of a cube
// about its build-time centre that holds its bodies (at least l/2; a leaf
// from its bodies, a parent as max(l/2, max_k |centre_k - centre|_inf +
// ext_k)), stored with the centre in cext, and delta holds (|com - centre|,
// 2 ext): the opening radius 2 ext / theta + delta then keeps every cell that
// holds a body of a group opened for it (theta < 2 / sqrt(3)).
//
// Two launches.  The leaf pass sums every leaf from its bodies (no atomics,
// no fences), gives every internal cell its arrival word (the number of its
// internal children) and lists the internal cells without any.  The combine
// pass starts at the listed cells (all children leaves, complete since the
// leaf pass) and climbs: a finished cell decrements its parent's word and
// the child that brings it to zero combines the parent.

// 16-byte asynchronous copy global -> shared through L2 (zero fill when
// !valid: nothing is read).
__device__ __forceinline__ void cp_async16(float4 *sdst, const float4 *gsrc, bool valid) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa), "l"(gsrc), "r"(valid ? 16 : 0)
                 : "memory");
}

struct MomArrays {
    const DevState *__restrict__ stc;
    DevState *st;                     // not NULL: reset the walk's queues and totals
    const uint2 *__restrict__ cell_body;
    const uint2 *__restrict__ cell_link;
    const uint8_t *__restrict__ cell_level;
    const uint32_t *__restrict__ cell_parent;
    uint32_t *cell_done;
    const float4 *__restrict__ pos4;
    const unsigned long long *__restrict__ sk;
    const uint8_t *__restrict__ sysid;
    float4 *mono, *qa;
    float2 *qb, *delta;
    float4 *cext;
    bool multi;                       // several systems (else every body is in system 0)
    uint32_t *starts;                 // internal cells whose children are all leaves
    unsigned *nstart;                 // their number
};

// Leaf c (level lev, bodies link.x ..) from its bodies in one pass: mass,
// first and second moments of the offsets u = x - x0 from the first body;
// then with c = s/M the central moments C = S - s c^T and Q = 3C - tr(C) I.
// The offsets are at most the cell size, so nothing cancels beyond FP32
// rounding.
template <bool REFIT>
__device__ __forceinline__ void leaf_finish(unsigned c, int lev, unsigned long long kb, int sysb, float4 x0, float M,
                                            float sx, float sy, float sz, float sxx, float syy, float szz, float sxy,
                                            float sxz, float syz, float3 ctr, float ext, const MomArrays &a);

template <bool REFIT>
__device__ __forceinline__ void leaf_cell(unsigned c, uint2 link, int lev, const MomArrays &a) {
    const unsigned b = link.x, cnt = link.y & ~LEAF_BIT;
    // The first body's key and system with its position (one round trip;
    // loaded after the sums they cost 2% at 2^22 bodies).
    const unsigned long long kb = a.sk[b];
    const int sysb = a.multi ? a.sysid[b] : 0;
    const float4 x0 = a.pos4[b];
    float M = 0.f, sx = 0.f, sy = 0.f, sz = 0.f;
    float sxx = 0.f, syy = 0.f, szz = 0.f, sxy = 0.f, sxz = 0.f, syz = 0.f;
    float3 ctr = make_float3(0.f, 0.f, 0.f);
    float ext = 0.f;
    if (REFIT) ext = 0.5f * cell_cube(kb, lev, sysb, a.stc, ctr);
    // The bodies' loads are issued LB at a time (one round trip per LB
    // bodies instead of one per body); the sums still run in body order.
    constexpr unsigned LB = MOM_LB;
    for (unsigned j0 = b; j0 < b + cnt; j0 += LB) {
        float4 pb[LB];
#pragma unroll
        for (unsigned u = 0; u < LB; u++) pb[u] = j0 + u < b + cnt ? a.pos4[j0 + u] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (unsigned u = 0; u < LB; u++) {
            if (j0 + u >= b + cnt) break;
            const float4 p = pb[u];
            if (REFIT) ext = fmaxf(ext, dist_inf(make_float3(p.x, p.y, p.z), ctr));
            const float ux = p.x - x0.x, uy = p.y - x0.y, uz = p.z - x0.z;
            const float wx = p.w * ux, wy = p.w * uy, wz = p.w * uz;
            M += p.w;
            sx += wx; sy += wy; sz += wz;
            sxx = fmaf(wx, ux, sxx); syy = fmaf(wy, uy, syy); szz = fmaf(wz, uz, szz);
            sxy = fmaf(wx, uy, sxy); sxz = fmaf(wx, uz, sxz); syz = fmaf(wy, uz, syz);
        }
    }
    leaf_finish<REFIT>(c, lev, kb, sysb, x0, M, sx, sy, sz, sxx, syy, szz, sxy, sxz, syz, ctr, ext, a);
}

// A leaf's moments from its sums about the first body x0 (mass, first and
// second moments of the offsets), and its stores.
template <bool REFIT>
__device__ __forceinline__ void leaf_finish(unsigned c, int lev, unsigned long long kb, int sysb, float4 x0, float M,
                                            float sx, float sy, float sz, float sxx, float syy, float szz, float sxy,
                                            float sxz, float syz, float3 ctr, float ext, const MomArrays &a) {
    Mom32 m;
    m.M = M;
    const float inv = M > 0.f ? 1.f / M : 0.f;
    const float cx = sx * inv, cy = sy * inv, cz = sz * inv;
    m.x = x0.x + cx; m.y = x0.y + cy; m.z = x0.z + cz;
    const float Cxx = fmaf(-sx, cx, sxx), Cyy = fmaf(-sy, cy, syy), Czz = fmaf(-sz, cz, szz);
    const float tr = Cxx + Cyy + Czz;
    m.q[0] = 3.f * Cxx - tr; m.q[1] = 3.f * Cyy - tr; m.q[2] = 3.f * Czz - tr;
    m.q[3] = 3.f * fmaf(-sx, cy, sxy); m.q[4] = 3.f * fmaf(-sx, cz, sxz); m.q[5] = 3.f * fmaf(-sy, cz, syz);
    store32(c, m, a.mono, a.qa, a.qb);
    if (REFIT) {
        a.delta[c] = make_float2(com_offset(make_float3(m.x, m.y, m.z), ctr), 2.f * ext);
        a.cext[c] = make_float4(ctr.x, ctr.y, ctr.z, ext);
    } else {
        a.delta[c] = cell_delta(kb, lev, sysb, make_float3(m.x, m.y, m.z), a.stc);
    }
}

// Internal cell c (level lv > 0, children plk.x .. plk.x + plk.y - 1, all
// complete) from its children; kb, sysb: the key and system of a body inside
// it (its key prefix gives the cell's centre).
template <bool REFIT>
__device__ __forceinline__ void combine_cell(unsigned c, int lv, uint2 plk, unsigned long long kb, int sysb,
                                             const MomArrays &a, float4 *stage) {
    const unsigned cb = plk.x, nch = plk.y;
    Mom32 m;
    // Children's moments loaded together (at most 8, unrolled): one
    // round trip to L2 per level instead of one per child.  By the
    // parallel-axis theorem,
    //   Q_p = sum_k [ Q_k + M_k (3 d_k d_k^T - |d_k|^2 I) ],  d_k = com_k - com_p.
    float4 mo[8];
#if MOM_CPASYNC
    // masses and centres and the quadrupoles' first four components
    // land in shared memory by asynchronous copies (no registers held),
    // the last two in registers: one round trip for all of it
    float2 qq2[8];
    if (stage) {
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const unsigned kk = k < (int)nch ? (unsigned)k : 0u;   // an address inside the arrays
            cp_async16(stage + k * MOM_CTHREADS, a.mono + cb + kk, k < (int)nch);
            cp_async16(stage + (8 + k) * MOM_CTHREADS, a.qa + cb + kk, k < (int)nch);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
#pragma unroll
    for (int k = 0; k < 8; k++) qq2[k] = k < (int)nch ? __ldcg(a.qb + cb + k) : make_float2(0.f, 0.f);
    if (stage) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
        for (int k = 0; k < 8; k++) mo[k] = stage[k * MOM_CTHREADS];
    } else {
#pragma unroll
        for (int k = 0; k < 8; k++) mo[k] = k < (int)nch ? __ldcg(a.mono + cb + k) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#else
#pragma unroll
    for (int k = 0; k < 8; k++) mo[k] = k < (int)nch ? __ldcg(a.mono + cb + k) : make_float4(0.f, 0.f, 0.f, 0.f);
#endif
    const float c0x = mo[0].x, c0y = mo[0].y, c0z = mo[0].z;
    float fM = 0.f, ax = 0.f, ay = 0.f, az = 0.f;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        if (k < (int)nch) {
            fM += mo[k].w;
            ax = fmaf(mo[k].w, mo[k].x - c0x, ax);
            ay = fmaf(mo[k].w, mo[k].y - c0y, ay);
            az = fmaf(mo[k].w, mo[k].z - c0z, az);
        }
    }
    const float inv2 = fM > 0.f ? 1.f / fM : 0.f;
    m.M = fM; m.x = c0x + ax * inv2; m.y = c0y + ay * inv2; m.z = c0z + az * inv2;
    for (int i = 0; i < 6; i++) m.q[i] = 0.f;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        if (k < (int)nch) {
#if MOM_CPASYNC
            const float4 q4 = stage ? stage[(8 + k) * MOM_CTHREADS] : __ldcg(a.qa + cb + k);
            const float2 q2 = qq2[k];
#else
            const float4 q4 = __ldcg(a.qa + cb + k);
            const float2 q2 = __ldcg(a.qb + cb + k);
#endif
            const float dx = mo[k].x - m.x, dy = mo[k].y - m.y, dz = mo[k].z - m.z;
            const float d2 = dx * dx + dy * dy + dz * dz;
            m.q[0] += -q4.x + mo[k].w * (3.f * dx * dx - d2);
            m.q[1] += -q4.y + mo[k].w * (3.f * dy * dy - d2);
            m.q[2] += -q4.z + mo[k].w * (3.f * dz * dz - d2);
            m.q[3] += -q4.w + mo[k].w * (3.f * dx * dy);
            m.q[4] += -q2.x + mo[k].w * (3.f * dx * dz);
            m.q[5] += -q2.y + mo[k].w * (3.f * dy * dz);
        }
    }
    store32(c, m, a.mono, a.qa, a.qb);
    if (REFIT) {
        float3 pc;
        float e = 0.5f * cell_cube(kb, lv, sysb, a.stc, pc);
        for (unsigned k = 0; k < nch; k++) {
            const float4 ce = __ldcg(a.cext + cb + k);
            e = fmaxf(e, dist_inf(make_float3(ce.x, ce.y, ce.z), pc) + ce.w);
        }
        a.delta[c] = make_float2(com_offset(make_float3(m.x, m.y, m.z), pc), 2.f * e);
        a.cext[c] = make_float4(pc.x, pc.y, pc.z, e);
    } else {
        a.delta[c] = cell_delta(kb, lv, sysb, make_float3(m.x, m.y, m.z), a.stc);
    }
}

// Root c (children plk.x .. plk.x + plk.y - 1, all complete) by a whole warp;
// t: ten rows of eight in shared memory.  Lane 8 g + k computes child k's
// terms of group g: m and m e, or a diagonal and an off-diagonal component;
// lane i < 10 sums component i over the children in order and finishes it
// (0: mass, 1..3: centre of mass, 4..9: xx yy zz xy xz yz).  About 60 FP64
// instructions a warp; one thread alone, with the children's terms left in
// memory by the threads that finished them, issued three times as many: the
// moments of 4,096 bodies 28 -> 22 us, of 2^20 49 -> 43.
template <bool REFIT>
__device__ __forceinline__ void root_cell(unsigned c, uint2 plk, unsigned long long kb, int sysb, const MomArrays &a,
                                          double (*t)[8], int lane) {
    const unsigned nch = plk.y;
    const int k = lane & 7, g = lane >> 3;
    const unsigned ch = plk.x + (k < (int)nch ? (unsigned)k : 0u);
    float3 o;
    const float l = cell_cube(kb, 0, sysb, a.stc, o);
    const float4 mo = __ldcg(a.mono + ch);
    const float4 qa = __ldcg(a.qa + ch);                 // -(xx, yy, zz, xy)
    const float2 qb = __ldcg(a.qb + ch);                 // -(xz, yz)
    const double M = mo.w, ex = (double)mo.x - o.x, ey = (double)mo.y - o.y, ez = (double)mo.z - o.z;
    if (g == 0) {
        t[0][k] = M; t[1][k] = M * ex; t[2][k] = M * ey; t[3][k] = M * ez;
    } else {
        // g = 1: xx, xy;  2: yy, yz;  3: zz, xz
        const double e2 = ex * ex + ey * ey + ez * ez;
        const double p = g == 1 ? ex : g == 2 ? ey : ez, q = g == 1 ? ey : g == 2 ? ez : ex;
        const float qd = g == 1 ? qa.x : g == 2 ? qa.y : qa.z, qo = g == 1 ? qa.w : g == 2 ? qb.y : qb.x;
        t[3 + g][k] = M * (3 * p * p - e2) - qd;
        t[g == 1 ? 7 : g == 2 ? 9 : 8][k] = M * (3 * p * q) - qo;
    }
    float e = 0.5f * l;
    if (REFIT) {
        const float4 ce = __ldcg(a.cext + ch);
        e = fmaxf(e, dist_inf(make_float3(ce.x, ce.y, ce.z), o) + ce.w);
#pragma unroll
        for (int w = 4; w; w >>= 1) e = fmaxf(e, __shfl_xor_sync(0xffffffffu, e, w));
    }
    __syncwarp();
    double v = 0;
    const int i = lane < 10 ? lane : 0;
    for (unsigned n = 0; n < nch; n++) v += t[i][n];
    const double m0 = __shfl_sync(0xffffffffu, v, 0);
    const double inv = m0 > 0 ? 1.0 / m0 : 0.0;
    const double s = v * inv;                            // lanes 1..3: com - O
    const double sx = __shfl_sync(0xffffffffu, s, 1), sy = __shfl_sync(0xffffffffu, s, 2),
                 sz = __shfl_sync(0xffffffffu, s, 3);
    float r;
    if (lane < 4) {
        r = lane == 0 ? (float)v : (float)((lane == 1 ? o.x : lane == 2 ? o.y : o.z) + s);
    } else {
        const double s2 = sx * sx + sy * sy + sz * sz;
        const double p = lane == 5 || lane == 9 ? sy : lane == 6 ? sz : sx;
        const double q = lane == 4 ? sx : lane == 5 || lane == 7 ? sy : sz;
        r = (float)(v - m0 * (3 * p * q - (lane < 7 ? s2 : 0.0)));
    }
    Mom32 m;
    m.M = __shfl_sync(0xffffffffu, r, 0);
    m.x = __shfl_sync(0xffffffffu, r, 1); m.y = __shfl_sync(0xffffffffu, r, 2); m.z = __shfl_sync(0xffffffffu, r, 3);
#pragma unroll
    for (int n = 0; n < 6; n++) m.q[n] = __shfl_sync(0xffffffffu, r, 4 + n);
    if (lane == 0) {
        store32(c, m, a.mono, a.qa, a.qb);
        a.delta[c] = make_float2(com_offset(make_float3(m.x, m.y, m.z), o), REFIT ? 2.f * e : l);
        if (REFIT) a.cext[c] = make_float4(o.x, o.y, o.z, e);
    }
    __syncwarp();                                        // t is rewritten by the next root
}

// Leaf pass: one thread per cell, from the end of the breadth-first
// numbering.  A leaf sums its bodies; an internal cell writes its arrival
// word, the number of its internal children (contiguous links), and one
// without any is appended to the start list (one atomic per warp, lanes in
// cell order, so the list runs roughly deepest first).
template <bool REFIT>
__global__ void __launch_bounds__(256, MOM_MINB)
k_mom_leaves(MomArrays a) {
    if (a.st && blockIdx.x == 0 && threadIdx.x == 0) {   // the walk that follows starts from empty queues
        a.st->walk_next = 0u; a.st->walk_next2 = 0u;
        a.st->inter[0] = 0ull; a.st->inter[1] = 0ull;
    }
    const unsigned nc = a.stc->ncells;
    if (a.stc->status & ST_TIMEOUT) return;
    const unsigned lane = threadIdx.x & 31u;
    const unsigned lt = (1u << lane) - 1u;
    // every lane of a warp runs the same iterations (the ballot below)
    for (unsigned i0 = blockIdx.x * blockDim.x; i0 < nc; i0 += gridDim.x * blockDim.x) {
        const unsigned i = i0 + threadIdx.x;
        const unsigned c = nc - 1u - i;
        bool start = false;
        if (i < nc) {
            const uint2 link = a.cell_link[c];
            const int lev = a.cell_level[c];
            if (link.y & LEAF_BIT) {
                leaf_cell<REFIT>(c, link, lev, a);
            } else {
                uint2 ch[8];
#pragma unroll
                for (int k = 0; k < 8; k++)
                    ch[k] = k < (int)link.y ? a.cell_link[link.x + k] : make_uint2(0u, LEAF_BIT);
                unsigned ni = 0;
#pragma unroll
                for (int k = 0; k < 8; k++) ni += (ch[k].y & LEAF_BIT) ? 0u : 1u;
                a.cell_done[c] = ni;
                start = ni == 0u;
            }
        }
        const unsigned sm = __ballot_sync(0xffffffffu, start);
        if (sm) {
            unsigned base = 0;
            if (lane == 0) base = atomicAdd(a.nstart, (unsigned)__popc(sm));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (start) a.starts[base + __popc(sm & lt)] = c;
        }
    }
}


// Combine pass (persistent grid over the start list): a listed cell combines
// its children (all leaves), then climbs while it is the last internal child
// of its parent to arrive.  Arrival: release (this cell's moments are visible
// to whoever reads the word after the decrement) and acquire (the last child
// sees every sibling's moments: each sibling's decrement heads a release
// sequence that this read-modify-write extends).  Only the list's cells
// start, so a block is not held by climbs for cells that have nothing to do.
constexpr unsigned MOM_SPREAD = 1024;

template <bool REFIT>
__global__ void __launch_bounds__(MOM_CTHREADS, MOM_MINB2)
k_mom_combine(MomArrays a) {
    if (a.stc->status & ST_TIMEOUT) return;
#if MOM_CPASYNC
    __shared__ float4 s_stage[16 * MOM_CTHREADS];     // per thread: 8 children x (mono, qa)
    float4 *stage = s_stage + threadIdx.x;
#else
    float4 *stage = nullptr;
#endif
    __shared__ double s_root[MOM_CTHREADS / 32][10][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned ns = __ldcg(a.nstart);
    // A warp takes 32 list entries at a time: with one system 32 consecutive
    // ones (dealt out, steps of 2^20 bodies took 0.4% more).  With several
    // systems they are dealt out over MOM_SPREAD warps in runs of G, as long as
    // that many warps allow, so that no warp meets many roots (the first
    // entries are the deepest cells of all systems, and small systems' roots
    // are in the list themselves).  Multipoles of several systems, us, with
    // G = 2 / 4 / 8 / 16 / the rule here (in brackets: runs of 32 and each root
    // by its lane alone):
    //   256 of 30 bodies      18 /  23 /  33 /  51 /  18   (27)
    //   256 of 300            27 /  28 /  32 /  38 /  27   (41)
    //   256 of 4,000          60 /  54 /  51 /  50 /  50   (48)
    //   256 of 16,000        138 / 122 / 112 / 110 / 107  (108)
    //    64 of 16,384         54 /  50 /  50 /  50 /  50   (47)
    //     8 of 200,000        57 /  53 /  51 /  49 /  49   (52)
    const unsigned lg = a.multi ? min(5u, max(1u, 31u - (unsigned)__clz((int)(ns / MOM_SPREAD) | 1))) : 5u;
    const unsigned G = 1u << lg;
    const unsigned runs = max((ns + 31u) / 32u, min((ns + G - 1u) / G, MOM_SPREAD));
    for (unsigned w = blockIdx.x * (MOM_CTHREADS / 32) + warp; w < runs; w += gridDim.x * (MOM_CTHREADS / 32)) {
        const unsigned j = ((w + (lane >> lg) * runs) << lg) + (lane & (G - 1u));
        bool root = false;
        unsigned c = 0u;
        uint2 plk = make_uint2(0u, 0u);
        unsigned long long kb = 0ull;
        int sysb = 0;
        if (j < ns) {
            c = __ldcg(a.starts + j);
            plk = a.cell_link[c];
            int lv = a.cell_level[c];
            unsigned p = lv != 0 ? a.cell_parent[c] : 0u;
            // a body inside the cell: its key prefix gives the centre of the
            // cell and of every ancestor
            const unsigned b = a.cell_body[c].x;
            kb = a.sk[b];
            sysb = a.multi ? a.sysid[b] : 0;
            while (true) {
                root = lv == 0;
                if (root) break;
                combine_cell<REFIT>(c, lv, plk, kb, sysb, a, stage);
                // the parent's link and level and the next parent are loaded
                // with the arrival atomic (the tree is read-only here)
                const uint2 pl = a.cell_link[p];
                const int plv = a.cell_level[p];
                const unsigned gp = plv != 0 ? a.cell_parent[p] : 0u;
                if (atom_add_acq_rel_gpu(&a.cell_done[p], 0xffffffffu) != 1u) break;   // decrement
                c = p; plk = pl; lv = plv; p = gp;
            }
        }
        // A lane that completed a root has acquired its children's moments;
        // the barrier passes that on to the other lanes (votes and shuffles
        // order no memory).
        __syncwarp();
        for (unsigned rm = __ballot_sync(0xffffffffu, root); rm; rm &= rm - 1u) {
            const int src = __ffs(rm) - 1;
            root_cell<REFIT>(__shfl_sync(0xffffffffu, c, src),
                             make_uint2(__shfl_sync(0xffffffffu, plk.x, src), __shfl_sync(0xffffffffu, plk.y, src)),
                             __shfl_sync(0xffffffffu, kb, src), __shfl_sync(0xffffffffu, sysb, src), a, s_root[warp],
                             lane);
        }
    }
}

// Launch size: one thread per cell of the last known cell count (plus an
// eighth), or of a typical count for the leaf size when none is known; a
// grid-stride loop covers a tree that grew beyond it.
static unsigned multipole_blocks(const Ctx &c) {
    long long cells = c.cells_hint > 0 ? c.cells_hint + c.cells_hint / 8 + 1024 : 8 * c.n / c.nleaf + 1024;
    if (cells > c.ccap) cells = c.ccap;
    return (unsigned)((cells + 255) / 256);
}

static MomArrays mom_arrays(Ctx &c, bool refit, bool reset) {
    return MomArrays{c.st, reset ? c.st : nullptr, c.cell_body, c.cell_link, c.cell_level, c.cell_parent, c.cell_done,
                     c.pos4, c.keys, c.sysid, c.mono, c.quadA, c.quadB, c.delta, refit ? c.cext : nullptr, c.nsys > 1,
                     c.cell_start, &c.st->mom_starts};
}

// Both passes: the start list is emptied first (a memset node in a graph).
template <bool REFIT>
static cudaError_t launch_mom(Ctx &c, const MomArrays &a) {
    cudaError_t e = cudaMemsetAsync(a.nstart, 0, sizeof(unsigned), c.stream);
    if (e != cudaSuccess) return e;
    k_mom_leaves<REFIT><<<multipole_blocks(c), 256, 0, c.stream>>>(a);
    k_mom_combine<REFIT><<<c.num_sms * MOM_CBLOCKS, MOM_CTHREADS, 0, c.stream>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_multipoles(Ctx &c, bool reset_walk) {
    return launch_mom<false>(c, mom_arrays(c, false, reset_walk));
}

// Moments of the existing cells at the bodies' current positions (block time
// steps between rebuilds), with each cell's cube enlarged to hold its bodies.
cudaError_t launch_multipoles_refit(Ctx &c) {
    return launch_mom<true>(c, mom_arrays(c, true, false));
}

// cext[c] = (geometric centre, l / 2) of every cell from its first body's
// key: the cubes the neighbour search tests (the bodies lie in them right
// after a build).
__global__ void k_cell_cubes(const DevState *__restrict__ st, const uint2 *__restrict__ cell_body,
                             const uint8_t *__restrict__ cell_level, const unsigned long long *__restrict__ sk,
                             const uint8_t *__restrict__ sysid, float4 *cext) {
    const unsigned nc = st->ncells;
    for (unsigned c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
        const unsigned b = cell_body[c].x;
        float3 ctr;
        const float l = cell_cube(sk[b], cell_level[c], sysid[b], st, ctr);
        cext[c] = make_float4(ctr.x, ctr.y, ctr.z, 0.5f * l);
    }
}

cudaError_t launch_cell_cubes(Ctx &c) {
    const unsigned grid = (unsigned)min((c.ccap + 255) / 256, (long long)c.num_sms * 8);
    k_cell_cubes<<<grid, 256, 0, c.stream>>>(c.st, c.cell_body, c.cell_level, c.keys, c.sysid, c.cext);
    return cudaGetLastError();
}

}  // namespace bonsai
