// k_judge.cu -- direct summation on a sample of bodies: the labels of the
// learned correction and the per-step judge of its error (paper Sect. 1: the
// O(N^2) method is the exact reference the tree approximates).
//
// For T target bodies (sorted positions) the softened acceleration from all N
// bodies: sources are streamed through shared memory in
// tiles, each tile summed in FP32 and added with Kahan compensation; the
// source range is split over blocks and the partial sums are added in FP32
// with Kahan compensation too (FP64 on the GPU is kept to the root
// multipoles and the energy diagnostics).
// Tiles run on packed FP32x2 arithmetic, two targets per thread.
// The judge then ranks the relative errors of the current accelerations at
// the targets and compares their 99th percentile with a budget.
#include <algorithm>

#include "common.cuh"

namespace bonsai {

#ifndef DS_PAIRS
#define DS_PAIRS 2                     // packed target pairs per thread (1: 2% slower)
#endif
constexpr int DS_THREADS = 128;        // threads per block, 2 DS_PAIRS targets each
constexpr int DS_TILE = 256;           // sources per shared tile

__device__ __forceinline__ void kadd(float &s, float &c, float v) {
    float y = __fsub_rn(v, c);
    float t = __fadd_rn(s, y);
    c = __fsub_rn(__fsub_rn(t, s), y);
    s = t;
}

// Partial sums of split blockIdx.y over sources [chunk*y, chunk*(y+1)).
// Each thread owns 2 DS_PAIRS targets, k + i DS_THREADS (i < 2 DS_PAIRS),
// as DS_PAIRS packed FP32x2 operands; the tile holds every source twice per
// component ((x, x, y, y), (z, z, m, m)), so two broadcast loads feed
// 12 DS_PAIRS packed operations.  Per target the arithmetic and its order
// are those of one scalar loop over the sources.  A non-null gate that
// reads 0 skips the work (all kernels of this file).
__global__ void __launch_bounds__(DS_THREADS)
k_direct_partial(const float4 *__restrict__ pos4, int n, const uint32_t *__restrict__ targets, int ntar,
                 float eps2, int chunk, float4 *partial, const unsigned *__restrict__ gate) {
    if (gate && *gate == 0u) return;
    constexpr int P = DS_PAIRS, TT = 2 * DS_PAIRS;
    __shared__ float4 tile[2 * DS_TILE];
    int kk[TT];
    bool live[TT];
    float2 nx[P], ny[P], nz[P];
#pragma unroll
    for (int i = 0; i < TT; i++) {
        kk[i] = blockIdx.x * TT * DS_THREADS + i * DS_THREADS + threadIdx.x;
        live[i] = kk[i] < ntar;
    }
#pragma unroll
    for (int q = 0; q < P; q++) {
        const float4 m0 = live[2 * q] ? pos4[targets[kk[2 * q]]] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 m1 = live[2 * q + 1] ? pos4[targets[kk[2 * q + 1]]] : make_float4(0.f, 0.f, 0.f, 0.f);
        nx[q] = make_float2(-m0.x, -m1.x); ny[q] = make_float2(-m0.y, -m1.y); nz[q] = make_float2(-m0.z, -m1.z);
    }
    const float2 e2 = make_float2(eps2, eps2);
    float ax[TT], ay[TT], az[TT], cx[TT], cy[TT], cz[TT];
#pragma unroll
    for (int i = 0; i < TT; i++) ax[i] = ay[i] = az[i] = cx[i] = cy[i] = cz[i] = 0.f;
    const int s0 = blockIdx.y * chunk, s1 = min(n, s0 + chunk);
    for (int b = s0; b < s1; b += DS_TILE) {
        __syncthreads();
        for (int i = threadIdx.x; i < DS_TILE; i += DS_THREADS) {
            const float4 v = b + i < s1 ? pos4[b + i] : make_float4(1e18f, 1e18f, 1e18f, 0.f);
            tile[2 * i] = make_float4(v.x, v.x, v.y, v.y);
            tile[2 * i + 1] = make_float4(v.z, v.z, v.w, v.w);
        }
        __syncthreads();
        float2 px[P], py[P], pz[P];
#pragma unroll
        for (int q = 0; q < P; q++) px[q] = py[q] = pz[q] = make_float2(0.f, 0.f);
#pragma unroll 8
        for (int j = 0; j < DS_TILE; j++) {
            const float4 u = tile[2 * j], w = tile[2 * j + 1];
#pragma unroll
            for (int q = 0; q < P; q++) {
                const float2 dx = __fadd2_rn(make_float2(u.x, u.y), nx[q]);
                const float2 dy = __fadd2_rn(make_float2(u.z, u.w), ny[q]);
                const float2 dz = __fadd2_rn(make_float2(w.x, w.y), nz[q]);
                const float2 r2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __ffma2_rn(dx, dx, e2)));
                const float2 rinv = make_float2(rsqrt_mufu(r2.x), rsqrt_mufu(r2.y));
                const float2 mr = __fmul2_rn(make_float2(w.z, w.w), rinv);
                const float2 mr3 = __fmul2_rn(__fmul2_rn(mr, rinv), rinv);
                px[q] = __ffma2_rn(mr3, dx, px[q]);
                py[q] = __ffma2_rn(mr3, dy, py[q]);
                pz[q] = __ffma2_rn(mr3, dz, pz[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < P; q++) {
            kadd(ax[2 * q], cx[2 * q], px[q].x); kadd(ay[2 * q], cy[2 * q], py[q].x);
            kadd(az[2 * q], cz[2 * q], pz[q].x);
            kadd(ax[2 * q + 1], cx[2 * q + 1], px[q].y); kadd(ay[2 * q + 1], cy[2 * q + 1], py[q].y);
            kadd(az[2 * q + 1], cz[2 * q + 1], pz[q].y);
        }
    }
#pragma unroll
    for (int i = 0; i < TT; i++)
        if (live[i])
            partial[(size_t)blockIdx.y * ntar + kk[i]] =
                make_float4(ax[i] - cx[i], ay[i] - cy[i], az[i] - cz[i], 0.f);
}

// Sum the splits in order with Kahan compensation (FP32); 16 splits' loads in
// flight per thread (one at a time: 36 us for 128 splits of 4096 targets).
constexpr int RED_THREADS = 64;
__global__ void __launch_bounds__(RED_THREADS)
k_direct_reduce(int ntar, int nsplit, const float4 *__restrict__ partial, float4 *out,
                const unsigned *__restrict__ gate) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= ntar || (gate && *gate == 0u)) return;
    float ax = 0.f, ay = 0.f, az = 0.f, cx = 0.f, cy = 0.f, cz = 0.f;
    for (int y0 = 0; y0 < nsplit; y0 += 16) {
        float4 p[16];
#pragma unroll
        for (int q = 0; q < 16; q++)
            p[q] = y0 + q < nsplit ? partial[(size_t)(y0 + q) * ntar + k] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < 16; q++)
            if (y0 + q < nsplit) { kadd(ax, cx, p[q].x); kadd(ay, cy, p[q].y); kadd(az, cz, p[q].z); }
    }
    out[k] = make_float4(ax - cx, ay - cy, az - cz, 0.f);
}

// Source splits: as many as fill the GPU's resident blocks once (at most
// nsplit), so that no half-empty second wave follows (128 splits of 4096
// targets by 256 were 2048 blocks, 1.35 waves).  4096 targets, 2^20 sources:
// 1837 us with that, one target pair per thread and the potential, which
// nothing reads, summed too; 1746 us in one wave without it; 1705 us with two
// pairs per thread, half the shared-memory reads.
cudaError_t launch_direct(Ctx &c, const uint32_t *targets, int ntar, float eps, float4 *partial,
                          int nsplit, float4 *out, const unsigned *gate) {
    const int n = (int)c.n;
    static int occ[MAX_DEVICES] = {};
    if (c.device < 0 || c.device >= MAX_DEVICES) return cudaErrorInvalidDevice;
    if (occ[c.device] == 0) {
        int per = 0;
        const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_direct_partial, DS_THREADS, 0);
        if (e != cudaSuccess) return e;
        occ[c.device] = per < 1 ? 1 : per;
    }
    const int gx = (ntar + 2 * DS_PAIRS * DS_THREADS - 1) / (2 * DS_PAIRS * DS_THREADS);
    const int want = std::min(nsplit, std::max(1, c.num_sms * occ[c.device] / gx));
    const int chunk = ((n + want - 1) / want + DS_TILE - 1) / DS_TILE * DS_TILE;
    const int used = (n + chunk - 1) / chunk;
    k_direct_partial<<<dim3(gx, used), DS_THREADS, 0, c.stream>>>(c.pos4, n, targets, ntar, eps * eps, chunk, partial,
                                                                 gate);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_direct_reduce<<<(ntar + RED_THREADS - 1) / RED_THREADS, RED_THREADS, 0, c.stream>>>(ntar, used, partial, out,
                                                                                          gate);
    return cudaGetLastError();
}

// Judge: relative errors |a - a_direct| / |a_direct| at the targets, their
// 99th percentile (linear interpolation between order statistics, as numpy's
// default), and the fallback flag p99 > budget (where asked for).  One block of 1024 threads;
// the two order statistics by bisection on the errors' bits (non-negative
// floats order as their bits), one block count per bit: 38 us with a bitonic
// sort of the 4096 errors, 18 us here.  An error that is not finite (forces
// that a diverged network made NaN) ranks as infinite, above every other and
// below the places of absent targets, so that p99 is over every finite budget.
// Skipped by the gate, it leaves the last judgement (p99 and flag) in place.
__global__ void __launch_bounds__(1024)
k_judge_p99(const float4 *__restrict__ acc4, const uint32_t *__restrict__ targets, int ntar,
            const float4 *__restrict__ direct, float budget, float *p99_out, unsigned *fallback,
            const unsigned *__restrict__ gate) {
    if (gate && *gate == 0u) return;
    constexpr int PER = JUDGE_MAX / 1024;
    __shared__ unsigned s_next;
    unsigned v[PER];                              // bits of this thread's errors
#pragma unroll
    for (int k = 0; k < PER; k++) {
        const int i = threadIdx.x + k * 1024;
        v[k] = 0x7fffffffu;
        if (i < ntar) {
            const float4 a = acc4[targets[i]], d = direct[i];
            const float ex = a.x - d.x, ey = a.y - d.y, ez = a.z - d.z;
            const float en = sqrtf(ex * ex + ey * ey + ez * ez);
            const float dn = sqrtf(d.x * d.x + d.y * d.y + d.z * d.z);
            const float e = dn == 0.f && en < INFINITY ? 0.f : en / dn;
            v[k] = __float_as_uint(e < INFINITY ? e : INFINITY);
        }
    }
    if (threadIdx.x == 0) s_next = 0xffffffffu;
    auto at_most = [&](unsigned x) {              // errors <= x, block-wide
        int c = 0;
#pragma unroll
        for (int k = 0; k < PER; k++) c += __syncthreads_count(v[k] <= x);
        return c;
    };
    const float pos = 0.99f * (float)(ntar - 1);
    const int i0 = (int)pos;
    const int i1 = min(i0 + 1, ntar - 1);
    unsigned lo = 0u, hi = 0x7fffffffu;           // smallest value with at least i0 + 1 errors up to it
    while (lo < hi) {
        const unsigned mid = lo + ((hi - lo) >> 1);
        if (at_most(mid) >= i0 + 1) hi = mid; else lo = mid + 1u;
    }
    const bool tie = at_most(lo) >= i1 + 1;       // the next order statistic is equal
#pragma unroll
    for (int k = 0; k < PER; k++)
        if (v[k] > lo) atomicMin(&s_next, v[k]);
    __syncthreads();
    if (threadIdx.x == 0) {
        const float v0 = __uint_as_float(lo), v1 = tie ? v0 : __uint_as_float(s_next);
        const float f = pos - (float)i0;
        const float p99 = v1 < INFINITY ? v0 + f * (v1 - v0) : f > 0.f ? v1 : v0;
        *p99_out = p99;
        if (fallback) *fallback = p99 <= budget ? 0u : 1u;
    }
}

// The judgement of the learned path (p99, fallback by budget; skipped by the
// gate).
cudaError_t launch_judge(Ctx &c, const uint32_t *targets, int ntar, const float4 *direct, float budget,
                         const unsigned *gate) {
    k_judge_p99<<<1, 1024, 0, c.stream>>>(c.acc4, targets, ntar, direct, budget, &c.st->judge_p99, &c.st->fallback,
                                          gate);
    return cudaGetLastError();
}

// The p99 of the current accelerations alone: the learned path's judgement
// stays.
cudaError_t launch_judge_own(Ctx &c, const uint32_t *targets, int ntar, const float4 *direct) {
    k_judge_p99<<<1, 1024, 0, c.stream>>>(c.acc4, targets, ntar, direct, 0.f, &c.st->own_p99, nullptr, nullptr);
    return cudaGetLastError();
}

}  // namespace bonsai
