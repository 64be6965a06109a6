// mlp.cu -- the learned far-field correction: a per-body MLP 12 -> 64 -> 64
// -> 3 (ReLU) that predicts, from features the walk already produces, the
// residual between the coarse-theta tree acceleration and the direct sum:
//   y = (a_direct - a_tree) / |a_tree| / ysig,   a_corrected = a_tree + ysig y |a_tree|.
//
// Arithmetic (the same in training and inference): inputs normalised in FP32
// ((x - mu) / sigma), then inputs, weights and hidden activations rounded to
// BF16, products accumulated in FP32, biases FP32.  Inference runs on the
// tensor cores (mma.sync m16n8k16, BF16 x BF16 -> FP32; the accumulator
// layout of one layer is the A-fragment layout of the next, so activations
// never leave registers).  Training: forward and backward of 32-sample tiles
// in FP32 on the same BF16-rounded values, gradients in registers, AdamW on
// FP32 master weights.
//
// The correction is rotation-equivariant: the 12 inputs are invariants of
// the body (log|a_tree|, log(-phi_tree), log(1 + accepted cells) in the level
// bins 0-3, 4-6, 7-9, 10-21, log(1 + body-body interactions), log of the
// group density n_G / (e_G^3 + eps^3), log((d_G + eps)/eps), the offset o of
// the body from its group box's centre as |o| / (d_G / 2) and the cosine
// between o and a_tree, log n_G), and the 3 outputs are the coefficients of
// the residual along a body-local frame: e0 = a_tree/|a_tree|, e1 = the unit
// part of o orthogonal to e0 (the coordinate axis least aligned with e0 when
// o is parallel to e0 or zero), e2 = e0 x e1.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "common.cuh"

namespace bonsai {

// Parameter block layout (FP32 master copy, row-major W[out][in]).
constexpr int OFF_W1 = 0;                       // 64 x 12
constexpr int OFF_B1 = OFF_W1 + MLP_H * MLP_IN;  // 64
constexpr int OFF_W2 = OFF_B1 + MLP_H;           // 64 x 64
constexpr int OFF_B2 = OFF_W2 + MLP_H * MLP_H;   // 64
constexpr int OFF_W3 = OFF_B2 + MLP_H;           // 3 x 64
constexpr int OFF_B3 = OFF_W3 + MLP_OUT * MLP_H; // 3
static_assert(OFF_B3 + MLP_OUT == MLP_NPARAM, "parameter count");

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}

struct Frame {
    float3 e0, e1, e2;
    float an;
};

// The 12 raw (unnormalised) inputs of a body and its local frame, from its
// tree acceleration/potential and its walk features f (FEAT_STRIDE floats).
__device__ __forceinline__ void body_inputs(const float4 a, const float *__restrict__ f, float (&x)[MLP_IN],
                                            Frame &F) {
    const float an = sqrtf(a.x * a.x + a.y * a.y + a.z * a.z);
    F.an = an;
    float3 e0 = an > 0.f ? make_float3(a.x / an, a.y / an, a.z / an) : make_float3(1.f, 0.f, 0.f);
    const float ox = f[7], oy = f[8], oz = f[9];
    const float on = sqrtf(ox * ox + oy * oy + oz * oz);
    const float od = ox * e0.x + oy * e0.y + oz * e0.z;
    float px = ox - od * e0.x, py = oy - od * e0.y, pz = oz - od * e0.z;
    float pn = sqrtf(px * px + py * py + pz * pz);
    if (!(pn > 1e-6f * on && pn > 0.f)) {      // o zero or along e0: least-aligned axis
        const float ax = fabsf(e0.x), ay = fabsf(e0.y), az = fabsf(e0.z);
        const float ux = (ax <= ay && ax <= az) ? 1.f : 0.f;
        const float uy = (ux == 0.f && ay <= az) ? 1.f : 0.f;
        const float uz = (ux == 0.f && uy == 0.f) ? 1.f : 0.f;
        const float ud = ux * e0.x + uy * e0.y + uz * e0.z;
        px = ux - ud * e0.x; py = uy - ud * e0.y; pz = uz - ud * e0.z;
        pn = sqrtf(px * px + py * py + pz * pz);
    }
    const float3 e1 = make_float3(px / pn, py / pn, pz / pn);
    F.e0 = e0;
    F.e1 = e1;
    F.e2 = make_float3(e0.y * e1.z - e0.z * e1.y, e0.z * e1.x - e0.x * e1.z, e0.x * e1.y - e0.y * e1.x);
    const float diag = f[11];
    x[0] = logf(fmaxf(an, 1e-30f));
    x[1] = logf(fmaxf(-a.w, 1e-30f));
#pragma unroll
    for (int k = 0; k < 7; k++) x[2 + k] = f[k];
    x[9] = diag > 0.f ? on / (0.5f * diag) : 0.f;
    x[10] = on > 0.f ? od / on : 0.f;
    x[11] = f[10];
}

// The 12 inputs of a body, normalised (FP32, before BF16 rounding).
__device__ __forceinline__ void body_features(const float4 a, const float *__restrict__ wf,
                                              const float *__restrict__ norm, float (&x)[MLP_IN], Frame &F) {
    body_inputs(a, wf, x, F);
#pragma unroll
    for (int k = 0; k < MLP_IN; k++) x[k] = (x[k] - norm[k]) / norm[MLP_IN + k];
}

// ---------------------------------------------------------------------------
// Inference on tensor cores.  One warp per 32 bodies: every lane forms the
// inputs and the frame of its own body, the two 16-row halves share each
// weight fragment read from shared memory, whose rows are padded so that the
// eight rows of a fragment fall in different banks.  Bound: the per-body
// input arithmetic (two logarithms, four roots, ten divisions) and latency.
// With 16 lanes forming inputs, rows of 32 words (eight-way conflicts on
// every weight read) and the frames in shared memory 2^20 bodies took 191 us,
// 62 us now.
// ---------------------------------------------------------------------------
constexpr int INF_WARPS = 4;

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Weights as BF16 pairs in shared memory: W1 64 x 16 (inputs padded to 16),
// W2 64 x 64, W3 8 x 64 (outputs padded to 8); row n holds W[n][k..].
constexpr int LD1 = 12, LD2 = 36;   // row strides in words: 12 g + t and 36 g + t are 32 different banks
struct InfShared {
    uint32_t w1[MLP_H * LD1];
    uint32_t w2[MLP_H * LD2];
    uint32_t w3[8 * LD2];
    float b1[MLP_H], b2[MLP_H], b3[8];
    float norm[2 * MLP_IN], ysig;
    float xs[INF_WARPS][32][17];
    float ys[INF_WARPS][32][5];
};

__device__ void stage_weights(InfShared &S, const float *__restrict__ P, const float *__restrict__ norm) {
    const int tid = threadIdx.x;
    for (int i = tid; i < MLP_H * 8; i += blockDim.x) {
        const int r = i / 8, c = 2 * (i % 8);
        const float a = c < MLP_IN ? P[OFF_W1 + r * MLP_IN + c] : 0.f;
        const float b = c + 1 < MLP_IN ? P[OFF_W1 + r * MLP_IN + c + 1] : 0.f;
        S.w1[r * LD1 + i % 8] = pack_bf16(a, b);
    }
#pragma unroll 8
    for (int i = tid; i < MLP_H * 32; i += blockDim.x) {
        const int r = i / 32, c = 2 * (i % 32);
        S.w2[r * LD2 + i % 32] = pack_bf16(P[OFF_W2 + r * MLP_H + c], P[OFF_W2 + r * MLP_H + c + 1]);
    }
    for (int i = tid; i < 8 * 32; i += blockDim.x) {
        const int r = i / 32, c = 2 * (i % 32);
        S.w3[r * LD2 + i % 32] = r < MLP_OUT ? pack_bf16(P[OFF_W3 + r * MLP_H + c], P[OFF_W3 + r * MLP_H + c + 1]) : 0u;
    }
    for (int i = tid; i < MLP_H; i += blockDim.x) { S.b1[i] = P[OFF_B1 + i]; S.b2[i] = P[OFF_B2 + i]; }
    if (tid < 8) S.b3[tid] = tid < MLP_OUT ? P[OFF_B3 + tid] : 0.f;
    if (tid < 2 * MLP_IN) S.norm[tid] = norm[tid];
    if (tid == 0) S.ysig = norm[2 * MLP_IN];
}

__device__ __forceinline__ void relu_pack(const float (&h)[8][4], uint32_t (&a2)[4][4]) {
#pragma unroll
    for (int kc = 0; kc < 4; kc++) {
        a2[kc][0] = pack_bf16(fmaxf(h[2 * kc][0], 0.f), fmaxf(h[2 * kc][1], 0.f));
        a2[kc][1] = pack_bf16(fmaxf(h[2 * kc][2], 0.f), fmaxf(h[2 * kc][3], 0.f));
        a2[kc][2] = pack_bf16(fmaxf(h[2 * kc + 1][0], 0.f), fmaxf(h[2 * kc + 1][1], 0.f));
        a2[kc][3] = pack_bf16(fmaxf(h[2 * kc + 1][2], 0.f), fmaxf(h[2 * kc + 1][3], 0.f));
    }
}

// Forward of 32 rows (normalised inputs xs[32][<=16]) on the tensor cores;
// the raw outputs land in ys[32][0..2].  Whole warp.
__device__ __forceinline__ void mma_forward32(const InfShared &S, const float (*xs)[17], float (*ys)[5], int lane) {
    const int g = lane >> 2, t = lane & 3;
    uint32_t a[2][4], a2[2][4][4];
    float h[2][8][4];
#pragma unroll
    for (int r = 0; r < 2; r++) {
        const float *x0 = xs[16 * r + g], *x1 = xs[16 * r + g + 8];
        a[r][0] = pack_bf16(x0[2 * t], x0[2 * t + 1]); a[r][1] = pack_bf16(x1[2 * t], x1[2 * t + 1]);
        a[r][2] = pack_bf16(x0[2 * t + 8], x0[2 * t + 9]); a[r][3] = pack_bf16(x1[2 * t + 8], x1[2 * t + 9]);
    }
#pragma unroll
    for (int j = 0; j < 8; j++) {                 // layer 1: 8 n-tiles of 8 hidden units
        const int col = 8 * j + 2 * t, row = 8 * j + g;
        const float c0 = S.b1[col], c1 = S.b1[col + 1];
        const uint32_t w0 = S.w1[row * LD1 + t], w1 = S.w1[row * LD1 + t + 4];
#pragma unroll
        for (int r = 0; r < 2; r++) {
            h[r][j][0] = c0; h[r][j][1] = c1; h[r][j][2] = c0; h[r][j][3] = c1;
            mma_bf16(h[r][j], a[r], w0, w1);
        }
    }
    relu_pack(h[0], a2[0]);                       // accumulator layout == next A layout
    relu_pack(h[1], a2[1]);
#pragma unroll
    for (int j = 0; j < 8; j++) {                 // layer 2
        const int col = 8 * j + 2 * t, row = 8 * j + g;
        const float c0 = S.b2[col], c1 = S.b2[col + 1];
#pragma unroll
        for (int r = 0; r < 2; r++) { h[r][j][0] = c0; h[r][j][1] = c1; h[r][j][2] = c0; h[r][j][3] = c1; }
#pragma unroll
        for (int kc = 0; kc < 4; kc++) {
            const uint32_t w0 = S.w2[row * LD2 + 8 * kc + t], w1 = S.w2[row * LD2 + 8 * kc + t + 4];
#pragma unroll
            for (int r = 0; r < 2; r++) mma_bf16(h[r][j], a2[r][kc], w0, w1);
        }
    }
    relu_pack(h[0], a2[0]);
    relu_pack(h[1], a2[1]);
    float y[2][4];
#pragma unroll
    for (int r = 0; r < 2; r++) { y[r][0] = S.b3[2 * t]; y[r][1] = S.b3[2 * t + 1]; y[r][2] = y[r][0]; y[r][3] = y[r][1]; }
#pragma unroll
    for (int kc = 0; kc < 4; kc++) {              // layer 3 (outputs padded to 8)
        const uint32_t w0 = S.w3[g * LD2 + 8 * kc + t], w1 = S.w3[g * LD2 + 8 * kc + t + 4];
#pragma unroll
        for (int r = 0; r < 2; r++) mma_bf16(y[r], a2[r][kc], w0, w1);
    }
    if (t < 2)
#pragma unroll
        for (int r = 0; r < 2; r++) {
            float *y0 = ys[16 * r + g], *y1 = ys[16 * r + g + 8];
            y0[2 * t] = y[r][0]; y0[2 * t + 1] = y[r][1];
            y1[2 * t] = y[r][2]; y1[2 * t + 1] = y[r][3];
        }
}

// Corrects the tree accelerations in place: a += ysig |a| (y0 e0 + y1 e1 + y2 e2).
__global__ void __launch_bounds__(INF_WARPS * 32)
k_mlp_infer(const float *__restrict__ P, const float *__restrict__ norm, float4 *acc4,
            const float *__restrict__ feat, int n, const DevState *__restrict__ st) {
    __shared__ InfShared S;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (st->status & ST_TIMEOUT) return;
    stage_weights(S, P, norm);
    __syncthreads();
    const int step = gridDim.x * INF_WARPS * 32;
    for (int base = (blockIdx.x * INF_WARPS + warp) * 32; base < n; base += step) {
        const int i = base + lane;
        float4 av = make_float4(0.f, 0.f, 0.f, 0.f);
        float x[MLP_IN];
        Frame F{};
        if (i < n) {
            av = acc4[i];
            float f[FEAT_STRIDE];                 // a row of features is three aligned 16-byte words
            const float4 *fp = reinterpret_cast<const float4 *>(feat + FEAT_STRIDE * (size_t)i);
#pragma unroll
            for (int q = 0; q < 3; q++) {
                const float4 v = fp[q];
                f[4 * q] = v.x; f[4 * q + 1] = v.y; f[4 * q + 2] = v.z; f[4 * q + 3] = v.w;
            }
            body_features(av, f, S.norm, x, F);
        } else {
#pragma unroll
            for (int k = 0; k < MLP_IN; k++) x[k] = 0.f;
        }
#pragma unroll
        for (int k = 0; k < 16; k++) S.xs[warp][lane][k] = k < MLP_IN ? x[k] : 0.f;
        __syncwarp();
        mma_forward32(S, S.xs[warp], S.ys[warp], lane);
        __syncwarp();
        if (i < n) {
            const float s = F.an * S.ysig;
            const float c0 = S.ys[warp][lane][0] * s, c1 = S.ys[warp][lane][1] * s, c2 = S.ys[warp][lane][2] * s;
            av.x += c0 * F.e0.x + c1 * F.e1.x + c2 * F.e2.x;
            av.y += c0 * F.e0.y + c1 * F.e1.y + c2 * F.e2.y;
            av.z += c0 * F.e0.z + c1 * F.e1.z + c2 * F.e2.z;
            acc4[i] = av;
        }
        __syncwarp();
    }
}

// Raw network outputs for feature rows X (n x 12, not normalised) -> Y (n x 3).
__global__ void __launch_bounds__(INF_WARPS * 32)
k_mlp_rows(const float *__restrict__ P, const float *__restrict__ norm, const float *__restrict__ X,
           float *Y, int n) {
    __shared__ InfShared S;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    stage_weights(S, P, norm);
    __syncthreads();
    const long long step = (long long)gridDim.x * INF_WARPS * 32;
    for (long long base = (blockIdx.x * INF_WARPS + warp) * 32; base < n; base += step) {
        const long long i = base + lane;
#pragma unroll
        for (int k = 0; k < 16; k++)
            S.xs[warp][lane][k] = (k < MLP_IN && i < n)
                                      ? (X[(size_t)i * MLP_IN + k] - S.norm[k]) / S.norm[MLP_IN + k]
                                      : 0.f;
        __syncwarp();
        mma_forward32(S, S.xs[warp], S.ys[warp], lane);
        __syncwarp();
        if (i < n)
            for (int o = 0; o < MLP_OUT; o++) Y[(size_t)i * MLP_OUT + o] = S.ys[warp][lane][o];
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// Training: forward + backward of tiles of 32 samples per block.
//
// Bound: FP32 issue and shared-memory wavefronts.  A tile is five small
// products (units x samples forward and backward, units x units for the
// gradient of W2); each thread holds a register tile of 4 units x 2 samples
// (4 x 4 parameters for the gradient of W2), so that one 16-byte broadcast
// and one 8-byte read feed eight multiply-adds and both pipes take about as
// long (some 3600 cycles a tile each way).  32 samples a tile: a batch of
// 4096 is 128 blocks, one per SM.  One thread per sample with whole
// activation vectors in local memory and a five-step warp reduction and
// shared atomic per parameter took 956 us for a batch of 4096; this takes
// about 12 us (27 us before inputs were fetched a tile ahead and the weights
// staged in one round trip, 20 us with an atomic per parameter and block
// instead of the blocks' own rows of sums; all from a cold cache).  An epoch
// of 65,536 rows in 16 batches, device time: 265 us, 16.6 a batch.
//
// Every activation and every back-propagated value is one chain of fused
// multiply-adds over its inputs in index order, so it does not depend on the
// tiling; the parameter gradients are summed over the tile's samples in
// registers, across the tiles of a block, then over the blocks in a fixed
// order by the kernel that uses them.
// ---------------------------------------------------------------------------
constexpr int TR_THREADS = 256;                   // (512 with half the register tile: 293 us an epoch, 265 here)
constexpr int TR_U = MLP_H * 32 / 2 / TR_THREADS; // units of a thread's register tile
constexpr int TR_GA = 4 * TR_U / 4;               // W2 gradient rows of a thread (of 4 columns)
constexpr int TR_GJ = MLP_H / TR_GA;              // threads across the rows
constexpr int TR_S = 32;          // samples per tile (two per thread, 16 threads across)
constexpr int TR_LD = 36;         // row stride of the sample-major arrays: 16 rows apart read without conflicts
constexpr int TR_W2T = MLP_H + 4; // row stride of the transposed W2

struct __align__(16) TrShared {
    float w1t[MLP_IN][MLP_H];     // BF16-rounded weights; [in][out] for the forward products
    float w2t[MLP_H][TR_W2T];
    float w2[MLP_H][MLP_H];       // [out][in] for the backward product
    float w3[MLP_OUT][MLP_H];
    float b1[MLP_H], b2[MLP_H], b3[4];
    float norm[2 * MLP_IN];
    float x[MLP_IN][TR_LD];       // [unit][sample]
    float h1[MLP_H][TR_LD], h2[MLP_H][TR_LD], d2[MLP_H][TR_LD], d1[MLP_H][TR_LD];
    float dy[MLP_OUT][TR_LD];
};
static_assert(TR_U == 4 && MLP_H * MLP_H % TR_THREADS == 0, "16-byte weight reads, W2 staged in whole rounds");
static_assert(TR_S * MLP_IN <= 2 * TR_THREADS && TR_THREADS >= 32 * MLP_OUT, "a tile's inputs are two per thread");

// acc[u][s] <- chain over k of w[k][j0 + u] * in[k][s0 + s], k ascending.
template <int K, int LDW>
__device__ __forceinline__ void tile_units(const float *w, const float *in, int j0, int s0, float (&acc)[TR_U][2]) {
#pragma unroll 8
    for (int k = 0; k < K; k++) {
        const float4 v = *reinterpret_cast<const float4 *>(w + k * LDW + j0);
        const float a[TR_U] = {v.x, v.y, v.z, v.w};
        const float2 b = *reinterpret_cast<const float2 *>(in + k * TR_LD + s0);
#pragma unroll
        for (int u = 0; u < TR_U; u++) {
            acc[u][0] = fmaf(a[u], b.x, acc[u][0]);
            acc[u][1] = fmaf(a[u], b.y, acc[u][1]);
        }
    }
}

// Sum over the tile's samples of a[s] * b[s], added to acc in sample order.
__device__ __forceinline__ float dot_rows(const float *a, const float *b, float acc) {
#pragma unroll
    for (int s = 0; s < TR_S; s += 4) {
        const float4 u = *reinterpret_cast<const float4 *>(a + s), v = *reinterpret_cast<const float4 *>(b + s);
        acc = fmaf(u.x, v.x, acc); acc = fmaf(u.y, v.y, acc);
        acc = fmaf(u.z, v.z, acc); acc = fmaf(u.w, v.w, acc);
    }
    return acc;
}

__device__ __forceinline__ float sum_row(const float *a, float acc) {
#pragma unroll
    for (int s = 0; s < TR_S; s += 4) {
        const float4 u = *reinterpret_cast<const float4 *>(a + s);
        acc += u.x; acc += u.y; acc += u.z; acc += u.w;
    }
    return acc;
}

// X: n x 12 raw features, Y: n x 3 targets (divided by ysig here), idx:
// the samples of this batch (NULL: rows 0..bsz-1).  Each block writes its
// share of d(loss)/dP and of the loss, the mean over the batch and the 3
// outputs of the squared error, to its row of part.
__global__ void __launch_bounds__(TR_THREADS, 2)
k_mlp_grad(const float *__restrict__ P, const float *__restrict__ norm, const float *__restrict__ X,
           const float *__restrict__ Y, const uint32_t *__restrict__ idx, int bsz, float *part) {
    extern __shared__ float4 smem_tr[];
    TrShared &S = *reinterpret_cast<TrShared *>(smem_tr);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // This thread's raw inputs (two of the tile's 384) and target of a tile,
    // fetched a tile ahead: their two dependent round trips (index, row)
    // overlap the weights' staging or the tile before.  NaN-free zeros where
    // the batch ends.
    float xr[2] = {0.f, 0.f}, yr = 0.f;
    bool on = false;
    auto fetch = [&](int t0) {
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int e = tid + h * TR_THREADS, k = t0 + e / MLP_IN;
            if (e < TR_S * MLP_IN && k < bsz) xr[h] = X[(size_t)(idx ? idx[k] : (uint32_t)k) * MLP_IN + e % MLP_IN];
        }
        on = t0 + lane < bsz;
        if (warp < MLP_OUT && on)
            yr = Y[(size_t)(idx ? idx[t0 + lane] : (uint32_t)(t0 + lane)) * MLP_OUT + warp];
    };
    fetch(blockIdx.x * TR_S);
    {
        // all loads in flight at once
        constexpr int W1R = (MLP_H * MLP_IN + TR_THREADS - 1) / TR_THREADS;
        float w2r[MLP_H * MLP_H / TR_THREADS], w1r[W1R];
#pragma unroll
        for (int r = 0; r < MLP_H * MLP_H / TR_THREADS; r++) w2r[r] = P[OFF_W2 + tid + r * TR_THREADS];
#pragma unroll
        for (int r = 0; r < W1R; r++) w1r[r] = tid + r * TR_THREADS < MLP_H * MLP_IN ? P[OFF_W1 + tid + r * TR_THREADS] : 0.f;
        if (tid < MLP_OUT * MLP_H) S.w3[tid / MLP_H][tid % MLP_H] = bf16r(P[OFF_W3 + tid]);
        if (tid < MLP_H) { S.b1[tid] = P[OFF_B1 + tid]; S.b2[tid] = P[OFF_B2 + tid]; }
        if (tid < MLP_OUT) S.b3[tid] = P[OFF_B3 + tid];
        if (tid < 2 * MLP_IN) S.norm[tid] = norm[tid];
#pragma unroll
        for (int r = 0; r < MLP_H * MLP_H / TR_THREADS; r++) {
            const int i = tid + r * TR_THREADS;
            const float v = bf16r(w2r[r]);
            S.w2[i / MLP_H][i % MLP_H] = v;
            S.w2t[i % MLP_H][i / MLP_H] = v;
        }
#pragma unroll
        for (int r = 0; r < W1R; r++) {
            const int i = tid + r * TR_THREADS;
            if (i < MLP_H * MLP_IN) S.w1t[i % MLP_IN][i / MLP_IN] = bf16r(w1r[r]);
        }
    }
    __syncthreads();

    const int j0 = TR_U * (2 * warp + (lane >> 4)), s0 = 2 * (lane & 15);   // TR_U units x 2 samples
    const int gi = lane & 15, gj = 2 * warp + (lane >> 4);     // W2 parameters (gj + TR_GJ a, gi + 16 b)
    constexpr int NW1 = (MLP_H * MLP_IN + TR_THREADS - 1) / TR_THREADS;
    const int wj = tid & (MLP_H - 1), wi = tid >> 6;           // W1 parameters (wj, wi + TR_THREADS / 64 k)
    float g2[TR_GA][4], g1[NW1] = {}, g3 = 0.f, gb = 0.f, l = 0.f;
#pragma unroll
    for (int a = 0; a < TR_GA; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) g2[a][b] = 0.f;
    const float sc = 2.f / (3.f * (float)bsz), ysig = norm[2 * MLP_IN];

    for (int t0 = blockIdx.x * TR_S; t0 < bsz; t0 += gridDim.x * TR_S) {
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int e = tid + h * TR_THREADS, sm = e / MLP_IN, i = e % MLP_IN;
            if (e < TR_S * MLP_IN) S.x[i][sm] = t0 + sm < bsz ? bf16r((xr[h] - S.norm[i]) / S.norm[MLP_IN + i]) : 0.f;
        }
        const float target = yr / ysig;
        const bool live = on;
        if (t0 + (int)gridDim.x * TR_S < bsz) fetch(t0 + gridDim.x * TR_S);
        __syncthreads();
        float v[TR_U][2];
#pragma unroll
        for (int u = 0; u < TR_U; u++) v[u][0] = v[u][1] = S.b1[j0 + u];
        tile_units<MLP_IN, MLP_H>(&S.w1t[0][0], &S.x[0][0], j0, s0, v);
#pragma unroll
        for (int u = 0; u < TR_U; u++)
            *reinterpret_cast<float2 *>(&S.h1[j0 + u][s0]) =
                make_float2(bf16r(fmaxf(v[u][0], 0.f)), bf16r(fmaxf(v[u][1], 0.f)));
        __syncthreads();
#pragma unroll
        for (int u = 0; u < TR_U; u++) v[u][0] = v[u][1] = S.b2[j0 + u];
        tile_units<MLP_H, TR_W2T>(&S.w2t[0][0], &S.h1[0][0], j0, s0, v);
#pragma unroll
        for (int u = 0; u < TR_U; u++)
            *reinterpret_cast<float2 *>(&S.h2[j0 + u][s0]) =
                make_float2(bf16r(fmaxf(v[u][0], 0.f)), bf16r(fmaxf(v[u][1], 0.f)));
        __syncthreads();
        if (warp < MLP_OUT) {                      // outputs: warp = output, lane = sample
            float o = S.b3[warp];
#pragma unroll 16
            for (int i = 0; i < MLP_H; i++) o = fmaf(S.w3[warp][i], S.h2[i][lane], o);
            const float res = live ? o - target : 0.f;
            l += res * res;
            S.dy[warp][lane] = sc * res;
        }
        __syncthreads();
        // Backward: d2 = W3^T dy (ReLU gate), d1 = W2^T d2 (ReLU gate).
        for (int i = warp; i < MLP_H; i += TR_THREADS / 32) {
            float d = 0.f;
#pragma unroll
            for (int o = 0; o < MLP_OUT; o++) d = fmaf(S.w3[o][i], S.dy[o][lane], d);
            S.d2[i][lane] = S.h2[i][lane] > 0.f ? d : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < TR_U; u++) v[u][0] = v[u][1] = 0.f;
        tile_units<MLP_H, MLP_H>(&S.w2[0][0], &S.d2[0][0], j0, s0, v);
#pragma unroll
        for (int u = 0; u < TR_U; u++) {
            const float2 h = *reinterpret_cast<const float2 *>(&S.h1[j0 + u][s0]);
            *reinterpret_cast<float2 *>(&S.d1[j0 + u][s0]) =
                make_float2(h.x > 0.f ? v[u][0] : 0.f, h.y > 0.f ? v[u][1] : 0.f);
        }
        // Gradients of W2, W3 and the last two biases (need no d1).
#pragma unroll 2
        for (int s = 0; s < TR_S; s += 4) {
            float4 p[TR_GA], q[4];
#pragma unroll
            for (int a = 0; a < TR_GA; a++) p[a] = *reinterpret_cast<const float4 *>(&S.d2[gj + TR_GJ * a][s]);
#pragma unroll
            for (int b = 0; b < 4; b++) q[b] = *reinterpret_cast<const float4 *>(&S.h1[gi + 16 * b][s]);
#pragma unroll
            for (int a = 0; a < TR_GA; a++)
#pragma unroll
                for (int b = 0; b < 4; b++) {
                    g2[a][b] = fmaf(p[a].x, q[b].x, g2[a][b]); g2[a][b] = fmaf(p[a].y, q[b].y, g2[a][b]);
                    g2[a][b] = fmaf(p[a].z, q[b].z, g2[a][b]); g2[a][b] = fmaf(p[a].w, q[b].w, g2[a][b]);
                }
        }
        // (the small sums from the last threads down, W1's below from the first up)
        const int r3 = TR_THREADS - 1 - tid;
        if (r3 < MLP_OUT * MLP_H) g3 = dot_rows(S.dy[r3 / MLP_H], S.h2[r3 % MLP_H], g3);
        if (tid < MLP_H) gb = sum_row(S.d2[tid], gb);
        __syncthreads();
#pragma unroll
        for (int k = 0; k < NW1; k++)
            if (wi + TR_THREADS / MLP_H * k < MLP_IN) g1[k] = dot_rows(S.d1[wj], S.x[wi + TR_THREADS / MLP_H * k], g1[k]);
        if (tid >= MLP_H && tid < 2 * MLP_H) gb = sum_row(S.d1[tid - MLP_H], gb);
        if (tid >= 2 * MLP_H && tid < 2 * MLP_H + MLP_OUT) gb = sum_row(S.dy[tid - 2 * MLP_H], gb);
        __syncthreads();                            // the arrays are rewritten by the next tile
    }
    // The block's sums, coalesced, for the kernel that adds the blocks up.
    float *out = part + (size_t)blockIdx.x * TR_PART;
#pragma unroll
    for (int a = 0; a < TR_GA; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) out[OFF_W2 + (gj + TR_GJ * a) * MLP_H + gi + 16 * b] = g2[a][b];
#pragma unroll
    for (int k = 0; k < NW1; k++)
        if (wi + TR_THREADS / MLP_H * k < MLP_IN) out[OFF_W1 + wj * MLP_IN + wi + TR_THREADS / MLP_H * k] = g1[k];
    const int r3 = TR_THREADS - 1 - tid;
    if (r3 < MLP_OUT * MLP_H) out[OFF_W3 + r3] = g3;
    if (tid < MLP_H) out[OFF_B2 + tid] = gb;
    else if (tid < 2 * MLP_H) out[OFF_B1 + tid - MLP_H] = gb;
    else if (tid < 2 * MLP_H + MLP_OUT) out[OFF_B3 + tid - 2 * MLP_H] = gb;
    if (warp < MLP_OUT) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) S.dy[warp][0] = l;
    }
    __syncthreads();
    if (tid == 0) out[MLP_NPARAM] = (S.dy[0][0] + S.dy[1][0] + S.dy[2][0]) / (3.f * (float)bsz);
}

// Sum of the blocks' partial sums of parameter i (i == MLP_NPARAM: the
// loss), the same for every run: RED_SLICES threads each add every
// RED_SLICES-th block's, all loads independent, then a shared-memory sum.
// Result valid in slice 0.  Blocks adding with atomics instead (128 on each
// address) held the gradient kernel for about 8 us after its last tile.
constexpr int RED_PARAMS = 32, RED_SLICES = 8;
__device__ __forceinline__ float reduce_part(const float *__restrict__ part, int nblk, int i,
                                             float (&red)[RED_SLICES][RED_PARAMS]) {
    const int p = threadIdx.x % RED_PARAMS, sl = threadIdx.x / RED_PARAMS;
    float s = 0.f;
    if (i <= MLP_NPARAM) {
#pragma unroll 16
        for (int b = sl; b < nblk; b += RED_SLICES) s += part[(size_t)b * TR_PART + i];
    }
    red[sl][p] = s;
    __syncthreads();
    float t = 0.f;
    if (sl == 0)
#pragma unroll
        for (int k = 0; k < RED_SLICES; k++) t += red[k][p];
    return t;
}

__global__ void __launch_bounds__(RED_PARAMS * RED_SLICES)
k_grad_reduce(const float *__restrict__ part, int nblk, float *grad, float *loss) {
    __shared__ float red[RED_SLICES][RED_PARAMS];
    const int i = blockIdx.x * RED_PARAMS + threadIdx.x % RED_PARAMS;
    const float g = reduce_part(part, nblk, i, red);
    if (threadIdx.x >= RED_PARAMS) return;
    if (i < MLP_NPARAM) grad[i] = g;
    else if (i == MLP_NPARAM) *loss = g;
}

// AdamW (decoupled weight decay on the weight matrices, not the biases) on
// the sum of the blocks' gradients; adds the batch's loss to *loss.
__global__ void __launch_bounds__(RED_PARAMS * RED_SLICES)
k_adamw(float *P, const float *__restrict__ part, int nblk, float *m, float *v, float *loss, float lr, float b1,
        float b2, float eps, float wd, float bc1, float bc2) {
    __shared__ float red[RED_SLICES][RED_PARAMS];
    const int i = blockIdx.x * RED_PARAMS + threadIdx.x % RED_PARAMS;
    const float g = reduce_part(part, nblk, i, red);
    if (threadIdx.x >= RED_PARAMS || i > MLP_NPARAM) return;
    if (i == MLP_NPARAM) { *loss += g; return; }
    const bool bias = (i >= OFF_B1 && i < OFF_W2) || (i >= OFF_B2 && i < OFF_W3) || i >= OFF_B3;
    const float mi = b1 * m[i] + (1.f - b1) * g;
    const float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    float w = P[i];
    w -= lr * ((mi / bc1) / (sqrtf(vi / bc2) + eps) + (bias ? 0.f : wd * w));
    P[i] = w;
}

cudaError_t launch_mlp_infer(Ctx &c, const float *P, const float *norm) {
    const int n = (int)c.n;
    int blocks = (n + INF_WARPS * 32 - 1) / (INF_WARPS * 32);
    const int cap = c.num_sms * 8;
    if (blocks > cap) blocks = cap;
    k_mlp_infer<<<blocks, INF_WARPS * 32, 0, c.stream>>>(P, norm, c.acc4, c.feat, n, c.st);
    return cudaGetLastError();
}

cudaError_t launch_mlp_rows(cudaStream_t s, const float *P, const float *norm, const float *X, float *Y, int n) {
    int blocks = (n + INF_WARPS * 32 - 1) / (INF_WARPS * 32);
    if (blocks > 1216) blocks = 1216;
    k_mlp_rows<<<blocks, INF_WARPS * 32, 0, s>>>(P, norm, X, Y, n);
    return cudaGetLastError();
}

// The partial sums of a batch: nblk blocks' into part (TR_BLOCKS x TR_PART).
static cudaError_t launch_grad_part(cudaStream_t s, const float *P, const float *norm, const float *X,
                                    const float *Y, const uint32_t *idx, int bsz, float *part, int &nblk) {
    static size_t attr_done[MAX_DEVICES] = {};
    const size_t smem = sizeof(TrShared);
    cudaError_t e = allow_dyn_smem((const void *)k_mlp_grad, smem, attr_done);
    if (e != cudaSuccess) return e;
    nblk = std::min((bsz + TR_S - 1) / TR_S, TR_BLOCKS);
    k_mlp_grad<<<nblk, TR_THREADS, smem, s>>>(P, norm, X, Y, idx, bsz, part);
    return cudaGetLastError();
}

constexpr int RED_GRID = (MLP_NPARAM + 1 + RED_PARAMS - 1) / RED_PARAMS;

// Gradient and loss of a batch (idx NULL: rows 0..bsz-1).
cudaError_t launch_mlp_grad(cudaStream_t s, const float *P, const float *norm, const float *X, const float *Y,
                            const uint32_t *idx, int bsz, float *part, float *grad, float *loss) {
    int nblk = 0;
    cudaError_t e = launch_grad_part(s, P, norm, X, Y, idx, bsz, part, nblk);
    if (e != cudaSuccess) return e;
    k_grad_reduce<<<RED_GRID, RED_PARAMS * RED_SLICES, 0, s>>>(part, nblk, grad, loss);
    return cudaGetLastError();
}

// One training batch: its gradient and the AdamW update; *loss grows by the
// batch's loss.
cudaError_t launch_mlp_batch(cudaStream_t s, float *P, const float *norm, const float *X, const float *Y,
                             const uint32_t *idx, int bsz, float *part, float *m, float *v, float *loss, float lr,
                             float wd, int step) {
    int nblk = 0;
    cudaError_t e = launch_grad_part(s, P, norm, X, Y, idx, bsz, part, nblk);
    if (e != cudaSuccess) return e;
    const float b1 = 0.9f, b2 = 0.999f;
    const float bc1 = 1.f - powf(b1, (float)step), bc2 = 1.f - powf(b2, (float)step);
    k_adamw<<<RED_GRID, RED_PARAMS * RED_SLICES, 0, s>>>(P, part, nblk, m, v, loss, lr, b1, b2, 1e-8f, wd, bc1, bc2);
    return cudaGetLastError();
}

// Per-body features in caller-independent form for training sets:
// X[k] (12 raw inputs) of the sampled sorted positions.
__global__ void k_gather_features(const float4 *__restrict__ acc4, const float *__restrict__ feat,
                                  const uint32_t *__restrict__ targets, int ntar, float *X,
                                  const uint32_t *__restrict__ id, uint32_t *ids) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= ntar) return;
    const uint32_t i = targets[k];
    if (ids) ids[k] = id[i];
    float x[MLP_IN];
    Frame F;
    body_inputs(acc4[i], feat + FEAT_STRIDE * (size_t)i, x, F);
    for (int j = 0; j < MLP_IN; j++) X[(size_t)k * MLP_IN + j] = x[j];
}

cudaError_t launch_gather_features(Ctx &c, const uint32_t *targets, int ntar, float *X, uint32_t *ids) {
    k_gather_features<<<(ntar + 255) / 256, 256, 0, c.stream>>>(c.acc4, c.feat, targets, ntar, X, c.id, ids);
    return cudaGetLastError();
}

// Training targets: the relative residual r = (a_direct - a_tree) / |a_tree|
// at target k in the body's local frame, Y[k] = (r.e0, r.e1, r.e2).
__global__ void k_labels(const float4 *__restrict__ acc4, const float *__restrict__ feat,
                         const uint32_t *__restrict__ targets, int ntar, const float4 *__restrict__ direct,
                         float *Y) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= ntar) return;
    const uint32_t i = targets[k];
    const float4 a = acc4[i], d = direct[k];
    float x[MLP_IN];
    Frame F;
    body_inputs(a, feat + FEAT_STRIDE * (size_t)i, x, F);
    const float inv = F.an > 0.f ? 1.f / F.an : 0.f;
    const float rx = (d.x - a.x) * inv, ry = (d.y - a.y) * inv, rz = (d.z - a.z) * inv;
    Y[3 * (size_t)k] = rx * F.e0.x + ry * F.e0.y + rz * F.e0.z;
    Y[3 * (size_t)k + 1] = rx * F.e1.x + ry * F.e1.y + rz * F.e1.z;
    Y[3 * (size_t)k + 2] = rx * F.e2.x + ry * F.e2.y + rz * F.e2.z;
}

cudaError_t launch_labels(Ctx &c, const uint32_t *targets, int ntar, const float4 *direct, float *Y) {
    k_labels<<<(ntar + 255) / 256, 256, 0, c.stream>>>(c.acc4, c.feat, targets, ntar, direct, Y);
    return cudaGetLastError();
}

// Input normalisation of a training set: per-feature mean and standard
// deviation (FP64 sums), and the RMS of the targets.  Each block sums its
// rows (a warp reduction per block, no atomics), the last block to finish
// adds the blocks' sums in block order.  FP64 adds bound it (1/64 of the
// FP32 rate), so the rows go over STATS_BLOCKS blocks: 801 us for 65,536
// rows in one block, 27 us here.
__global__ void __launch_bounds__(STATS_THREADS)
k_feature_stats(const float *__restrict__ X, const float *__restrict__ Y, int n, double *part, unsigned *arrived,
                float *norm) {
    constexpr int NV = MLP_NNORM, NW = STATS_THREADS / 32;
    __shared__ double red[NW][NV];
    __shared__ bool s_last;
    double s[MLP_IN], q[MLP_IN], yy = 0.0;
#pragma unroll
    for (int k = 0; k < MLP_IN; k++) { s[k] = 0.0; q[k] = 0.0; }
    for (long long i = blockIdx.x * STATS_THREADS + threadIdx.x; i < n; i += (long long)gridDim.x * STATS_THREADS) {
#pragma unroll
        for (int k = 0; k < MLP_IN; k++) {
            const double v = X[(size_t)i * MLP_IN + k];
            s[k] += v; q[k] += v * v;
        }
#pragma unroll
        for (int o = 0; o < MLP_OUT; o++) { const double v = Y[(size_t)i * MLP_OUT + o]; yy += v * v; }
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < MLP_IN; k++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
            q[k] += __shfl_xor_sync(0xffffffffu, q[k], o);
        }
        if (lane == 0) { red[w][k] = s[k]; red[w][MLP_IN + k] = q[k]; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) yy += __shfl_xor_sync(0xffffffffu, yy, o);
    if (lane == 0) red[w][2 * MLP_IN] = yy;
    __syncthreads();
    if (threadIdx.x < NV) {
        double t = 0.0;
        for (int j = 0; j < NW; j++) t += red[j][threadIdx.x];
        part[(size_t)blockIdx.x * NV + threadIdx.x] = t;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(arrived, 1u) == gridDim.x - 1u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (threadIdx.x < NV) {
        double t = 0.0;
        for (unsigned j = 0; j < gridDim.x; j++) t += __ldcg(part + (size_t)j * NV + threadIdx.x);
        red[0][threadIdx.x] = t;
    }
    if (threadIdx.x == 0) *arrived = 0u;
    __syncthreads();
    if (threadIdx.x < MLP_IN) {
        const int k = threadIdx.x;
        const double mu = red[0][k] / n, var = red[0][MLP_IN + k] / n - mu * mu;
        norm[k] = (float)mu;
        norm[MLP_IN + k] = (float)fmax(sqrt(fmax(var, 0.0)), 1e-6);
    }
    if (threadIdx.x == 0) norm[2 * MLP_IN] = (float)fmax(sqrt(red[0][2 * MLP_IN] / (3.0 * n)), 1e-12);
}

cudaError_t launch_feature_stats(cudaStream_t s, const float *X, const float *Y, int n, double *part,
                                 unsigned *arrived, float *norm) {
    const int grid = std::min((n + STATS_THREADS - 1) / STATS_THREADS, STATS_BLOCKS);
    k_feature_stats<<<grid, STATS_THREADS, 0, s>>>(X, Y, n, part, arrived, norm);
    return cudaGetLastError();
}

}  // namespace bonsai
