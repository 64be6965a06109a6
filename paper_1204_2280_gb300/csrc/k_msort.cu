// k_msort.cu -- stable merge sort of (63-bit Morton key, u32 index) for
// small and medium body counts, with the key computation at its start and
// the body reorder at its end (paper Sect. 2, "sorting" and "moving").
//
// The radix sort (k_sort.cu) runs eight dependent passes whatever the size;
// below about a million bodies each pass is one tile's latency (9 us: load,
// ranking, look-back, scatter), 74 us even for one tile.  Here a tile of
// MS_TILE keys is sorted in shared memory by one block, then runs are merged
// pairwise, one launch per doubling:
//   * tile sort: each thread computes MS_IPT keys from positions and sorts
//     them in registers (odd-even transposition), then log2(MS_THREADS)
//     rounds of merges in shared memory, each thread finding its share by
//     merge path;
//   * merge: a block writes one tile of the merged run; two warps find the
//     tile's ends in the two runs with 32-way searches (three rounds of
//     dependent loads for runs of 4,608 keys, five for 2^21), the tile's keys
//     go to shared memory and each thread merges MS_IPT of them;
//   * the launch that finishes the order also moves the bodies (positions,
//     velocities, ids) instead of writing the permutation for a further pass.
// No block waits on another.  MS_IPT is odd, so that the threads' runs of
// keys start in different banks.
#include "morton.cuh"

namespace bonsai {

constexpr int MS_THREADS = 512;
constexpr int MS_IPT = 9;
constexpr int MS_TILE = MS_THREADS * MS_IPT;      // 4608 keys
constexpr unsigned long long MS_PAD = ~0ull;      // after every key; pads are last in position order

using u64 = unsigned long long;

// Number of elements of a[0, na) among the first d of the merged order of
// a and b (equal keys: a first).
__device__ __forceinline__ int merge_path(const u64 *a, int na, const u64 *b, int nb, int d) {
    int lo = max(0, d - nb), hi = min(d, na);
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (a[mid] <= b[d - 1 - mid]) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// The same over global memory by a whole warp: 32 places at a time.
__device__ __forceinline__ int merge_path_warp(const u64 *a, int na, const u64 *b, int nb, int d, int lane) {
    int lo = max(0, d - nb), hi = min(d, na);
    while (lo < hi) {
        const int len = hi - lo;
        const bool few = len <= 32;
        const int at = few ? lane : (int)((long long)(lane + 1) * len / 33);
        const int mid = lo + at;
        const bool before = (!few || lane < len) && a[mid] <= b[d - 1 - mid];
        const int c = __popc(__ballot_sync(0xffffffffu, before));
        if (few) return lo + c;
        const int m_lo = (int)((long long)c * len / 33), m_hi = (int)((long long)(c + 1) * len / 33);
        hi = c == 32 ? hi : lo + m_hi;
        lo = c == 0 ? lo : lo + m_lo + 1;
    }
    return lo;
}

// MS_IPT outputs of the merge of s[a, aend) and s[b, bend): keys and the
// places they came from.  One read per output whichever side it is taken
// from (no divergence); s has MS_SLACK readable places after its keys.
constexpr int MS_SLACK = MS_IPT + 1;
__device__ __forceinline__ void serial_merge(const u64 *s, int a, int aend, int b, int bend, u64 (&k)[MS_IPT],
                                             int (&from)[MS_IPT]) {
    u64 ka = s[a], kb = s[b];
#pragma unroll
    for (int i = 0; i < MS_IPT; i++) {
        const bool p = b >= bend || (a < aend && ka <= kb);
        const int at = p ? a : b;
        k[i] = p ? ka : kb;
        from[i] = at;
        const u64 next = s[at + 1];
        a += p ? 1 : 0;
        b += p ? 0 : 1;
        ka = p ? next : ka;
        kb = p ? kb : next;
    }
}

struct ReorderArgs {
    const float4 *pin, *vin;
    const uint32_t *idin;
    float4 *pout, *vout;
    uint32_t *idout;
};

__device__ __forceinline__ void move_body(const ReorderArgs &r, int to, uint32_t from) {
    const float4 p = r.pin[from], v = r.vin[from];
    const uint32_t id = r.idin[from];
    r.pout[to] = p;
    r.vout[to] = v;
    r.idout[to] = id;
}

// The launches of a sort follow one another closely (programmatic dependent
// launch): a kernel lets its successor be set up while it runs, and waits
// until its predecessor is complete and its writes are visible (a hardware
// wait, no polling) before it reads.  As every kernel of the chain waits for
// the one before, all earlier work is complete too.  The buffers that the
// chain writes change while its later kernels are already resident, so these
// kernels read memory by ordinary loads only, which the wait orders and the
// compiler keeps behind it: no const __restrict__ pointers and no __ldg, whose
// data must not change while a kernel lives.  A static sort of 65,536 keys
// 71 -> 65 us; the same for the build's and the multipoles' launches measured
// no gain at 2^12..2^17 and 0.5% more time at 2^20.
__device__ __forceinline__ void follow_previous() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <class... P, class... A>
inline cudaError_t launch_after(void (*fn)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                                A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, static_cast<P>(args)...);
}

// Sorts tile blockIdx.x.  POS: keys of the positions r.pin in the cube of
// st->dom (one system; block 0 stores the cube), else from keys.  MOVE (one
// tile): moves the bodies, else writes the sorted indices.
template <bool POS, bool MOVE>
__global__ void __launch_bounds__(MS_THREADS, 2)
k_tile_sort(const u64 *keys, u64 *kout, uint32_t *vout, int n, DevState *st, ReorderArgs r) {
    extern __shared__ u64 ms_smem[];
    u64 *s_k = ms_smem;
    unsigned short *s_v = reinterpret_cast<unsigned short *>(ms_smem + MS_TILE + MS_SLACK);
    __shared__ float4 s_dom;
    follow_previous();
    const int tid = threadIdx.x, base = blockIdx.x * MS_TILE;
    if (POS) {
        float4 q[MS_IPT];
#pragma unroll
        for (int i = 0; i < MS_IPT; i++) {
            const int j = base + tid + i * MS_THREADS;
            q[i] = j < n ? r.pin[j] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (tid == 0) {
            float mn[3], side;
            const float scale = domain_of(st->dom, mn, side);
            s_dom = make_float4(mn[0], mn[1], mn[2], scale);
            if (blockIdx.x == 0) {
                for (int d = 0; d < 3; d++) st->mn[d] = mn[d];
                st->side[0] = side;
                st->scale[0] = scale;
            }
        }
        __syncthreads();
        const float4 dm = s_dom;
#pragma unroll
        for (int i = 0; i < MS_IPT; i++)
            s_k[tid + i * MS_THREADS] = base + tid + i * MS_THREADS < n ? morton_key(q[i], dm) : MS_PAD;
    } else {
#pragma unroll
        for (int i = 0; i < MS_IPT; i++) {
            const int j = base + tid + i * MS_THREADS;
            s_k[tid + i * MS_THREADS] = j < n ? keys[j] : MS_PAD;
        }
    }
    __syncthreads();
    u64 k[MS_IPT];
    int v[MS_IPT];
#pragma unroll
    for (int i = 0; i < MS_IPT; i++) { k[i] = s_k[tid * MS_IPT + i]; v[i] = tid * MS_IPT + i; }
    // odd-even transposition: only neighbours swap, and only when out of
    // order, so equal keys keep their places
#pragma unroll
    for (int p = 0; p < MS_IPT; p++)
#pragma unroll
        for (int i = p & 1; i + 1 < MS_IPT; i += 2)
            if (k[i + 1] < k[i]) {
                const u64 tk = k[i]; k[i] = k[i + 1]; k[i + 1] = tk;
                const int tv = v[i]; v[i] = v[i + 1]; v[i + 1] = tv;
            }
    for (int w = 1; w < MS_THREADS; w <<= 1) {    // pairs of runs of w threads (inside a warp below 32)
        if (w < 32) __syncwarp(); else __syncthreads();
#pragma unroll
        for (int i = 0; i < MS_IPT; i++) {
            s_k[tid * MS_IPT + i] = k[i];
            s_v[tid * MS_IPT + i] = (unsigned short)v[i];
        }
        if (w < 32) __syncwarp(); else __syncthreads();
        const int pair = tid & ~(2 * w - 1), a0 = pair * MS_IPT, len = w * MS_IPT, b0 = a0 + len;
        const int d = (tid - pair) * MS_IPT;
        const int ai = merge_path(s_k + a0, len, s_k + b0, len, d);
        int from[MS_IPT];
        serial_merge(s_k, a0 + ai, b0, b0 + d - ai, b0 + len, k, from);
#pragma unroll
        for (int i = 0; i < MS_IPT; i++) v[i] = s_v[from[i]];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < MS_IPT; i++) {
        s_k[tid * MS_IPT + i] = k[i];
        s_v[tid * MS_IPT + i] = (unsigned short)v[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < MS_IPT; i++) {
        const int p = tid + i * MS_THREADS, j = base + p;
        if (j < n) {
            const uint32_t src = (uint32_t)(base + s_v[p]);
            kout[j] = s_k[p];
            if (MOVE) move_body(r, j, src); else vout[j] = src;
        }
    }
}

constexpr size_t MS_TILE_SMEM = (size_t)(MS_TILE + MS_SLACK) * sizeof(u64) + MS_TILE * sizeof(unsigned short);
constexpr size_t MS_MERGE_SMEM = (size_t)(MS_TILE + MS_SLACK) * (sizeof(u64) + sizeof(uint32_t));

// Merges neighbouring sorted runs of `run` keys (a multiple of MS_TILE) into
// runs twice as long; block t writes outputs [t MS_TILE, (t + 1) MS_TILE).
template <bool MOVE>
__global__ void __launch_bounds__(MS_THREADS, 2)
k_merge(const u64 *kin, const uint32_t *vin, u64 *kout, uint32_t *vout, int n, int run, ReorderArgs r) {
    extern __shared__ u64 ms_smem[];
    u64 *s_k = ms_smem;
    uint32_t *s_v = reinterpret_cast<uint32_t *>(ms_smem + MS_TILE + MS_SLACK);
    __shared__ int s_cut[2];
    follow_previous();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long o0 = (long long)blockIdx.x * MS_TILE;
    const int p0 = (int)(o0 / (2ll * run) * (2ll * run));           // first key of the pair of runs
    const int na = min(run, n - p0), nb = max(0, (int)min((long long)run, (long long)n - p0 - run));
    const int d0 = (int)(o0 - p0), d1 = min(d0 + MS_TILE, na + nb);
    const u64 *ga = kin + p0, *gb = ga + na;
    if (warp < 2) {
        const int c = merge_path_warp(ga, na, gb, nb, warp == 0 ? d0 : d1, lane);
        if (lane == 0) s_cut[warp] = c;
    }
    __syncthreads();
    const int a0 = s_cut[0], a1 = s_cut[1], b0 = d0 - a0;
    const int la = a1 - a0, total = d1 - d0;
#pragma unroll
    for (int i = 0; i < MS_IPT; i++) {
        const int p = tid + i * MS_THREADS;
        if (p < total) {
            const int src = p0 + (p < la ? a0 + p : na + b0 + (p - la));
            s_k[p] = kin[src];
            s_v[p] = vin[src];
        }
    }
    __syncthreads();
    const int d = min(tid * MS_IPT, total);
    const int ai = merge_path(s_k, la, s_k + la, total - la, d);
    u64 k[MS_IPT];
    int from[MS_IPT];
    serial_merge(s_k, ai, la, la + d - ai, total, k, from);
    uint32_t v[MS_IPT];
#pragma unroll
    for (int i = 0; i < MS_IPT; i++) v[i] = s_v[from[i]];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < MS_IPT; i++) { s_k[tid * MS_IPT + i] = k[i]; s_v[tid * MS_IPT + i] = v[i]; }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < MS_IPT; i++) {
        const int p = tid + i * MS_THREADS;
        if (p < total) {
            const int j = (int)o0 + p;
            kout[j] = s_k[p];
            if (MOVE) move_body(r, j, s_v[p]); else vout[j] = s_v[p];
        }
    }
}

// Which sort a context uses: this one for a single system of at most
// MERGE_MAX_N bodies (an ensemble's order has the system id above the key,
// 71 bits), unless the testing aid holds a tile, which needs the sort whose
// tiles wait on one another.  Keys, sort and reorder of a step, radix / merge
// sort: 80 / 31 us at 2^12, 88 / 47 at 2^15, 98 / 68 at 2^18, 150 / 115 at
// 2^20, 256 / 197 at 2^21, 438 / 377 at 2^22, 786 / 876 at 2^23 and
// 1452 / 1812 at 2^24: each merge moves every key once more, so past 2^22 the
// radix sort's fixed eight passes win.
#ifndef MERGE_MAX_N
#define MERGE_MAX_N (1 << 22)
#endif
bool sort_by_merge(const Ctx &c) { return c.nsys == 1 && c.n <= MERGE_MAX_N && !c.hold_tile; }

template <bool POS, bool MOVE>
static cudaError_t tile_sort(const u64 *keys, u64 *kout, uint32_t *vout, int n, DevState *st, const ReorderArgs &r,
                             cudaStream_t s) {
    static size_t attr_done[MAX_DEVICES] = {};
    const cudaError_t e = allow_dyn_smem((const void *)k_tile_sort<POS, MOVE>, MS_TILE_SMEM, attr_done);
    if (e != cudaSuccess) return e;
    return launch_after(k_tile_sort<POS, MOVE>, (n + MS_TILE - 1) / MS_TILE, MS_THREADS, MS_TILE_SMEM, s, keys, kout,
                        vout, n, st, r);
}

static int merge_levels(long long n) {
    int m = 0;
    for (long long run = MS_TILE; run < n; run <<= 1) m++;
    return m;
}

template <bool MOVE>
static cudaError_t merge_level(const u64 *kin, const uint32_t *vin, u64 *kout, uint32_t *vout, int n, int run,
                               const ReorderArgs &r, cudaStream_t s) {
    static size_t attr_done[MAX_DEVICES] = {};
    const cudaError_t e = allow_dyn_smem((const void *)k_merge<MOVE>, MS_MERGE_SMEM, attr_done);
    if (e != cudaSuccess) return e;
    return launch_after(k_merge<MOVE>, (n + MS_TILE - 1) / MS_TILE, MS_THREADS, MS_MERGE_SMEM, s, kin, vin, kout,
                        vout, n, run, r);
}

static ReorderArgs reorder_args(Ctx &c) {
    return ReorderArgs{c.pos4_alt, c.vel4_alt, c.id_alt, c.pos4, c.vel4, c.id};
}

// Keys and tile sort; the tiles land where the merges that follow end in
// c.keys.
cudaError_t launch_tile_sort(Ctx &c) {
    const int n = (int)c.n, m = merge_levels(n);
    u64 *k = m & 1 ? c.keys_alt : c.keys;
    uint32_t *v = m & 1 ? c.vals_alt : c.vals;
    return m == 0 ? tile_sort<true, true>(nullptr, k, v, n, c.st, reorder_args(c), c.stream)
                  : tile_sort<true, false>(nullptr, k, v, n, c.st, reorder_args(c), c.stream);
}

cudaError_t launch_merges(Ctx &c) {
    const int n = (int)c.n, m = merge_levels(n);
    u64 *kb[2] = {c.keys, c.keys_alt};
    uint32_t *vb[2] = {c.vals, c.vals_alt};
    long long run = MS_TILE;
    for (int l = 0; l < m; l++, run <<= 1) {
        const int in = (m - l) & 1, out = in ^ 1;
        const cudaError_t e = l + 1 < m ? merge_level<false>(kb[in], vb[in], kb[out], vb[out], n, (int)run,
                                                             reorder_args(c), c.stream)
                                        : merge_level<true>(kb[in], vb[in], kb[out], vb[out], n, (int)run,
                                                            reorder_args(c), c.stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Sorted keys and indices of n keys in out / vout; tmp / vtmp: scratch of
// the same size.  out may be keys.
cudaError_t sort_pairs_small(const u64 *keys, u64 *out, u64 *tmp, uint32_t *vout, uint32_t *vtmp, int n,
                             cudaStream_t s) {
    const int m = merge_levels(n);
    u64 *kb[2] = {out, tmp};
    uint32_t *vb[2] = {vout, vtmp};
    cudaError_t e = tile_sort<false, false>(keys, kb[m & 1], vb[m & 1], n, nullptr, ReorderArgs{}, s);
    long long run = MS_TILE;
    for (int l = 0; l < m && e == cudaSuccess; l++, run <<= 1) {
        const int in = (m - l) & 1;
        e = merge_level<false>(kb[in], vb[in], kb[in ^ 1], vb[in ^ 1], n, (int)run, ReorderArgs{}, s);
    }
    return e;
}

}  // namespace bonsai
