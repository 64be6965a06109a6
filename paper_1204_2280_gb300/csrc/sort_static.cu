// sort_static.cu -- bonsai_sort_keys_static: the stable sort of 63-bit
// keys with all of its scratch in one file-scope device array, for callers
// that must not allocate device memory.
//
// Who needs this: code that cannot call cudaMalloc/cudaFree around a sort --
// a latency-critical loop (cudaMalloc and cudaFree can synchronise the whole
// device and take milliseconds), or a host application whose own caching
// allocator has already reserved the device memory (a second allocator would
// fail or fragment it).  Such a caller passes its own input and output
// buffers and this entry point takes nothing else from the device heap.
// The call synchronises its stream before it returns, so it cannot be
// recorded into a CUDA graph by stream capture.
//
// The scratch (0.75 MiB) is a static __device__ array: every GPU on
// which the library is loaded holds it until the process exits, and every
// call shares it.  Calls whose GPU work overlaps (two host threads, or two
// streams) would race on it, so callers must serialise them.
#include <mutex>

#include "common.cuh"

namespace bonsai {

constexpr int STATIC_SORT_MAX_N = 1 << 16;                       // 65536 keys

struct StaticSortScratch {                                       // the merges' other buffer
    unsigned long long keys_alt[STATIC_SORT_MAX_N];
    uint32_t vals_alt[STATIC_SORT_MAX_N];
};

// Device-resident scratch.  Host code must never pass this name to a kernel:
// on the host it is only a stand-in; its device address comes from
// cudaGetSymbolAddress below.
static __device__ __align__(256) StaticSortScratch g_sort_scratch;

void set_global_error(const char *msg);   // api.cu: text of bonsai_last_error(NULL)

namespace {
std::mutex g_setup_mu;
StaticSortScratch *g_dev_ptr[MAX_DEVICES] = {};

int set_err(int code, const char *msg) {
    cudaGetLastError();
    set_global_error(msg);
    return code;
}
}  // namespace

}  // namespace bonsai

using namespace bonsai;

extern "C" int bonsai_sort_keys_static(const uint64_t *keys, uint64_t *sorted_keys, uint32_t *perm,
                                       long long n, void *cuda_stream) {
    if (!keys || !sorted_keys || !perm || n < 1)
        return set_err(BONSAI_ERR_INVALID_ARG, "bonsai_sort_keys_static: need device keys, outputs and n >= 1");
    if (n > STATIC_SORT_MAX_N)
        return set_err(BONSAI_ERR_INVALID_ARG,
                       "bonsai_sort_keys_static: n exceeds the static scratch limit of 65536 keys");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES)
        return set_err(BONSAI_ERR_CUDA, "bonsai_sort_keys_static: no usable current device");
    StaticSortScratch *s = nullptr;
    {
        // Once per device, with that device current: the device address of
        // the static scratch.
        std::lock_guard<std::mutex> lock(g_setup_mu);
        if (!g_dev_ptr[dev]) {
            void *p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, g_sort_scratch);
            if (e != cudaSuccess || !p)
                return set_err(BONSAI_ERR_CUDA, "bonsai_sort_keys_static: cudaGetSymbolAddress failed");
            g_dev_ptr[dev] = (StaticSortScratch *)p;
        }
        s = g_dev_ptr[dev];
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // a tile sort and merges, four for 65536 keys; nothing in them waits on
    // another block
    if (sort_pairs_small((const unsigned long long *)keys, (unsigned long long *)sorted_keys, s->keys_alt, perm,
                         s->vals_alt, (int)n, st) != cudaSuccess)
        return set_err(BONSAI_ERR_CUDA, "bonsai_sort_keys_static: kernel launch failed");
    if (cudaStreamSynchronize(st) != cudaSuccess)
        return set_err(BONSAI_ERR_CUDA, "bonsai_sort_keys_static: device error");
    return BONSAI_OK;
}
