// Tree attention for callers that cannot allocate device memory.
//
// Some embedders of this library run inside a memory arena they do not control: a serving process
// that has handed every byte of the device to its own pool at start-up, a plug-in loaded after
// that point, or a latency-critical loop in which cudaMalloc (a device-wide synchronising call)
// is forbidden. llmcad_tree_attention() needs a context, and creating one allocates its work
// buffers. The variant below needs no context: the kernels make the mask table in shared memory, and the
// status word, when the caller does not want it, lives in a static device array that comes with the
// library image, so nothing is allocated at any time.
#include <cstdio>

#include "attention_tc.cuh"
#include "common.cuh"

namespace {

constexpr int kMaxNodes = LLMCAD_MAX_TREE;      // 128 tree nodes
constexpr size_t kScratchBytes = 256;           // a status word

// One copy per GPU that loads the library, held until the process exits.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

constexpr int kMaxDevices = 64;
void *g_scratch_ptr[kMaxDevices] = {};          // device address of the array on each device

thread_local char g_err[160] = "";

}  // namespace

extern "C" const char *llmcad_noalloc_last_error(void) { return g_err; }

extern "C" int llmcad_tree_attention_noalloc(const void *q, const void *k, const void *v, int32_t n_heads, int32_t kv_stride,
                                             int32_t prefix_len, const int32_t *parent_idx, int32_t n, void *o,
                                             int32_t *status_out, void *stream)
{
    using namespace llmcad;
    if (!q || !k || !v || !parent_idx || !o) { snprintf(g_err, sizeof(g_err), "null pointer"); return LLMCAD_ERR_INVALID_ARG; }
    if (n < 1 || prefix_len < 0 || n_heads < 1 || kv_stride < prefix_len + n) {
        snprintf(g_err, sizeof(g_err), "bad sizes: n=%d prefix_len=%d n_heads=%d kv_stride=%d", n, prefix_len, n_heads, kv_stride);
        return LLMCAD_ERR_INVALID_ARG;
    }
    if (n > kMaxNodes) {
        snprintf(g_err, sizeof(g_err), "n=%d exceeds the %d nodes a mask table holds", n, kMaxNodes);
        return LLMCAD_ERR_UNSUPPORTED;
    }
    if (n_heads > 65535) { snprintf(g_err, sizeof(g_err), "n_heads=%d exceeds 65535", n_heads); return LLMCAD_ERR_UNSUPPORTED; }
    // the kernels move rows as 16-byte vectors and bulk copies: a misaligned buffer would fault on the device
    if (((reinterpret_cast<uintptr_t>(q) | reinterpret_cast<uintptr_t>(k) | reinterpret_cast<uintptr_t>(v) |
          reinterpret_cast<uintptr_t>(o)) & 15) != 0) {
        snprintf(g_err, sizeof(g_err), "q, k, v and o must be 16-byte aligned");
        return LLMCAD_ERR_INVALID_ARG;
    }

    // Set-up, once per device, with that device current: in host code the array's name is only a
    // stand-in, the address the kernels need comes from the runtime.
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        snprintf(g_err, sizeof(g_err), "no usable current device");
        return LLMCAD_ERR_CUDA;
    }
    // (two host threads making their first call at once both look the address up and store the same value)
    if (__atomic_load_n(&g_scratch_ptr[dev], __ATOMIC_ACQUIRE) == nullptr) {
        void *ptr = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
        if (e != cudaSuccess || ptr == nullptr) {
            snprintf(g_err, sizeof(g_err), "cudaGetSymbolAddress: %s", cudaGetErrorString(e));
            return LLMCAD_ERR_CUDA;
        }
        __atomic_store_n(&g_scratch_ptr[dev], ptr, __ATOMIC_RELEASE);
    }
    int32_t *status = status_out != nullptr ? status_out : static_cast<int32_t *>(__atomic_load_n(&g_scratch_ptr[dev], __ATOMIC_ACQUIRE));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) {
        // neither kernel needs global scratch, and both make the mask table and set the status word themselves; same
        // choice as the regular entry point
        if (attention_prefers_t5(n))
            e = launch_attention_t5(q, k, v, n_heads, 128, kv_stride, prefix_len, n, nullptr, o, sms, status, st, nullptr, nullptr, 0, nullptr, 0, 0,
                                    kDefaultWaitLimitNs, nullptr, parent_idx);
        else
            e = launch_attention_tc(q, k, v, n_heads, 128, kv_stride, prefix_len, n, nullptr, o, sms, status, st, nullptr, nullptr, 0, nullptr, 0, 0,
                                    nullptr, parent_idx);
    }
    if (e != cudaSuccess) {
        snprintf(g_err, sizeof(g_err), "CUDA: %s", cudaGetErrorString(e));
        return LLMCAD_ERR_CUDA;
    }
    return LLMCAD_OK;
}
