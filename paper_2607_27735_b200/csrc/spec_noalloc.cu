// spec_verify_attn_noalloc: verification attention for callers that cannot provide a workspace.
//
// Some hosts of this library never get to call cudaMalloc themselves: a plugin that is handed
// its input and output buffers by a runtime that owns all device memory, or code that runs
// after the framework's memory pool has taken the whole GPU.  For them the scratch that
// spec_verify_attn needs (cross-CTA counters, per-CTA partial outputs) lives in a fixed array
// inside the library image, kStaticScratchBytes per GPU, present on every device that loads the
// library until the process exits.
#include <mutex>

#include "spec_common.cuh"
#include "verify_sm100.cuh"

namespace {

constexpr size_t kStaticScratchBytes = 16u << 20;  // 16 MiB: one layer of the 8B shape at 32K context needs 11 MiB
constexpr int kMaxDevices = 64;

// In host code this name is only a handle for cudaGetSymbolAddress: it is not a device address.
static __device__ __align__(256) unsigned char g_scratch[kStaticScratchBytes];

std::mutex g_mutex;
void* g_scratch_ptr[kMaxDevices] = {};

// Device address of the scratch array on the current device (looked up once per device).
int scratch_address(void** out)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return SPEC_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_mutex);
    if (!g_scratch_ptr[dev]) {
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_scratch) != cudaSuccess || !ptr) {
            cudaGetLastError();
            return SPEC_ERR_CUDA;
        }
        g_scratch_ptr[dev] = ptr;
    }
    *out = g_scratch_ptr[dev];
    return SPEC_OK;
}

}  // namespace

extern "C" {

size_t spec_noalloc_scratch_bytes(void) { return kStaticScratchBytes; }

int spec_verify_attn_noalloc(const spec_kv_t* kv, const void* q, int32_t n_q, const int32_t* ctx_len,
                             int32_t max_ctx_len, int32_t stat_window, float* out, float* lse, float* stats,
                             int64_t stat_stride, void* cuda_stream)
{
    const int ctas = spec::verify_ctas_within(kv, n_q, max_ctx_len, kStaticScratchBytes);
    if (ctas < 0) return ctas;
    void* scratch = nullptr;
    const int rc = scratch_address(&scratch);
    if (rc != SPEC_OK) return rc;
    // The array keeps whatever the previous call left (possibly laid out for another shape): the
    // cross-CTA counters behind the status block must start at zero.  The status word itself is left alone, so that
    // an error nobody has read yet survives until spec_noalloc_read_status(), as with a caller's workspace.
    spec::KvView shape = {};
    shape.n_layers = kv->n_layers;
    shape.batch = kv->batch;
    shape.n_kv_heads = kv->n_kv_heads;
    size_t head = spec::verify_counter_bytes(shape);
    if (head > kStaticScratchBytes - spec::kStatusBytes) head = kStaticScratchBytes - spec::kStatusBytes;
    if (cudaMemsetAsync(static_cast<char*>(scratch) + spec::kStatusBytes, 0, head,
                        static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess)
        return SPEC_ERR_CUDA;
    return spec::verify_call(kv, q, n_q, ctx_len, max_ctx_len, stat_window, out, lse, stats, stat_stride, scratch,
                             kStaticScratchBytes, 0u, nullptr, ctas, cuda_stream);
}

int spec_noalloc_read_status(void* cuda_stream)
{
    void* scratch = nullptr;
    const int rc = scratch_address(&scratch);
    if (rc != SPEC_OK) return rc;
    return spec_read_status(scratch, cuda_stream);
}

}  // extern "C"
