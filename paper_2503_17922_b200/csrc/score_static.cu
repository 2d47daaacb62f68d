// wkv_score_windows_static: the scoring stage for callers that cannot provide scratch memory.
//
// Some hosts of this library run where device allocation is off the table: inside a serving
// engine that has handed every byte of HBM to its own KV-cache pool at start-up, in a callback
// that must not synchronise the device, or under a memory budget audited at load time.  Such a
// caller cannot size and allocate the workspace wkv_score_windows() asks for.  This entry point
// needs none: its partial row statistics live in a fixed array that is part of the library image.
// Every GPU that loads the library therefore holds twice WKV_STATIC_SCRATCH_BYTES of device memory
// until the process exits, whether or not the entry point is ever called.
#include "wkv_internal.cuh"

#include <atomic>
#include <mutex>

namespace wkv {
namespace {

// The one scratch area, shared by every call on a device.  In host code this name is only a
// handle for cudaGetSymbolAddress(); the device address is looked up once per device below.
// (Shapes are admitted by what they would need with statistics of eight bytes each; the tensor-core kernel's take sixteen.)
static __device__ __align__(256) unsigned char g_static_scratch[2 * WKV_STATIC_SCRATCH_BYTES];

std::mutex g_setup_mutex;
void *g_scratch_addr[kMaxDevices] = {};

// Device address of the scratch array on the current device (looked up on the first call per device).
int static_scratch(void **out)
{
    int dev = -1;
    int st = check_cuda(cudaGetDevice(&dev), "cudaGetDevice");
    if (st != WKV_OK) return st;
    if (dev < 0 || dev >= kMaxDevices) {
        set_error_detail("device ordinal %d outside 0..%d", dev, kMaxDevices - 1);
        return WKV_ERR_LIMIT;
    }
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_addr[dev]) {
        void *p = nullptr;
        st = check_cuda(cudaGetSymbolAddress(&p, g_static_scratch), "cudaGetSymbolAddress(static scratch)");
        if (st != WKV_OK) return st;
        if (!p || (reinterpret_cast<uintptr_t>(p) & 255u)) {
            set_error_detail("static scratch has no usable device address");
            return WKV_ERR_CUDA;
        }
        g_scratch_addr[dev] = p;
    }
    *out = g_scratch_addr[dev];
    return WKV_OK;
}

}  // namespace
}  // namespace wkv

using namespace wkv;

extern "C" int wkv_score_windows_static(const wkv_shape *s, const void *q_obs, const void *k_leader,
                                        float *window_scores, float *token_scores, int32_t *device_status,
                                        void *cuda_stream)
{
    KShape ks;
    int st = resolve(s, ks);
    if (st != WKV_OK) return st;
    if (!q_obs || !k_leader || !window_scores) {
        set_error_detail("q_obs / k_leader / window_scores is NULL");
        return WKV_ERR_NULL;
    }
    Workspace ws = plan_workspace(ks, 0);            // scoring alone uses no unit's words but in the form that clears them
    // window_scores is the caller's here, so the part of the workspace that would hold them is not needed
    if (ws.counted_off > (size_t)WKV_STATIC_SCRATCH_BYTES) {
        set_error_detail("this shape needs %zu bytes of scratch, the built-in area holds %zu: "
                         "use wkv_score_windows with a caller-provided workspace",
                         ws.counted_off, (size_t)WKV_STATIC_SCRATCH_BYTES);
        return WKV_ERR_LIMIT;
    }
    void *scratch = nullptr;
    st = static_scratch(&scratch);
    if (st != WKV_OK) return st;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    // Scoring alone starts from the status word and the count of blocks; the number of the launch behind them goes on
    // counting, so that nothing an earlier call left behind passes for this one's.  (Two calls that overlap upset the
    // count of blocks and may leave the number as it was: the salt tells the next calls from them.)
    static std::atomic<unsigned> calls{0};
    ws.salt = 1u + calls.fetch_add(1u, std::memory_order_relaxed) % 255u;
    st = check_cuda(cudaMemsetAsync(static_cast<char *>(scratch) + ws.status_off, 0, ws.count_off + 16 - ws.status_off, stream),
                    "clearing the status word");
    // the pipelined kernel's words and statistics must start from zero
    if (st == WKV_OK && s->score_impl == WKV_SCORE_TCGEN05_PIPELINED)
        st = check_cuda(cudaMemsetAsync(static_cast<char *>(scratch) + ws.sync_off, 0, ws.stats_off - ws.sync_off, stream),
                        "clearing the synchronisation words");
    if (st != WKV_OK) return st;
    st = do_score(s, ks, ws, q_obs, k_leader, window_scores, token_scores, nullptr, nullptr, scratch, stream);
    if (st != WKV_OK) return st;
    if (device_status)
        st = check_cuda(cudaMemcpyAsync(device_status, static_cast<char *>(scratch) + ws.status_off, sizeof(int),
                                        cudaMemcpyDeviceToDevice, stream),
                        "copy of the status word");
    return st;
}
