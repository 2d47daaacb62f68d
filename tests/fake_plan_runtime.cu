// The host side of a recorded group over a CUDA runtime that launches nothing: a graph of two kernels, each on a stream's
// list of what it was given, with failures where a case asks for them.  Built and driven by test_launch_rules.py; no GPU is
// involved.
#include "wkv_internal.cuh"

#include <stdarg.h>
#include <stdint.h>
#include <string.h>
#include <string>

namespace {

std::string calls;                  // what the runtime was asked to do, in order, done or refused
std::string fails;                  // the calls that fail, each with a blank behind it; a failure is used up
int device = 0;
bool capturing = false;
cudaGraphNode_t node(int i) { return reinterpret_cast<cudaGraphNode_t>((intptr_t)(i + 1)); }

cudaError_t did(const std::string &what)
{
    calls += (calls.empty() ? "" : " ") + what;
    const size_t at = fails.find(what + " ");
    if (at == std::string::npos) return cudaSuccess;
    fails.erase(at, what.size() + 1);
    return cudaErrorUnknown;
}
std::string name(cudaStream_t s) { return std::string(1, (char)('A' + (intptr_t)s)); }

}  // namespace

extern "C" {

cudaError_t fake_get_device(int *d) __asm__("cudaGetDevice");
cudaError_t fake_get_device(int *d) { return *d = device, cudaSuccess; }
cudaError_t fake_get_last_error() __asm__("cudaGetLastError");
cudaError_t fake_get_last_error() { return cudaSuccess; }
cudaError_t fake_synchronize() __asm__("cudaDeviceSynchronize");
cudaError_t fake_synchronize() { return did("device-synchronize"); }
cudaError_t fake_set_device(int) __asm__("cudaSetDevice");
cudaError_t fake_set_device(int d) { return device = d, cudaSuccess; }
cudaError_t fake_exchange(cudaStreamCaptureMode *) __asm__("cudaThreadExchangeStreamCaptureMode");
cudaError_t fake_exchange(cudaStreamCaptureMode *) { return cudaSuccess; }
cudaError_t fake_stream_create(cudaStream_t *s, unsigned) __asm__("cudaStreamCreateWithFlags");
cudaError_t fake_stream_create(cudaStream_t *s, unsigned) { return *s = reinterpret_cast<cudaStream_t>(25), cudaSuccess; }
cudaError_t fake_stream_destroy(cudaStream_t) __asm__("cudaStreamDestroy");
cudaError_t fake_stream_destroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { return *g = reinterpret_cast<cudaGraph_t>(1), cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s)
{
    *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamGetId(cudaStream_t s, unsigned long long *id) { return *id = 100 + (intptr_t)s, cudaSuccess; }
cudaError_t fake_event_create(cudaEvent_t *e, unsigned) __asm__("cudaEventCreateWithFlags");
cudaError_t fake_event_create(cudaEvent_t *e, unsigned) { return *e = reinterpret_cast<cudaEvent_t>(1), cudaSuccess; }
cudaError_t fake_event_destroy(cudaEvent_t) __asm__("cudaEventDestroy");
cudaError_t fake_event_destroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t fake_event_record(cudaEvent_t, cudaStream_t) __asm__("cudaEventRecord");
cudaError_t fake_event_record(cudaEvent_t, cudaStream_t s) { return did("record:" + name(s)); }
cudaError_t fake_wait(cudaStream_t, cudaEvent_t, unsigned) __asm__("cudaStreamWaitEvent");
cudaError_t fake_wait(cudaStream_t s, cudaEvent_t, unsigned) { return did("wait:" + name(s)); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long)
{
    return *e = reinterpret_cast<cudaGraphExec_t>(1), cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t fake_graph_launch(cudaGraphExec_t, cudaStream_t s) __asm__("cudaGraphLaunch");
cudaError_t fake_graph_launch(cudaGraphExec_t, cudaStream_t s)
{
    const cudaError_t e = did("graph:" + name(s));
    return capturing ? cudaErrorStreamCaptureUnsupported : e;
}
cudaError_t cudaGraphGetNodes(cudaGraph_t, cudaGraphNode_t *, size_t *n) { return *n = 2, cudaSuccess; }
cudaError_t cudaGraphGetRootNodes(cudaGraph_t, cudaGraphNode_t *nodes, size_t *n)
{
    if (nodes) nodes[0] = node(0);
    return *n = 1, cudaSuccess;
}
cudaError_t cudaGraphNodeGetType(cudaGraphNode_t, cudaGraphNodeType *t) { return *t = cudaGraphNodeTypeKernel, cudaSuccess; }
cudaError_t cudaGraphKernelNodeGetParams(cudaGraphNode_t n, cudaKernelNodeParams *p)
{
    memset(p, 0, sizeof(*p));
    p->func = reinterpret_cast<void *>(n);
    return cudaSuccess;
}
cudaError_t cudaGraphKernelNodeGetAttribute(cudaGraphNode_t, cudaLaunchAttributeID, cudaLaunchAttributeValue *v)
{
    memset(v, 0, sizeof(*v));
    return cudaSuccess;
}
cudaError_t cudaGraphNodeGetDependentNodes_v2(cudaGraphNode_t n, cudaGraphNode_t *next, cudaGraphEdgeData *, size_t *count)
{
    *count = n == node(0) ? 1 : 0;
    if (next && *count) next[0] = node(1);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *config, const void *kernel, void **)
{
    return did((kernel == node(0) ? "score:" : "gather:") + name(config->stream));
}

}  // extern "C"

namespace wkv {
void count_launches(int) {}
uint64_t launches_so_far() { return 0; }
void set_error_detail(const char *, ...) {}
int check_cuda(cudaError_t e, const char *) { return e == cudaSuccess ? WKV_OK : WKV_ERR_CUDA; }
int compress_group_entry(const wkv_shape *, int32_t, const void *, const float *, const void *const *, const void *const *, void *const *,
                         void *const *, float *, int32_t *, int32_t *, const int32_t *, int32_t, void *, size_t, void *)
{
    return WKV_OK;
}
}  // namespace wkv

// Replays a plan on the streams of `script` (A, B, ...; a digit makes that device current first, '!' makes the next stream one
// that is being recorded); `failing`: calls to fail, once each.  Writes the calls of the runtime into `log`, "|" behind each replay, with a
// "-" before it where the replay reported a failure.
extern "C" void fake_replays(const char *script, const char *failing, char *log, size_t log_bytes)
{
    wkv_group_plan *plan = nullptr;
    device = 0;
    fails.clear();
    const int st = wkv_group_plan_create(nullptr, 0, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0,
                                         nullptr, 0, &plan);
    calls = st == WKV_OK ? "" : "no plan";
    fails = failing;
    for (; plan && *script; ++script) {
        if (*script >= '0' && *script <= '9') device = *script - '0';
        else if (*script == '!') capturing = true;
        else {
            if (wkv_group_plan_launch(plan, reinterpret_cast<void *>((intptr_t)(*script - 'A'))) != WKV_OK) calls += " -";
            calls += " |";
            capturing = false;
        }
    }
    wkv_group_plan_destroy(plan);
    strncpy(log, calls.c_str(), log_bytes - 1);
}
