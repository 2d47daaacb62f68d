// A layer group as a replayable object.  An engine that keeps its K/V pools and compact caches at
// fixed addresses calls the same group with the same arguments for every request; the launches of that call are recorded
// once in a CUDA graph and replayed.  The plan holds the recorded launches and an event that orders its own replays; inputs,
// outputs and the workspace stay the caller's, and what a launch computes is exactly what wkv_compress_group
// computes on the buffers' contents at that moment.
//
// A graph starts behind the one in front when that has ended, on a tick of 2 us.  Where all recorded kernels are programmatic
// dependents (one wave on the tensor-core path) they are therefore launched one by one from the recorded parameters, so that
// the first comes into the tail of the replay in front.  Replays back to back, graph / kernels, us: 8 heads x 4,096 keys
// 18.4 / 16.6, 16,384 39.1 / 36.1, 32,768 56.0 / 53.6.  Two instances of one graph never run at once, whatever streams they
// are on; kernels of two streams might, so that an event is recorded behind each replay and another stream than the one
// before is put behind it, on the device.  (The next replay on the same stream still comes into the tail of the one in front:
// 52.06 / 52.12 us without and with the event, 8 heads x 32,768 keys.)
#include "wkv_internal.cuh"

#include <mutex>
#include <new>

struct wkv_group_plan {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    uint64_t kernels = 0;   // kernel launches one replay stands for
    static constexpr int kChain = 4;
    int chain = 0;          // kernels that may be launched one by one, 0: the graph is replayed
    cudaKernelNodeParams params[kChain];
    int cluster[kChain];
    int device = -1;
    cudaEvent_t done = nullptr;             // behind the last replay that was launched kernel by kernel
    std::mutex mutex;                       // of `chain` and what follows
    bool launched = false;                  // `done` has been recorded, on the stream of this number (no other has had it)
    unsigned long long stream_id = 0;
};

using namespace wkv;

// The recorded kernels, in order, where there are only programmatic dependents: every kernel of the group call that is not
// launched cooperatively is one (launch_pdl).
static void find_chain(wkv_group_plan *plan)
{
    constexpr int kChain = wkv_group_plan::kChain;
    cudaGraphNode_t node = nullptr;
    size_t n = 1, total = 0;
    int count = 0;
    if (cudaGetDevice(&plan->device) != cudaSuccess || cudaGraphGetNodes(plan->graph, nullptr, &total) != cudaSuccess ||
        cudaGraphGetRootNodes(plan->graph, nullptr, &n) != cudaSuccess || n != 1 ||
        cudaGraphGetRootNodes(plan->graph, &node, &n) != cudaSuccess)
        return (void)cudaGetLastError();
    for (;;) {
        cudaGraphNodeType type;
        cudaLaunchAttributeValue cooperative = {}, cluster = {};
        if (count == kChain || cudaGraphNodeGetType(node, &type) != cudaSuccess || type != cudaGraphNodeTypeKernel ||
            cudaGraphKernelNodeGetParams(node, &plan->params[count]) != cudaSuccess || plan->params[count].extra ||
            cudaGraphKernelNodeGetAttribute(node, cudaLaunchAttributeCooperative, &cooperative) != cudaSuccess || cooperative.cooperative ||
            cudaGraphKernelNodeGetAttribute(node, cudaLaunchAttributeClusterDimension, &cluster) != cudaSuccess)
            return (void)cudaGetLastError();
        plan->cluster[count++] = cluster.clusterDim.x > 1 ? (int)cluster.clusterDim.x : 1;
        cudaGraphEdgeData edges[2];
        cudaGraphNode_t next[2];
        n = 0;
        if (cudaGraphNodeGetDependentNodes_v2(node, nullptr, nullptr, &n) != cudaSuccess || n > 1) return (void)cudaGetLastError();
        if (n == 0) break;
        if (cudaGraphNodeGetDependentNodes_v2(node, next, edges, &n) != cudaSuccess) return (void)cudaGetLastError();
        node = next[0];
    }
    if ((size_t)count == total) plan->chain = count;
}

static cudaError_t launch_kernel(const cudaKernelNodeParams &p, int cluster, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = p.gridDim;
    cfg.blockDim = p.blockDim;
    cfg.dynamicSmemBytes = p.sharedMemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    cfg.numAttrs = pdl_attributes(attr, cluster);
    return cudaLaunchKernelExC(&cfg, p.func, p.kernelParams);
}

// whether this launch may go kernel by kernel: on a stream of the plan's device, whose number is then in `id`
static bool may_chain(const wkv_group_plan *plan, cudaStream_t stream, unsigned long long &id)
{
    int device = -1;
    if (plan->chain && cudaGetDevice(&device) == cudaSuccess && device == plan->device && cudaStreamGetId(stream, &id) == cudaSuccess)
        return true;
    (void)cudaGetLastError();
    return false;
}

// A replay, behind the one before it.  A failure leaves the plan as it was, but for kernels that have been launched: those
// are the replay before the next one.
static cudaError_t replay(wkv_group_plan *plan, cudaStream_t stream)
{
    cudaStreamCaptureStatus capture;
    if (cudaStreamIsCapturing(stream, &capture) != cudaSuccess || capture != cudaStreamCaptureStatusNone) {
        (void)cudaGetLastError();
        return cudaGraphLaunch(plan->exec, stream);     // a graph is not launched into a recording: refused as such
    }
    unsigned long long id = 0;
    const bool kernels = may_chain(plan, stream, id);
    cudaError_t err = cudaSuccess;
    if (plan->launched && (!kernels || plan->stream_id != id)) err = cudaStreamWaitEvent(stream, plan->done, 0);
    if (err != cudaSuccess) return err;
    if (!kernels) {
        err = cudaGraphLaunch(plan->exec, stream);
        if (err == cudaSuccess) plan->chain = 0;        // graphs order themselves, and nothing tells a kernel when one has ended
        return err;
    }
    int n = 0;
    while (n < plan->chain && (err = launch_kernel(plan->params[n], plan->cluster[n], stream)) == cudaSuccess) ++n;
    if (n > 0) {
        const cudaError_t recorded = cudaEventRecord(plan->done, stream);
        if (err == cudaSuccess) err = recorded;
        plan->launched = true;
        plan->stream_id = id;
    }
    return err;
}

extern "C" {

int wkv_group_plan_create(const wkv_shape *s, int32_t n_layers, const void *q_obs_leader, const float *lse_obs,
                          const void *const *k_layers, const void *const *v_layers, void *const *k_out_layers,
                          void *const *v_out_layers, float *window_scores, int32_t *window_idx,
                          int32_t *kept_len, const int32_t *cu_seqlens_out, int32_t keep_capacity,
                          void *workspace, size_t workspace_bytes, wkv_group_plan **plan_out)
{
    if (!plan_out) {
        set_error_detail("plan_out is NULL");
        return WKV_ERR_NULL;
    }
    *plan_out = nullptr;
    cudaStream_t cap = nullptr;
    int st = check_cuda(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking), "stream for recording the plan");
    if (st != WKV_OK) return st;
    wkv_group_plan *plan = new (std::nothrow) wkv_group_plan;
    if (!plan) {
        cudaStreamDestroy(cap);
        set_error_detail("out of host memory");
        return WKV_ERR_CUDA;
    }
    st = check_cuda(cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal), "begin recording the plan");
    if (st == WKV_OK) {
        const uint64_t before = launches_so_far();
        // the arguments are validated here exactly as by the direct call; nothing runs yet
        const int call = compress_group_entry(s, n_layers, q_obs_leader, lse_obs, k_layers, v_layers, k_out_layers,
                                              v_out_layers, window_scores, window_idx, kept_len, cu_seqlens_out,
                                              keep_capacity, workspace, workspace_bytes, cap);
        plan->kernels = launches_so_far() - before;
        const cudaError_t end = cudaStreamEndCapture(cap, &plan->graph);   // always ends the recording
        st = call != WKV_OK ? call : check_cuda(end, "end recording the plan");
        // what was counted while recording did not run
        count_launches(-(int)plan->kernels);
    }
    if (st == WKV_OK) st = check_cuda(cudaGraphInstantiate(&plan->exec, plan->graph, 0), "instantiating the plan");
    if (st == WKV_OK) st = check_cuda(cudaEventCreateWithFlags(&plan->done, cudaEventDisableTiming), "event of the plan");
    if (st == WKV_OK) find_chain(plan);
    cudaStreamDestroy(cap);
    if (st != WKV_OK) {
        wkv_group_plan_destroy(plan);
        return st;
    }
    *plan_out = plan;
    return WKV_OK;
}

int wkv_group_plan_launch(wkv_group_plan *plan, void *cuda_stream)
{
    if (!plan || !plan->exec) {
        set_error_detail("plan is NULL");
        return WKV_ERR_NULL;
    }
    const cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    std::lock_guard<std::mutex> lock(plan->mutex);
    const int st = check_cuda(replay(plan, stream), "launching the plan");
    if (st == WKV_OK) count_launches((int)plan->kernels);
    return st;
}

void wkv_group_plan_destroy(wkv_group_plan *plan)
{
    if (!plan) return;
    if (plan->done) cudaEventDestroy(plan->done);
    if (plan->exec) cudaGraphExecDestroy(plan->exec);
    if (plan->graph) cudaGraphDestroy(plan->graph);
    delete plan;
}

}  // extern "C"
