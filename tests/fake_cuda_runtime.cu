// The host side of the CUDA-core score path over a CUDA runtime that launches nothing: it answers the occupancy query,
// refuses what it is told to refuse, and writes down the kernels that it was asked to launch.  Built and driven by
// test_launch_rules.py; no GPU is involved.
#include "wkv_internal.cuh"

#include <map>
#include <string>
#include <string.h>

namespace {

struct Rules {
    int device = 0;             // ordinal that the calls run on; what the library remembers, it remembers per device
    size_t smem_limit = 0;      // dynamic shared memory that a kernel may ask for
    int clusters = 0;           // answer of the occupancy query
    int cooperative_error = 0;  // what a cooperative launch returns
} rules;
std::map<const void *, std::string> &kernels()      // filled by start-up code, whose order is nobody's
{
    static std::map<const void *, std::string> names;
    return names;
}
std::string launched;
cudaError_t last_error = cudaSuccess;

cudaError_t result(int e)
{
    if (e) last_error = (cudaError_t)e;
    return (cudaError_t)e;
}

}  // namespace

extern "C" {

// what the compiler's own start-up code calls
void **__cudaRegisterFatBinary(void *)
{
    static void *handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
char __cudaInitModule(void **) { return 1; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, CUstream_st *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaErrorNotSupported; }
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *)
{
    for (const char *known : {"score_fused_simt", "score_stats_simt", "score_pool_simt"})
        if (strstr(name, known)) kernels()[host] = known;
}
cudaError_t cudaLaunchKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t) { return result(cudaErrorNotSupported); }

// the runtime (two names are taken in this file, by the headers' versions for device code)
cudaError_t fake_get_device(int *device) __asm__("cudaGetDevice");
cudaError_t fake_get_last_error() __asm__("cudaGetLastError");
cudaError_t fake_get_device(int *device)
{
    *device = rules.device;
    return cudaSuccess;
}
cudaError_t fake_get_last_error()
{
    const cudaError_t e = last_error;
    last_error = cudaSuccess;
    return e;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int value)
{
    return result((size_t)value > rules.smem_limit ? cudaErrorInvalidValue : cudaSuccess);
}
cudaError_t cudaOccupancyMaxActiveClusters(int *clusters, const void *, const cudaLaunchConfig_t *)
{
    *clusters = rules.clusters;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *config, const void *kernel, void **)
{
    for (unsigned i = 0; i < config->numAttrs; ++i)
        if (config->attrs[i].id == cudaLaunchAttributeCooperative && rules.cooperative_error) return result(rules.cooperative_error);
    launched += (launched.empty() ? "" : " ") + kernels()[kernel];
    return cudaSuccess;
}

}  // extern "C"

namespace wkv {
void count_launches(int) {}
cudaError_t launch_topk(const KShape &, const float *, int *, int *, cudaStream_t)
{
    launched += " select_topk";
    return cudaSuccess;
}
}  // namespace wkv

// One select call on the CUDA-core path; returns its cudaError_t, writes the kernels launched into `log`, and leaves in
// *pending what a later cudaGetLastError() would report.
extern "C" int fake_select(int device, size_t smem_limit, int clusters, int cooperative_error, int f32, int rows, int head_dim,
                           int n, int window, char *log, size_t log_bytes, int *pending)
{
    rules.device = device;
    rules.smem_limit = smem_limit;
    rules.clusters = clusters;
    rules.cooperative_error = cooperative_error;
    launched.clear();
    last_error = cudaSuccess;
    wkv::KShape ks = {};
    ks.batch = ks.hkv = 1;
    ks.hq = ks.G = 1;
    ks.d = head_dim;
    ks.alpha = ks.R = rows;
    ks.omega = window;
    ks.p = 1;
    ks.max_seqlen = ks.total_rows = ks.n_cap = n;
    ks.kw_max = (n - rows + window - 1) / window;
    ks.k_max = 1;
    ks.nr_max = n - rows;
    wkv::Workspace ws = {};
    ws.r_pad = (rows + 63) / 64 * 64;
    ws.n_stat_chunks = (n + wkv::kStatChunk - 1) / wkv::kStatChunk;
    static char memory[16];          // never looked at: nothing runs
    const cudaError_t err = wkv::launch_score_simt(ks, f32 ? WKV_F32 : WKV_BF16, memory, memory, reinterpret_cast<float *>(memory),
                                                   nullptr, memory, ws, nullptr, nullptr, reinterpret_cast<int *>(memory),
                                                   reinterpret_cast<int *>(memory));
    strncpy(log, launched.c_str(), log_bytes - 1);
    *pending = last_error;
    return err;
}
