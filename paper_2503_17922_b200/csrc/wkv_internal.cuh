// Internal declarations shared by the library's translation units (host side of
// the C ABI and the kernel launchers).  Not part of the public interface.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>
#include <stddef.h>

#include "wkv.h"

namespace wkv {

// Shape as the kernels see it: plain values, device pointers only.
struct KShape {
    int batch, hq, hkv, d;
    int alpha, omega, p;       // p already resolved from task/top_p (Eq. 4)
    int max_seqlen, budget;
    int total_rows;            // sum of the sequence lengths (rows of the packed layout)
    int G, R;                  // query heads per KV head; observation rows per unit = G*alpha
    int kw_max, k_max, nr_max; // leading sizes of window_scores / window_idx / token_scores
    int n_cap;                 // no sequence is taken to be longer than this on the device:
                               // min(max_seqlen, alpha + kw_max * omega), so that a device copy of
                               // cu_seqlens that disagrees with the host copy cannot lead a kernel
                               // past the arrays that were sized from the host copy
    const int *cu;             // device cu_seqlens or nullptr
    const int *budgets;        // device budgets or nullptr
    long long sb, sh, st;      // K/V element strides
    long long qsb, qsh, qst;   // Q_obs element strides
    float scale_log2;          // log2(e)/sqrt(d): logits are handled in base 2
};

// Per-sequence integers, the same formulas on host and device (Eq. 3 and the
// budget sentence after Eq. 4).
__host__ __device__ inline int num_windows(int n, int alpha, int omega)
{
    return n <= alpha ? 0 : (n - alpha + omega - 1) / omega;
}
__host__ __device__ inline int num_selected(int n, int alpha, int omega, int budget)
{
    int kw = num_windows(n, alpha, omega);
    int k = budget > alpha ? (budget - alpha) / omega : 0;
    return k < kw ? k : kw;
}
// the same, never beyond the leading size of window_idx (device side: budgets_dev is not trusted further)
__host__ __device__ inline int num_selected_capped(int n, int alpha, int omega, int budget, int k_max)
{
    const int k = num_selected(n, alpha, omega, budget);
    return k < k_max ? k : k_max;
}

struct SeqInfo {
    int n;          // context length
    long long off;  // first row of the sequence in the packed layout (0 when dense)
    int budget;
};

// EARLY: ahead of pdl_wait().  The kernel in front may still write the lengths, so they are read from L2 alone: a line that
// an ordinary load has put into L1 could serve the one behind the wait.
template <bool EARLY>
__device__ __forceinline__ int length_word(const int *p)
{
    return EARLY ? __ldcg(p) : *p;
}
template <bool EARLY = false>
__device__ inline SeqInfo seq_info(const KShape &s, int b)
{
    SeqInfo r;
    if (s.cu) {
        int lo = length_word<EARLY>(s.cu + b);
        r.n = length_word<EARLY>(s.cu + b + 1) - lo;
        // a device copy that disagrees with the host copy must not lead outside the packed tensor
        lo = lo < 0 ? 0 : (lo > s.total_rows ? s.total_rows : lo);
        r.n = r.n < 0 ? 0 : (r.n > s.n_cap ? s.n_cap : r.n);
        if (r.n > s.total_rows - lo) r.n = s.total_rows - lo;
        r.off = lo;
    } else {
        r.n = s.max_seqlen;
        r.off = 0;
    }
    r.budget = !EARLY && s.budgets ? s.budgets[b] : s.budget;
    return r;
}

// Workspace carve-up (all offsets 256-byte aligned).
struct Workspace {
    size_t status_off;   // int: device status word, only ever OR-ed by the kernels (0 = no error)
    size_t count_off;    // LaunchCount of the kernels that publish words, inside the status word's 64 bytes
    size_t sync_off;     // int [kSyncTickets + kSyncWordsPerUnit * units], self-resetting
    size_t pstats_off;   // u64 [units][n_stat_chunks][128]: self-validating (max, sum) entries of the pipelined kernel;
                         // zero between launches (the kernel that writes them clears them again)
    size_t stats_off;    // partial (max, sum) per row: float2 [units][n_stat_chunks][R_pad], or published words of 16 bytes
                         // [units][chunks][R_pad] (tensor-core kernel, CUDA-core form of one launch)
    size_t lse_off;      // float  [units][R_pad]                 log2 of the row normaliser
    size_t scores_off;   // float  [units][kw_max]                window scores when the caller passes none
    size_t entries_off;  // published window scores [units][kw_max] of 16 bytes (the same two, with selection)
    size_t total;
    size_t counted_off;  // scores_off as it would be with float2 statistics: what the built-in area admits shapes by
    unsigned salt;       // goes into the tags of published words (0 but for the built-in area)
    int looks;           // how often a block that can do without another's words looks for them
    bool alone;          // it does without all statistics but its own (test aid)
    int n_stat_chunks;
    int r_pad;
};

// words of the synchronisation area before the per-unit words; unit u owns four words from
// sync[kSyncTickets + 4u]: ticket count, and in the pipelined kernel arrivals of the statistics sweep, "selection
// published" flag and gather job counter; the second is the "selection left over" flag of the tensor-core kernel of one wave
constexpr int kSyncTickets = 16;
constexpr int kSyncWordsPerUnit = 4;
// The area has room for at least this many units whatever the shape (32 KB), so that what lies behind it never lands on
// the words of another shape: one workspace may serve shapes of up to so many units in turn.
constexpr int kSyncUnits = 2048;

// A look is a trip to L2 of 0.6 us or more.  The blocks of a launch that has the GPU to itself begin within a few us of one
// another, those of one that shares it with short kernels of other streams within some tens: 600 us and more of looking
// before a block takes it that another one cannot start.  (With 100 us two streams of different priority took 112 us for the
// pair of groups that takes 105 so, and 106 in cooperative launches.)
constexpr int kPatientLooks = 1000;

// per-device host state (kernel attributes, device properties) is kept for this many device ordinals
constexpr int kMaxDevices = 64;

constexpr int kStatChunk = 512;   // keys per partial-statistics chunk of the CUDA-core kernels

// Tensor-core kernels: key tiles of 128 (at most 16, +1 for window alignment, per item of the pipelined kernel;
// tc_max_chunk_tiles below for the other), and a grid aimed at one wave of the 148 SMs of a B200 when the
// problem is small enough for that.
constexpr int kTcTileKeys = 128;
constexpr int kTcMaxChunkTiles = 16;
constexpr int kTcTargetBlocks = 148;
constexpr int kTcMaxWindow = 1024;

// The pipelined kernel works through the units in waves whose keys fit the L2 cache together.
constexpr long long kTcWaveBytes = 80ll << 20;

// Key tiles a block of the tensor-core kernel may take per item: what its buffer of token scores holds when the
// chunk is rounded up to whole windows (37 tiles for windows of up to 128 tokens, 30 for 1,024).
constexpr int kTcChunkCap = 4864;
__host__ __device__ inline int tc_max_chunk_tiles(int omega) { return (kTcChunkCap - omega) / kTcTileKeys; }

// Shapes that the CUDA-core path may score and select in one launch, if its blocks, one per 64 keys, are resident together:
// up to 128 observation rows and windows that do not straddle 64 keys.
inline bool simt_fused_shape(const KShape &ks)
{
    const long long chunks = (ks.max_seqlen + kStatChunk - 1) / kStatChunk;
    return ks.R <= 128 && 64 % ks.omega == 0 && chunks * ks.batch * ks.hkv <= 128;
}

struct TcPlan {
    int units_per_wave;   // units swept together
    int chunks_per_unit;  // work items per unit
};
// What a wave costs beside its key tiles, in tiles per block: filling the pipeline, the hand-over of the
// statistics and the pooling take about 8 us, a tile 0.65 us per sweep with up to 128 observation rows and, with two
// accumulators per tile, about twice that with more.  Measured on shapes where the number decides (select call, us):
//   R = 128   35 units of 54 tiles, 1 wave of 27 tiles / 2 of 11: 62 / 69      40 of 465, 4 of 34 / 5 of 26: 261 / 273
//   R = 256   128 units of 165 tiles, 5 waves of 33 / 8 of 19: 530 / 509       40 of 465, 4 of 34 / 5 of 26: 429 / 426
//             32 of 460, 3 of 36 / 4 of 26: 343 / 345                          112 of 39, 2 of 20 / 4 of 8: 147 / 152
constexpr int tc_wave_overhead(int rows) { return rows <= 128 ? 6 : 4; }
inline TcPlan tc_plan(int units, int max_seqlen, int omega, int rows)
{
    // Every number of units per wave whose blocks are resident together is tried, and the one with the least (waves x
    // (tiles per block + overhead)) taken; tiles are those of the longest sequence.  The largest is not the best when
    // it leaves a last wave nearly empty: 24 units of 256 tiles as 21 + 3 are two waves of 37 tiles per block, as 12 + 12
    // two of 22.  Whether a wave's keys fit L2 between the two sweeps does not count: a wave costs more than reading
    // keys from HBM again beside the exponentials (8 sequences of 32-64 K keys, R = 256, one layer: 669 us with waves of at
    // most 104 MB, 599 us with up to 170 MB).
    TcPlan best;
    best.units_per_wave = 1;
    best.chunks_per_unit = 1;
    const int max_tiles = (max_seqlen + kTcTileKeys - 1) / kTcTileKeys;
    // a unit needs at least this many blocks (the token scores of a chunk live in shared memory)
    const int chunk_tiles = tc_max_chunk_tiles(omega);
    const int min_chunks = (max_tiles + chunk_tiles - 1) / chunk_tiles;
    int most = kTcTargetBlocks / min_chunks;
    if (most > units) most = units;
    if (most < 1) most = 1;
    long long best_cost = -1;
    for (int upw = most; upw >= 1; --upw) {
        int chunks = kTcTargetBlocks / upw;
        if (chunks < min_chunks) chunks = min_chunks;
        if (chunks > max_tiles) chunks = max_tiles;
        const long long waves = (units + upw - 1) / upw, tiles = (max_tiles + chunks - 1) / chunks;
        const long long cost = waves * (tiles + tc_wave_overhead(rows));
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best.units_per_wave = upw;
            best.chunks_per_unit = chunks;
        }
    }
    return best;
}
// The pipelined group kernel takes the units in waves too, but keeps TWO waves in flight (the
// statistics sweep runs one wave ahead of the scoring sweep), so two waves' keys share the L2 budget;
// with at least two units it always makes at least two waves, so that the gather of one wave's rows
// can run beside the scoring of the next.
struct PipePlan {
    int units_per_wave, chunks_per_unit, skew;
};
__host__ __device__ inline PipePlan pipe_plan(int units, int max_seqlen, int head_dim)
{
    PipePlan p;
    const long long unit_bytes = (long long)max_seqlen * head_dim * 2;
    const int max_tiles = (max_seqlen + kTcTileKeys - 1) / kTcTileKeys;
    const int min_chunks = (max_tiles + kTcMaxChunkTiles - 1) / kTcMaxChunkTiles;
    long long upw = (kTcWaveBytes / 2) / (unit_bytes > 0 ? unit_bytes : 1);
    if (upw > kTcTargetBlocks / min_chunks) upw = kTcTargetBlocks / min_chunks;
    if (upw > (units + 1) / 2) upw = (units + 1) / 2;
    if (upw < 1) upw = 1;
    p.units_per_wave = (int)upw;
    p.skew = units > p.units_per_wave ? 1 : 0;
    int a = kTcTargetBlocks / p.units_per_wave;
    if (a < 1) a = 1;
    if (a > max_tiles) a = max_tiles;
    p.chunks_per_unit = a > min_chunks ? a : min_chunks;
    return p;
}
// keys per block when `n_keys` keys are split over `chunks` blocks in whole tiles, rounded up to a
// multiple of `align` (1 for the statistics sweep, omega for the scoring sweep)
__host__ __device__ inline int tc_chunk_len(int n_keys, int chunks, int align)
{
    const int tiles = (n_keys + kTcTileKeys - 1) / kTcTileKeys;
    const int ct = (tiles + chunks - 1) / chunks;
    const int len = ct * kTcTileKeys;
    return (len + align - 1) / align * align;
}

// device status bits
constexpr int kStatusWaitExpired = 1;   // a bounded wait inside a kernel ran out; results are invalid

// Programmatic dependent launch: a kernel launched through launch_pdl() may be put on the SMs while the
// kernel before it in the stream still runs, once every block of that one has called pdl_trigger() or
// ended.  It must call pdl_wait() before it touches global memory; the wait ends when the kernel before it
// has completed and its writes are visible.  Because every kernel launched this way waits, "the kernel
// before it has completed" includes everything earlier in the stream.  Exceptions to waiting first: the CUDA-core
// score kernel reads Q, K and the lengths (which no kernel of this library writes) ahead of its wait, because the statistics
// kernel in front of it triggers only after its own wait, behind which everything that wrote them lies; what the
// statistics kernel writes is read, and anything is written, after the wait.  And the kernels that fetch rows into L2 ahead
// of theirs (fetch_window here, fetch_ahead in score_tc.cu) read lengths and indices for it, from L2 and for nothing else.
// Takes about 2 us off the gap
// between two kernels (a chain of short kernels: 4.1 us each without, 2.0 us with).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// A window's rows into L2, ahead of pdl_wait(): `lanes` lanes take its lines in turn.  Nothing is read that the kernel
// goes on with (L2 is where the GPU's memory is coherent: a line fetched early and written later is the written one), and
// an index that is not yet the final one is no more than a wasted fetch inside the tensor.
__device__ __forceinline__ void fetch_window(const KShape &s, const char *tensor, int elem_bytes, int unit, int window, int lane,
                                             int lanes)
{
    const int b = unit / s.hkv, h = unit - b * s.hkv;
    const SeqInfo si = seq_info<true>(s, b);
    const int n_r = si.n - s.alpha, row0 = window * s.omega;
    if (window < 0 || window >= num_windows(si.n, s.alpha, s.omega)) return;
    const long long row_bytes = s.st * elem_bytes;
    const int row_lines = (s.d * elem_bytes + 127) >> 7, rows = min(s.omega, n_r - row0);
    const char *at = tensor + (si.off * s.st + b * s.sb + h * s.sh) * (long long)elem_bytes + row0 * row_bytes;
    for (int x = lane; x < rows * row_lines; x += lanes) {
        const int r = x / row_lines;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(at + r * row_bytes + (long long)(x - r * row_lines) * 128));
    }
}
// `cluster`: blocks per cluster along x (1: none); the attributes of such a launch, and their number
inline int pdl_attributes(cudaLaunchAttribute (&attr)[2], int cluster)
{
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    return cluster > 1 ? 2 : 1;
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t stream,
                              int cluster, const Args &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    cfg.attrs = attr;
    cfg.numAttrs = pdl_attributes(attr, cluster);
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

Workspace plan_workspace(const KShape &ks, int sync_units = kSyncUnits);

// Launchers (each returns a cudaError_t from the launch).
cudaError_t launch_score_simt(const KShape &ks, int dtype, const void *q, const void *k,
                              float *window_scores, float *token_scores,
                              void *workspace, const Workspace &ws, cudaStream_t stream,
                              const float *lse_obs = nullptr, int *window_idx = nullptr,
                              int *kept_len = nullptr, bool group = false);
bool score_tc_supported(const KShape &ks, int dtype);
// window_idx / kept_len non-null: the selection is fused into the same launch.
// lse_obs non-null: float [B, H_q, alpha], natural log of Eq. 1's normaliser of every observation
// row, supplied by the caller; the statistics sweep is then skipped.
int launch_score_tc(const KShape &ks, const void *q, const void *k,
                    float *window_scores, float *token_scores, int *window_idx, int *kept_len,
                    void *workspace, const Workspace &ws, cudaStream_t stream, const float *lse_obs = nullptr);
// The pipelined group kernel (score_pipe.cu): scoring, selection and, with `gather`, the shared-index
// gather of every layer in one launch.  R <= 128 only.
struct LayerTable;
struct PipeGather {
    int n_tensors;
    const LayerTable *tab;
    const int *cu_out;
    int keep_capacity;
};
bool group_pipeline_supported(const KShape &ks, int dtype);
bool group_pipeline_can_gather(const KShape &ks, int elem_bytes, int n_tensors);
int launch_group_pipeline(const KShape &ks, const void *q, const void *k, float *window_scores, float *token_scores,
                          int *window_idx, int *kept_len, void *workspace, const Workspace &ws, cudaStream_t stream,
                          const float *lse_obs, const PipeGather *gather);
cudaError_t launch_topk(const KShape &ks, const float *window_scores, int *window_idx, int *kept_len,
                        cudaStream_t stream);

struct LayerTable {
    const void *src[2 * WKV_MAX_GROUP_LAYERS];
    void *dst[2 * WKV_MAX_GROUP_LAYERS];
};
// paged compact cache: strides of the page pool in elements
struct PagedOut {
    const int *block_table;   // device [batch][max_pages]
    int max_pages, page_size, num_pages;
    long long page_stride, head_stride, row_stride;
};
// over_bus: the rows are read from host memory (not for paged output).  early: the windows' rows are fetched into L2
// before the kernel in front has ended; for calls of their own, whose indices are final by then (a kernel that writes
// them releases nobody before it ends).  Not in the group call, whose gather may be released earlier.
cudaError_t launch_gather(const KShape &ks, int elem_bytes, int n_tensors, const LayerTable &tab,
                          const int *window_idx, const int *cu_out, int keep_capacity,
                          cudaStream_t stream, const PagedOut *paged = nullptr, bool over_bus = false,
                          bool early = false);
// compaction of every layer's K/V inside its own buffer (compact.cu)
struct InplaceTable {
    void *ptr[2 * WKV_MAX_GROUP_LAYERS];
};
cudaError_t launch_compact_inplace(const KShape &ks, int elem_bytes, int n_tensors, const InplaceTable &tab,
                                   const int *window_idx, cudaStream_t stream);

// Eq. 4 for one window of `size` values: mean of the p largest.  Elements are visited in the
// strict order (value descending, position ascending), so equal values are each taken once.
__device__ inline float pool_top_p(const float *w, int size, int p)
{
    if (p >= size) {
        float acc = 0.f;
        for (int x = 0; x < size; ++x) acc += w[x];
        return acc / (float)size;
    }
    float acc = 0.f, prev_v = INFINITY;
    int prev_i = -1;
    for (int round = 0; round < p; ++round) {
        float best_v = -INFINITY;
        int best_i = size;
        for (int x = 0; x < size; ++x) {
            float v = w[x];
            bool after_prev = v < prev_v || (v == prev_v && x > prev_i);
            if (after_prev && (v > best_v || best_i == size)) {
                best_v = v;
                best_i = x;
            }
        }
        acc += best_v;
        prev_v = best_v;
        prev_i = best_i;
    }
    return acc / (float)p;
}

// host side of the boundary, shared by the translation units that export entry points
int resolve(const wkv_shape *s, KShape &ks);            // validates the shape, fills the kernel-side copy
int check_cuda(cudaError_t e, const char *what);         // cudaError_t -> wkv_status with detail
// scoring; with window_idx / kept_len non-null also the selection (one launch on the tensor-core path)
// `gather` non-null: the caller wants the layers gathered as well; *gathered tells whether the launch
// that scored has done it (else the caller launches the gather kernel)
int do_score(const wkv_shape *s, const KShape &ks, const Workspace &ws, const void *q, const void *k,
             float *window_scores, float *token_scores, int *window_idx, int *kept_len, void *workspace,
             cudaStream_t stream, const float *lse_obs = nullptr, const PipeGather *gather = nullptr,
             bool *gathered = nullptr);

void count_launches(int n);
uint64_t launches_so_far();
// the group call behind wkv_compress_group / wkv_compress_group_lse (lse_obs may be null)
int compress_group_entry(const wkv_shape *s, int32_t n_layers, const void *q_obs_leader, const float *lse_obs,
                         const void *const *k_layers, const void *const *v_layers, void *const *k_out_layers,
                         void *const *v_out_layers, float *window_scores, int32_t *window_idx, int32_t *kept_len,
                         const int32_t *cu_seqlens_out, int32_t keep_capacity, void *workspace,
                         size_t workspace_bytes, void *cuda_stream);
void set_error_detail(const char *fmt, ...);

}  // namespace wkv
