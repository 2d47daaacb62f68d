// Shared-index gather (section 2.2.2): copies, for every layer tensor of the group, the rows of
// the selected review windows followed by the observation rows into the compact cache.  Pure bit
// copy with 16-byte vector accesses.
//
// The unit of work is one window (omega consecutive source rows = omega consecutive output rows)
// of one unit of one tensor, taken by one warp or a part of one: all its loads are issued before the first store
// (up to 8 x 16 bytes in flight per lane), and the index arithmetic is done once per window, not
// once per vector.  The observation rows are handled as extra windows behind the selected ones.
#include "wkv_internal.cuh"

#include <algorithm>

namespace wkv {
namespace {

constexpr int kThreads = 256;
// Rows that the GPU reads over the bus: so many blocks of 32 KB in flight, in all, fill it, and leave the copies that go
// back at the same time their share.  4 layers from pinned memory, one sequence of 8 heads x 8,192 keys: 851 us; 8 and 32
// blocks 858 and 868, all at once 883.  8 sequences x 4,096 keys: 3,100 us; with a block or more for each of the 128
// (unit, tensor) pairs 3,200.
constexpr int kBusBlocks = 16;
constexpr int kBatch = 8;             // independent 16-byte loads in flight per lane

struct GatherParams {
    KShape s;
    LayerTable tab;
    const int *window_idx;
    const int *cu_out;
    int keep_capacity;
    int vec_per_row;                  // 16-byte vectors per row
    int vec_shift;                    // log2(vec_per_row) when it is a power of two, else -1
    int elem_bytes;
    int lanes_shift;                  // log2 of the lanes that take one window
    int obs_slots;                    // ceil(alpha / omega)
    int pairs;                        // (unit, tensor) pairs
    bool early;                       // rows are fetched into L2 while the kernel in front still runs
    // paged output (page_size > 0): row r of unit (b, h) lives in page block_table[b][r / page_size]
    const int *block_table;           // [batch][max_pages]
    int max_pages, page_size, num_pages;
    long long page_vecs, head_vecs, row_vecs;   // strides of the page pool in 16-byte vectors
};

__device__ __forceinline__ int4 ld_stream(const int4 *p)
{
    int4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.s32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}
__device__ __forceinline__ void st_stream(int4 *p, const int4 &v)
{
    asm volatile("st.global.L1::no_allocate.v4.s32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y),
                 "r"(v.z), "r"(v.w)
                 : "memory");
}

// PAGED is a separate instantiation: its per-row page arithmetic would otherwise cost the plain copy
// registers it needs for its loads in flight; so is STRIDED, in which the grid may be smaller than the work: fewer blocks
// than a pair (unit, tensor) has windows for, and fewer than there are pairs.
template <bool PAGED, bool STRIDED>
__global__ void __launch_bounds__(kThreads, 4)
gather_kv_kernel(const __grid_constant__ GatherParams prm)
{
    const KShape &s = prm.s;
    pdl_trigger();
    const int lanes = 1 << prm.lanes_shift;
    if (!STRIDED && prm.early) {
        // A prefill that gathers layer by layer is a chain of these kernels, each with a ramp and a tail of its own: the
        // fetch fills the tail of the one in front.  Selection and four layers of 8 heads x 32,768 keys, 12 %: 53.4 us,
        // 56.1 without.
        const int slot = (blockIdx.x * kThreads + threadIdx.x) >> prm.lanes_shift;
        fetch_window(s, static_cast<const char *>(prm.tab.src[blockIdx.z]), prm.elem_bytes, blockIdx.y,
                     slot < s.k_max ? __ldcg(prm.window_idx + (size_t)blockIdx.y * s.k_max + slot) : -1, threadIdx.x & (lanes - 1), lanes);
    }
    pdl_wait();
    int pair = blockIdx.y;            // STRIDED: the pair, else the unit
    do {
        const int unit = STRIDED ? pair % (s.batch * s.hkv) : pair, tensor = STRIDED ? pair / (s.batch * s.hkv) : blockIdx.z;
        const int b = unit / s.hkv, h = unit % s.hkv;
        // The window and the unit's last one are looked up before it is known how many are selected (that takes a trip to
        // memory of its own): the chain from launch to the first row is one trip shorter.
        const int *idx = prm.window_idx + (size_t)unit * s.k_max;
        int slot = (blockIdx.x * kThreads + threadIdx.x) >> prm.lanes_shift;
        const int lane = threadIdx.x & (lanes - 1);
        int wi = slot < s.k_max ? idx[slot] : -1;
        const int wi_last = idx[s.k_max - 1];
        const SeqInfo si = seq_info(s, b);
        const int n = si.n;
        const int n_r = n > s.alpha ? n - s.alpha : 0;
        const int kw = num_windows(n, s.alpha, s.omega);
        const int k = num_selected_capped(n, s.alpha, s.omega, si.budget, s.k_max);

        // rows of the unit: the selected windows (only the last window of the sequence can be short,
        // and it can only be the last selected one), then the observation rows
        int review_rows = k * s.omega;
        if (k > 0 && (k == s.k_max ? wi_last : idx[k - 1]) == kw - 1) review_rows -= kw * s.omega - n_r;
        if (review_rows > n_r) review_rows = n_r;      // a list of all windows whose last entry is not the last window
        const int obs_rows = n - n_r;

        const int vpr = prm.vec_per_row;
        // strides are multiples of 16 bytes (checked on the host), so vector indexing is exact
        const long long src_row_vecs = s.st * prm.elem_bytes / 16;    // vectors between consecutive source rows
        const int4 *src = reinterpret_cast<const int4 *>(
            static_cast<const char *>(prm.tab.src[tensor]) +
            (si.off * s.st + b * s.sb + h * s.sh) * (long long)prm.elem_bytes);
        int4 *dst;
        long long dst_row_vecs;
        if (prm.cu_out) {
            dst = reinterpret_cast<int4 *>(prm.tab.dst[tensor]) +
                  ((long long)prm.cu_out[b] * s.hkv + h) * vpr;
            dst_row_vecs = (long long)s.hkv * vpr;
        } else {
            dst = reinterpret_cast<int4 *>(prm.tab.dst[tensor]) + (long long)unit * prm.keep_capacity * vpr;
            dst_row_vecs = vpr;
        }
        constexpr bool paged = PAGED;
        const bool src_dense = src_row_vecs == vpr, dst_dense = dst_row_vecs == vpr && !paged;
        const int *pages = paged ? prm.block_table + (size_t)b * prm.max_pages : nullptr;
        if (paged) dst = reinterpret_cast<int4 *>(prm.tab.dst[tensor]) + (long long)h * prm.head_vecs;

        auto move = [&](int slot, int wi) {
            int src_row0, dst_row0, n_rows;
            if (slot < k) {
                // an entry that is no window of this sequence (a list that no selection has written, or
                // that the caller filled wrongly) is skipped: the kernel never leaves the tensors
                if (wi < 0 || wi >= kw) return;
                src_row0 = wi * s.omega;
                n_rows = min(s.omega, n_r - src_row0);
                dst_row0 = slot * s.omega;
            } else {
                const int o = (slot - k) * s.omega;
                src_row0 = n_r + o;
                n_rows = min(s.omega, obs_rows - o);
                dst_row0 = review_rows + o;
            }
            if (n_rows <= 0) return;
            // dense output: a unit owns keep_capacity rows (cannot trigger while the device copies of
            // cu_seqlens / budgets equal the host copies the capacity was checked against)
            if (!prm.cu_out && !paged && dst_row0 + n_rows > prm.keep_capacity) return;
            if (paged) {
                // every row finds its page; a row whose page entry is missing or negative is skipped
                const int n_vec = n_rows * vpr;
                for (int v0 = lane; v0 < n_vec; v0 += lanes * kBatch) {
                    int4 val[kBatch];
                    long long doff[kBatch];
#pragma unroll
                    for (int u = 0; u < kBatch; ++u) {
                        const int v = v0 + u * lanes;
                        doff[u] = -1;
                        if (v < n_vec) {
                            const int r = prm.vec_shift >= 0 ? v >> prm.vec_shift : v / vpr;
                            const int c = v - r * vpr;
                            const int row = dst_row0 + r, page = row / prm.page_size;
                            const int phys = page < prm.max_pages ? pages[page] : -1;
                            if (phys >= 0 && phys < prm.num_pages)
                                doff[u] = (long long)phys * prm.page_vecs + (long long)(row - page * prm.page_size) * prm.row_vecs + c;
                            val[u] = ld_stream(src + (long long)(src_row0 + r) * src_row_vecs + c);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kBatch; ++u)
                        if (doff[u] >= 0) st_stream(dst + doff[u], val[u]);
                }
                return;
            }
            const int4 *sp = src + src_row0 * src_row_vecs;
            int4 *dp = dst + dst_row0 * dst_row_vecs;
            const int n_vec = n_rows * vpr;
            for (int v0 = lane; v0 < n_vec; v0 += lanes * kBatch) {
                int4 val[kBatch];
                int soff[kBatch], doff[kBatch];   // offsets inside one window: small
#pragma unroll
                for (int u = 0; u < kBatch; ++u) {
                    const int v = v0 + u * lanes;
                    if (v < n_vec) {
                        soff[u] = v;
                        doff[u] = v;
                        if (!src_dense || !dst_dense) {
                            const int r = prm.vec_shift >= 0 ? v >> prm.vec_shift : v / vpr;
                            const int c = v - r * vpr;
                            if (!src_dense) soff[u] = r * (int)src_row_vecs + c;
                            if (!dst_dense) doff[u] = r * (int)dst_row_vecs + c;
                        }
                        val[u] = ld_stream(sp + soff[u]);
                    }
                }
#pragma unroll
                for (int u = 0; u < kBatch; ++u)
                    if (v0 + u * lanes < n_vec) st_stream(dp + doff[u], val[u]);
            }
        };
        if (STRIDED) {
            const int stride = gridDim.x * (kThreads >> prm.lanes_shift);
            for (; slot < k + prm.obs_slots; slot += stride, wi = slot < k ? idx[slot] : -1) move(slot, wi);
        } else if (slot < k + prm.obs_slots) {
            move(slot, wi);
        }
    } while (STRIDED && (pair += gridDim.y) < prm.pairs);
}

}  // namespace

cudaError_t launch_gather(const KShape &ks, int elem_bytes, int n_tensors, const LayerTable &tab,
                          const int *window_idx, const int *cu_out, int keep_capacity,
                          cudaStream_t stream, const PagedOut *paged, bool over_bus, bool early)
{
    GatherParams prm;
    prm.block_table = nullptr;
    prm.max_pages = prm.page_size = prm.num_pages = 0;
    prm.page_vecs = prm.head_vecs = prm.row_vecs = 0;
    if (paged) {
        prm.block_table = paged->block_table;
        prm.max_pages = paged->max_pages;
        prm.page_size = paged->page_size;
        prm.num_pages = paged->num_pages;
        prm.page_vecs = paged->page_stride * elem_bytes / 16;
        prm.head_vecs = paged->head_stride * elem_bytes / 16;
        prm.row_vecs = paged->row_stride * elem_bytes / 16;
    }
    prm.s = ks;
    prm.tab = tab;
    prm.window_idx = window_idx;
    prm.cu_out = cu_out;
    prm.keep_capacity = keep_capacity;
    prm.vec_per_row = ks.d * elem_bytes / 16;
    prm.vec_shift = -1;
    for (int sh = 0; sh < 16; ++sh)
        if ((1 << sh) == prm.vec_per_row) prm.vec_shift = sh;
    prm.elem_bytes = elem_bytes;
    prm.obs_slots = (ks.alpha + ks.omega - 1) / ks.omega;
    // A window is taken by 32, 16 or 8 lanes, so that kBatch vectors per lane cover it in one go where that is possible.
    // One go per block is also best at any size: with 64 KB per block (up to four windows per warp, one after the
    // other) one layer of 8 heads x 983 rows in windows of 8 took 7.3 us instead of 5.4, four layers 10.4 instead of 7.2.
    const int window_vecs = ks.omega * prm.vec_per_row;
    prm.lanes_shift = 5;
    while (prm.lanes_shift > 3 && window_vecs <= (kBatch << (prm.lanes_shift - 1))) --prm.lanes_shift;
    const int slots_per_block = kThreads >> prm.lanes_shift;
    const int max_slots = ks.k_max + prm.obs_slots;
    int blocks = (max_slots + slots_per_block - 1) / slots_per_block;
    prm.early = early && !over_bus;
    prm.pairs = ks.batch * ks.hkv * n_tensors;
    dim3 grid(blocks, ks.batch * ks.hkv, n_tensors);
    if (over_bus) grid = dim3(std::max(1, std::min(blocks, kBusBlocks / prm.pairs)), std::min(prm.pairs, kBusBlocks));
    const cudaError_t err = launch_pdl(paged ? gather_kv_kernel<true, false> : (over_bus ? gather_kv_kernel<false, true> : gather_kv_kernel<false, false>), grid, kThreads, 0, stream, 1, prm);
    if (err != cudaSuccess) return err;
    count_launches(1);
    return cudaSuccess;
}

}  // namespace wkv
