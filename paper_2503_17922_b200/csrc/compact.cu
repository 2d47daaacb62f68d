// In-place compaction (section 2.2.2 during prefill: the compact cache of a layer takes the place of
// the layer's full K/V inside the buffer the prefill wrote them to).  The retained rows of a unit move
// to the front of the unit's own rows: output row r comes from source row src(r) >= r (window indices
// ascend, and the observation rows are the last rows of the sequence), so rows only ever move toward
// lower addresses.
//
// A parallel copy can still destroy a source row before it has been read: output window w lies on
// source window w, which an earlier output slot may need.  The kernel therefore gives a whole (unit,
// tensor) to one thread-block cluster and lets it walk the output rows in ascending batches: all source
// rows of a batch are read into registers, the cluster synchronises, then the batch is written.  Inside
// a batch every read precedes every write; a later batch reads only rows at or behind its own output
// rows, which lie behind everything written so far, so one barrier per batch is enough.  Clusters never
// touch each other's units.
//
// Bound by HBM (two passes over the retained rows) once enough SMs have loads in flight: 2 x 64 KB per
// SM in registers.  One block per (unit, tensor) left 132 of 148 SMs idle when a layer of 8 heads is
// compacted alone and needed four batches in a row (33 us for 16 MB moved); a cluster of eight takes the
// same layer in one batch.
#include "wkv_internal.cuh"

namespace wkv {
namespace {

constexpr int kThreads = 512;
constexpr int kVecs = 8;              // 16-byte vectors per thread and batch: 64 KB per block in flight, two blocks per SM
constexpr int kMaxCluster = 8;        // portable cluster size
constexpr int kMinVecs = 2;           // no more blocks per cluster than leave every thread this many vectors
constexpr int kResident = 264;        // blocks that fit at once in clusters of eight (33 clusters)

struct CompactParams {
    KShape s;
    InplaceTable tab;
    const int *window_idx;
    int cluster;          // blocks per (unit, tensor)
    int vec_per_row;
    int vec_shift, omega_shift;   // log2 of vec_per_row and of omega where they are powers of two, else -1
    int elem_bytes;
    int slots_per_block;  // chain form: slots whose chains' heads a block looks for
};

// every access of the cluster's threads before the barrier precedes every access after it
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__global__ void __launch_bounds__(kThreads, 2)
compact_inplace_kernel(const __grid_constant__ CompactParams prm)
{
    const KShape &s = prm.s;
    pdl_trigger();
    pdl_wait();
    const int cs = prm.cluster, unit = blockIdx.x / cs, rank = blockIdx.x - unit * cs, tensor = blockIdx.y;
    const int b = unit / s.hkv, h = unit % s.hkv;
    const int *idx = prm.window_idx + (size_t)unit * s.k_max;
    const int vpr = prm.vec_per_row;
    const int rows_per_batch = max(1, (cs * kThreads * kVecs) / vpr);
    // row and window slot of the thread's vectors in the batch at row r0
    auto over = [](int x, int by, int shift) { return shift >= 0 ? x >> shift : x / by; };
    auto row_of = [&](int r0, int u) { return r0 + over((int)threadIdx.x + (u * cs + rank) * kThreads, vpr, prm.vec_shift); };
    // A vector's window index waits in the registers that its 16 bytes go to.  The first batch's windows and the unit's
    // last one are looked up before it is known how many are selected, which takes a trip to memory of its own.
    int4 val[kVecs];
    auto load_windows = [&](int r0) {
#pragma unroll
        for (int u = 0; u < kVecs; ++u) {
            const int slot = over(row_of(r0, u), s.omega, prm.omega_shift);
            val[u].x = slot < s.k_max ? idx[slot] : -1;
        }
    };
    load_windows(0);
    const int wi_last = idx[s.k_max - 1];
    const SeqInfo si = seq_info(s, b);
    const int n = si.n;
    const int n_r = n > s.alpha ? n - s.alpha : 0;
    const int kw = num_windows(n, s.alpha, s.omega);
    const int k = num_selected_capped(n, s.alpha, s.omega, si.budget, s.k_max);
    int review_rows = k * s.omega;
    if (k > 0 && (k == s.k_max ? wi_last : idx[k - 1]) == kw - 1) review_rows -= kw * s.omega - n_r;
    const int kept = review_rows + (n - n_r);

    const long long row_vecs = s.st * prm.elem_bytes / 16;
    int4 *base = reinterpret_cast<int4 *>(static_cast<char *>(prm.tab.ptr[tensor]) +
                                          (si.off * s.st + b * s.sb + h * s.sh) * (long long)prm.elem_bytes);
    for (int r0 = 0; r0 < kept; r0 += rows_per_batch) {
        const int n_vec = min(rows_per_batch, kept - r0) * vpr;
        if (r0 > 0) load_windows(r0);
        unsigned moves = 0u;      // bit u: vector u of the thread has somewhere to go
#pragma unroll
        for (int u = 0; u < kVecs; ++u) {
            const int v = (int)threadIdx.x + (u * cs + rank) * kThreads;
            if (v < n_vec) {
                const int r = row_of(r0, u), slot = over(r, s.omega, prm.omega_shift), wi = val[u].x;
                int src_row;
                // an entry that is no window of this sequence, or that lies before its own slot (a
                // list that is not an ascending selection), is skipped: the row stays as it is
                if (r < review_rows) src_row = wi < slot || wi >= kw ? -1 : (wi - slot) * s.omega + r;
                else src_row = n_r + (r - review_rows);
                if (src_row >= 0 && src_row < n && src_row != r) {
                    val[u] = base[(long long)src_row * row_vecs + (v - (r - r0) * vpr)];
                    moves |= 1u << u;
                }
            }
        }
        cluster_barrier();      // every source row of the batch has been read
#pragma unroll
        for (int u = 0; u < kVecs; ++u)
            if (moves >> u & 1u) {
                const int v = (int)threadIdx.x + (u * cs + rank) * kThreads, r = row_of(r0, u);
                base[(long long)r * row_vecs + (v - (r - r0) * vpr)] = val[u];
            }
    }
}

// ---------------------------------------------------------------------------------------------
// Few of the windows retained, but more rows than a cluster holds at once: compaction by chains, without any barrier.
//
// Output slot t is exactly where source window t lies, so writing slot t must only come after the read of window
// t, which at most one other slot does: the slot p < t with idx[p] = t.  Slots linked this way form chains
// t, idx[t], idx[idx[t]], ..., as long as the window's number is also a slot's.  One warp walks a chain from
// its head (a slot whose own window is not selected): the copy of one slot has read the window that the next one
// overwrites.  Chains are independent of one another.  With a share f of the windows selected a chain grows by 1/f per
// link, so at most half of the windows leaves chains of a few links: the kernel above, which needs a barrier of all of a
// unit's blocks between reading and writing, serves the rest.  The observation rows overwrite a stretch of windows
// at the end of the compact cache; the warp that moves them first walks the chains that read that stretch.
// 8 heads x 65,536 keys, 12 %, one layer: 34.4 us -> 19.6 us; 32,768 keys: 18.6 us -> 14.8 us.
// ---------------------------------------------------------------------------------------------
constexpr int kChainThreads = 256;
constexpr int kChainWarps = kChainThreads / 32;
constexpr int kChainVecs = 8;             // 16-byte vectors in flight per lane
constexpr int kChainMaxK = 12288;         // window indices of a unit in 48 KB of shared memory

__device__ __forceinline__ int4 ld_once(const int4 *p)
{
    int4 v;
    asm volatile("ld.global.L1::no_allocate.v4.s32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}

__global__ void __launch_bounds__(kChainThreads, 4)
compact_chain_kernel(const __grid_constant__ CompactParams prm)
{
    extern __shared__ int idx[];          // the unit's window indices
    const KShape &s = prm.s;
    pdl_trigger();
    pdl_wait();
    const int unit = blockIdx.y, tensor = blockIdx.z;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < s.k_max; i += kChainThreads) idx[i] = prm.window_idx[(size_t)unit * s.k_max + i];
    const int b = unit / s.hkv, h = unit % s.hkv;
    const SeqInfo si = seq_info(s, b);
    const int n = si.n;
    const int n_r = n > s.alpha ? n - s.alpha : 0, obs_rows = n - n_r;
    const int kw = num_windows(n, s.alpha, s.omega);
    const int k = num_selected_capped(n, s.alpha, s.omega, si.budget, s.k_max);
    __syncthreads();
    int review_rows = k * s.omega;
    if (k > 0 && idx[k - 1] == kw - 1) review_rows -= kw * s.omega - n_r;

    const int vpr = prm.vec_per_row;
    const long long row_vecs = s.st * prm.elem_bytes / 16;
    int4 *base = reinterpret_cast<int4 *>(static_cast<char *>(prm.tab.ptr[tensor]) +
                                          (si.off * s.st + b * s.sb + h * s.sh) * (long long)prm.elem_bytes);
    // moves n_rows rows toward lower addresses, in ascending pieces: every piece is read before it is written
    auto move_rows = [&](int src_row, int dst_row, int n_rows) {
        const int n_vec = n_rows * vpr;
        const int4 *sp = base + (long long)src_row * row_vecs;
        int4 *dp = base + (long long)dst_row * row_vecs;
        for (int v0 = lane; v0 - lane < n_vec; v0 += 32 * kChainVecs) {
            int4 val[kChainVecs];
            long long off[kChainVecs];
#pragma unroll
            for (int u = 0; u < kChainVecs; ++u) {
                const int v = v0 + u * 32;
                const int r = prm.vec_shift >= 0 ? v >> prm.vec_shift : v / vpr;
                off[u] = r * row_vecs + (v - r * vpr);
                if (v < n_vec) val[u] = ld_once(sp + off[u]);
            }
            __syncwarp();
#pragma unroll
            for (int u = 0; u < kChainVecs; ++u)
                if (v0 + u * 32 < n_vec) dp[off[u]] = val[u];
            __syncwarp();
        }
    };
    // the window that slot c takes, or -1 when it takes none: an entry that is no window of the sequence or lies
    // before its own slot is skipped, and the slot's own window stays where it is
    auto window_of = [&](int c) { const int w = idx[c]; return w > c && w < kw ? w : -1; };
    // the slot that reads window w from elsewhere, or -1
    auto reader_of = [&](int w) {
        int lo = 0, hi = min(k, w);        // idx[p] >= p, so p < w
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (idx[mid] < w) lo = mid + 1;
            else hi = mid;
        }
        return lo < min(k, w) && idx[lo] == w && window_of(lo) == w ? lo : -1;
    };
    auto under_observation = [&](int w) {  // the observation rows will be written over this window
        return w * s.omega < review_rows + obs_rows && w * s.omega + s.omega > review_rows;
    };
    auto walk = [&](int c) {               // the whole chain from slot c on
        while (c < k) {
            const int w = window_of(c);
            if (w < 0) return;
            move_rows(w * s.omega, c * s.omega, min(s.omega, n_r - w * s.omega));
            c = w;
        }
    };
    auto leads_under = [&](int c) {        // a chain from slot c on reads what the observation rows overwrite
        while (c < k) {
            const int w = window_of(c);
            if (w < 0) return false;
            if (under_observation(w)) return true;
            c = w;
        }
        return false;
    };

    if (blockIdx.x + 1 < gridDim.x) {
        const int end = min(k, (int)(blockIdx.x + 1) * prm.slots_per_block);
        for (int t = blockIdx.x * prm.slots_per_block + warp; t < end; t += kChainWarps)
            if (window_of(t) >= 0 && reader_of(t) < 0 && !leads_under(t)) walk(t);
    } else if (warp == 0) {
        const int w_end = obs_rows > 0 ? (review_rows + obs_rows - 1) / s.omega : -1;
        for (int w = review_rows / s.omega; w <= w_end && w < kw; ++w) {
            int c = reader_of(w);
            if (c < 0 || leads_under(w)) continue;       // (leads on to a later window of the stretch: walked with that one)
            for (int p; (p = reader_of(c)) >= 0;) c = p;
            walk(c);
        }
        if (n_r != review_rows) move_rows(n_r, review_rows, obs_rows);
    }
}

}  // namespace

cudaError_t launch_compact_inplace(const KShape &ks, int elem_bytes, int n_tensors, const InplaceTable &tab,
                                   const int *window_idx, cudaStream_t stream)
{
    CompactParams prm;
    prm.s = ks;
    prm.tab = tab;
    prm.window_idx = window_idx;
    prm.vec_per_row = ks.d * elem_bytes / 16;
    prm.elem_bytes = elem_bytes;
    prm.vec_shift = prm.omega_shift = -1;
    for (int sh = 0; sh < 16; ++sh) {
        if ((1 << sh) == prm.vec_per_row) prm.vec_shift = sh;
        if ((1 << sh) == ks.omega) prm.omega_shift = sh;
    }
    // Blocks per (unit, tensor): as many as are resident at once (with one block of 1,024 threads per SM
    // only 15 clusters of eight fit, so the sixteenth of a layer of 8 heads ran alone), a power of two up to the portable cluster size, unless the rows are too few to occupy them.
    const int pairs = ks.batch * ks.hkv * n_tensors;
    const long long vecs = ((long long)ks.k_max * ks.omega + ks.alpha) * prm.vec_per_row;
    int cs = 1;
    while (cs < kMaxCluster && pairs * cs * 2 <= kResident && (long long)cs * kThreads * kMinVecs < vecs) cs *= 2;
    while (cs * kThreads * kVecs < prm.vec_per_row) cs *= 2;      // a batch is at least one row (of at most 128 KB)
    prm.cluster = cs;
    // By chains where a cluster would need more than one batch (every batch is a trip to memory and back behind a
    // barrier: 18.6 us against 14.8 us a layer at 8 heads x 32,768 keys, 12 %; with one batch the cluster is faster,
    // 7.2 us against 10.3 us at 8,192), at most half of the windows are retained (short chains) and the indices fit
    // shared memory.
    if (vecs > (long long)cs * kThreads * kVecs && 2ll * ks.k_max <= ks.kw_max && ks.k_max <= kChainMaxK) {
        prm.slots_per_block = 2 * kChainWarps;
        const dim3 grid((ks.k_max + prm.slots_per_block - 1) / prm.slots_per_block + 1, ks.batch * ks.hkv, n_tensors);
        const cudaError_t err = launch_pdl(compact_chain_kernel, grid, kChainThreads, (size_t)ks.k_max * sizeof(int), stream, 1, prm);
        if (err != cudaSuccess) return err;
        count_launches(1);
        return cudaSuccess;
    }
    const cudaError_t err = launch_pdl(compact_inplace_kernel, dim3(ks.batch * ks.hkv * cs, n_tensors), kThreads, 0, stream,
                                       cs, prm);
    if (err != cudaSuccess) return err;
    count_launches(1);
    return cudaSuccess;
}

}  // namespace wkv
