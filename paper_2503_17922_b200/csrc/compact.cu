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
    prm.cluster = cs;
    const cudaError_t err = launch_pdl(compact_inplace_kernel, dim3(ks.batch * ks.hkv * cs, n_tensors), kThreads, 0, stream,
                                       cs, prm);
    if (err != cudaSuccess) return err;
    count_launches(1);
    return cudaSuccess;
}

}  // namespace wkv
