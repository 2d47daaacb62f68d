// In-place compaction (section 2.2.2 during prefill: the compact cache of a layer takes the place of
// the layer's full K/V inside the buffer the prefill wrote them to).  The retained rows of a unit move
// to the front of the unit's own rows: output row r comes from source row src(r) >= r (window indices
// ascend, and the observation rows are the last rows of the sequence), so rows only ever move toward
// lower addresses.
//
// A parallel copy can still destroy a source row before it has been read: output window w lies on
// source window w, which an earlier output slot may need.  The kernel therefore gives a whole (unit,
// tensor) to one thread-block cluster and lets it walk the output rows in ascending batches of what its
// registers hold.  A batch reads only rows at or behind its own output rows, which lie behind everything written so
// far, so reads never wait.  Writes do: output row r may be written once every output row whose source is
// r has read it.  src(r) ascends, so when the cluster has read everything before output row r, no row before src(r)
// is needed any more, and output rows r .. src(r) - 1 are free to be written.  Where that stretch holds a
// batch or more, its batches are copied one after the other without any barrier; where it does not (rows that move by
// less than a batch), a batch is read whole, the cluster synchronises, and then it is written.  Clusters
// never touch each other's units.
//
// With a share f of the windows selected evenly the free stretch grows by 1/f each time, so nearly all rows are
// copied like the gather's; at worst (a contiguous run behind a small offset) every batch costs a barrier, a trip
// to memory and back.  Nothing takes more steps than that, whatever is selected.
//
// Bound by HBM (two passes over the retained rows) where there are enough of them, by launch, index, row, barrier and
// store one after the other where a layer is one batch.  One layer of 8 heads, 12 % of the windows retained, calls
// back to back, in us: scattered windows / windows 1..k (every window moves by one) / 90 % of the opening stretch
//   16,384 keys    9.0 /  8.9 /  8.8      32,768 keys   12.0 / 12.8 / 12.7      65,536 keys   18.8 / 21.3 / 21.1
// against 13.1 / 383 / 63 at 32,768 and 16.7 / 785 / 106 at 65,536 with one warp per chain of slots that read one
// another's windows (a chain is as long as the run is), and 34 at 65,536 with a barrier behind every batch.
#include "wkv_internal.cuh"

#include <mutex>

namespace wkv {
namespace {

constexpr int kThreads = 512;
constexpr int kVecs = 8;              // 16-byte vectors per thread and batch: 64 KB per block in flight, two blocks per SM
constexpr int kPortableCluster = 8;   // cluster size that every device takes; sixteen has to be asked for
constexpr int kWideClusters = 14;     // clusters of sixteen that fit at once
constexpr int kMinVecs = 2;           // no more blocks per cluster than leave every thread this many vectors
constexpr int kResident = 264;        // blocks that fit at once in clusters of eight (33 clusters)
constexpr int kListMax = 12288;       // window indices of a unit that are kept in shared memory (48 KB)

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
    extern __shared__ int list[];
    const KShape &s = prm.s;
    pdl_trigger();
    const int cs = prm.cluster, unit = blockIdx.x / cs, rank = blockIdx.x - unit * cs, tensor = blockIdx.y;
    // The cluster's first batch into L2 while the kernel in front still runs: index, row and store follow one another
    // here, and the first two are most of the time of a layer that is one batch.  Four layers of 8 heads x 16,384 keys, 12 %,
    // recorded and replayed, with / without, us: one set of buffers, whose rows lie in L2, 27.0 / 27.4; sixteen sets in turn,
    // 514 MB of retained rows, 27.0 / 29.1 (32,768 keys: 42.5 / 44.0 and 42.5 / 44.9).  A call with no kernel in front of it
    // gains nothing.
    {
        const int slots = (cs * kThreads * kVecs / prm.vec_per_row + s.omega - 1) / s.omega;
        const int warp = rank * (kThreads / 32) + (threadIdx.x >> 5);
        for (int slot = warp; slot < min(slots, s.k_max); slot += cs * (kThreads / 32))
            fetch_window(s, static_cast<const char *>(prm.tab.ptr[tensor]), prm.elem_bytes, unit,
                         __ldcg(prm.window_idx + (size_t)unit * s.k_max + slot), threadIdx.x & 31, 32);
    }
    pdl_wait();
    const int b = unit / s.hkv, h = unit % s.hkv;
    // the unit's window indices: every look-up in memory would be a trip of its own, ahead of the row's
    const int *idx = prm.window_idx + (size_t)unit * s.k_max;
    if (s.k_max <= kListMax) {
        for (int i = threadIdx.x; i < s.k_max; i += kThreads) list[i] = idx[i];
        idx = list;
    }
    const SeqInfo si = seq_info(s, b);
    const int n = si.n;
    const int n_r = n > s.alpha ? n - s.alpha : 0;
    const int kw = num_windows(n, s.alpha, s.omega);
    const int k = num_selected_capped(n, s.alpha, s.omega, si.budget, s.k_max);
    __syncthreads();
    int review_rows = k * s.omega;
    if (k > 0 && idx[k - 1] == kw - 1) review_rows -= kw * s.omega - n_r;
    if (review_rows > n_r) review_rows = n_r;      // a list of all windows whose last entry is not the last window
    const int kept = review_rows + (n - n_r);
    if (kept <= 0) return;

    const int vpr = prm.vec_per_row;
    const long long row_vecs = s.st * prm.elem_bytes / 16;
    int4 *base = reinterpret_cast<int4 *>(static_cast<char *>(prm.tab.ptr[tensor]) +
                                          (si.off * s.st + b * s.sb + h * s.sh) * (long long)prm.elem_bytes);
    auto over = [](int x, int by, int shift) { return shift >= 0 ? x >> shift : x / by; };
    // A batch is a stretch of the output rows' vectors, from vector `col` of row `row` on.  (Rows are compared as
    // unsigned numbers: one that a step has taken past 2^31 lies behind all.)
    struct Place {
        int row, col;
    };
    auto advance = [&](Place p, int vecs) {
        const int x = p.col + vecs, rows = over(x, vpr, prm.vec_shift);
        return Place{p.row + rows, x - rows * vpr};
    };
    auto inside = [&](int row) { return (unsigned)row < (unsigned)kept; };
    // the row that output row r < kept takes, or -1 when it takes none: an entry that is no window of this sequence, or
    // that lies before its own slot (a list that is not an ascending selection), is skipped and the row stays as it is
    auto source_of = [&](int r) {
        if (r >= review_rows) return n_r + (r - review_rows);
        const int slot = over(r, s.omega, prm.omega_shift), wi = idx[slot];
        const int src = wi < slot || wi >= kw ? -1 : (wi - slot) * s.omega + r;
        return src < n_r ? src : -1;
    };
    int4 val[kVecs];
    unsigned moves;           // bit u: vector u of the thread has somewhere to go
    auto read = [&](Place p) {
        moves = 0u;
#pragma unroll
        for (int u = 0; u < kVecs; ++u) {
            const Place at = advance(p, (int)threadIdx.x + (u * cs + rank) * kThreads);
            if (!inside(at.row)) continue;
            const int src = source_of(at.row);
            if (src >= 0 && src != at.row) {
                val[u] = base[(long long)src * row_vecs + at.col];
                moves |= 1u << u;
            }
        }
    };
    auto write = [&](Place p) {
#pragma unroll
        for (int u = 0; u < kVecs; ++u)
            if (moves >> u & 1u) {
                const Place at = advance(p, (int)threadIdx.x + (u * cs + rank) * kThreads);
                base[(long long)at.row * row_vecs + at.col] = val[u];
            }
    };
    const int batch = cs * kThreads * kVecs;
    for (Place p = {0, 0}; inside(p.row);) {
        // here the cluster has read everything before p
        const int free_end = source_of(p.row);
        Place next = advance(p, batch);
        if (free_end >= kept || next.row < free_end) {
            for (;;) {
                read(p);
                write(p);
                p = next;
                if (!inside(p.row)) return;
                next = advance(p, batch);
                if (free_end < kept && next.row >= free_end) break;
            }
            cluster_barrier();
        } else {
            read(p);
            cluster_barrier();
            write(p);
            p = next;
        }
    }
}

// clusters of sixteen: asked for once per device (a property of kernel and device); false where they are refused
bool allow_wide_clusters()
{
    static std::mutex mu;
    static signed char state[kMaxDevices] = {};      // 0: not asked yet, 1: allowed, -1: refused
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        (void)cudaGetLastError();
        return false;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (state[dev] == 0) {
        const bool ok = cudaFuncSetAttribute(reinterpret_cast<const void *>(compact_inplace_kernel),
                                             cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
        if (!ok) (void)cudaGetLastError();
        state[dev] = ok ? 1 : -1;
    }
    return state[dev] > 0;
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
    // Blocks per (unit, tensor): a power of two, as many as are resident at once, unless the rows are too few to occupy
    // them.  Sixteen where that leaves all clusters resident (the portable eight left three quarters of the SMs idle
    // for a layer of 2 heads: 65,536 keys 14.1 us, with sixteen 9.7 us; 8 heads are sixteen clusters, of which fourteen
    // fit: 11.6 us with eight blocks each and 12.7 us with sixteen at 32,768 keys).
    const int pairs = ks.batch * ks.hkv * n_tensors;
    const long long vecs = ((long long)ks.k_max * ks.omega + ks.alpha) * prm.vec_per_row;
    int cs = 1;
    while (cs < kPortableCluster && pairs * cs * 2 <= kResident && (long long)cs * kThreads * kMinVecs < vecs) cs *= 2;
    if (cs == kPortableCluster && pairs <= kWideClusters && (long long)cs * kThreads * kMinVecs < vecs && allow_wide_clusters()) cs *= 2;
    prm.cluster = cs;
    const cudaError_t err = launch_pdl(compact_inplace_kernel, dim3(ks.batch * ks.hkv * cs, n_tensors), kThreads,
                                       ks.k_max <= kListMax ? ks.k_max * sizeof(int) : 0, stream, cs, prm);
    if (err != cudaSuccess) return err;
    count_launches(1);
    return cudaSuccess;
}

}  // namespace wkv
