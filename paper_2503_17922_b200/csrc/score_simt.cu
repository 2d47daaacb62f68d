// CUDA-core (FFMA) score kernels: Eq. 1-4 for fp32 inputs and for shapes the
// tensor-core kernels do not cover.  One kernel per call where its blocks are resident together (score_fused_simt), else two:
//   stats : per row of the unit, partial (max, sum exp2) over a chunk of keys
//           (Eq. 1's normaliser, causal mask applied)
//   score : logits again, p = exp2(x - lse2), sum over the rows (Eq. 2), then the
//           Top-p window pooling of Eq. 3-4 and, when asked, the selection by the
//           block that finishes a unit last
// Summation orders are fixed, so results are bit-identical from run to run.
//
// These problems are small (a few thousand keys), so what bounds them is the length of the chain from
// launch to result and how many SMs take part: a block takes as little as one tile of 64 keys, the eight
// blocks of a 512-key statistics chunk form a cluster and combine their rows through distributed shared
// memory, and the score kernel is launched as a programmatic dependent that computes its logits while the
// statistics kernel is still running.  The row tile follows R (16, 32 or 64 rows), so few rows cost no
// padding.
// 2 heads x 1,024 keys, 16 rows, d = 64: one block per 512 keys took 31 + 25 us for the two kernels (whole
// group 84 us); see simt_tiles_per_block for the sizes where a block takes more tiles.
#include "score_math.cuh"
#include "topk_block.cuh"
#include "wkv_internal.cuh"

#include <mutex>

#include <math.h>

namespace wkv {
namespace {

constexpr int kThreads = 256;
constexpr int kKT = 64;       // keys per logit tile
constexpr int kKPad = kKT + 4;
constexpr int kChunkTiles = kStatChunk / kKT;

__device__ inline float to_float(float x) { return x; }
__device__ inline float to_float(__nv_bfloat16 x) { return __bfloat162float(x); }

template <typename T>
struct Vec;  // 16-byte vector of T
template <>
struct Vec<float> {
    static constexpr int N = 4;
    float v[4];
};
template <>
struct Vec<__nv_bfloat16> {
    static constexpr int N = 8;
    __nv_bfloat16 v[8];
};

template <typename T>
__device__ inline Vec<T> load_vec(const T *p)
{
    Vec<T> r;
    *reinterpret_cast<int4 *>(&r) = *reinterpret_cast<const int4 *>(p);
    return r;
}

// Q of the unit, transposed into shared memory: qs[c * r_tile + r]; rows >= R are zero.  Lanes take
// consecutive rows, so that the transposed stores hit different banks; a thread keeps its row for all of the
// row's vectors, so the index arithmetic is done once per row.  last[r]: the last key row r may attend to.
template <typename T, int RB>
__device__ void load_q_transposed(const KShape &s, const T *q_unit, float *qs, int *last, int n_r, int r_tile)
{
    constexpr int VN = Vec<T>::N;
    const int vec_per_row = s.d / VN;
    for (int r = threadIdx.x % RB; r < r_tile; r += RB) {
        const int g = r / s.alpha, i = r - g * s.alpha;
        const T *row = q_unit + g * s.qsh + i * s.qst;
        if (last && threadIdx.x < RB) last[r] = r < s.R ? n_r + i : -1;
#pragma unroll 4
        for (int cv = threadIdx.x / RB; cv < vec_per_row; cv += kThreads / RB) {
            Vec<T> v;
            if (r < s.R) {
                v = load_vec(row + cv * VN);
            } else {
#pragma unroll
                for (int e = 0; e < VN; ++e) v.v[e] = T(0.f);
            }
#pragma unroll
            for (int e = 0; e < VN; ++e) qs[(cv * VN + e) * r_tile + r] = to_float(v.v[e]);
        }
    }
}

// kKT keys starting at j0, transposed: ks[c * kKPad + jj]; keys >= n_valid are zero.
template <typename T>
__device__ void load_k_transposed(const KShape &s, const T *k_unit, float *ks, int j0, int n_valid)
{
    constexpr int VN = Vec<T>::N;
    const int vec_per_row = s.d / VN;
    const int jj = threadIdx.x % kKT;
    const T *row = k_unit + (long long)(j0 + jj) * s.st;
#pragma unroll 4
    for (int cv = threadIdx.x / kKT; cv < vec_per_row; cv += kThreads / kKT) {
        Vec<T> v;
        if (j0 + jj < n_valid) {
            v = load_vec(row + cv * VN);
        } else {
#pragma unroll
            for (int e = 0; e < VN; ++e) v.v[e] = T(0.f);
        }
#pragma unroll
        for (int e = 0; e < VN; ++e) ks[(cv * VN + e) * kKPad + jj] = to_float(v.v[e]);
    }
}

// How the threads share a tile of RB rows x kKT keys: 4 rows x KPT keys each.
template <int RB>
struct TileMap {
    static constexpr int KPT = RB / 16;            // 4, 2, 1
    static constexpr int TX = kKT / KPT;           // threads along the keys: 16, 32, 64
    static_assert(RB == 16 || RB == 32 || RB == 64, "row tile");
    static_assert(kThreads / TX * 4 == RB, "threads do not cover the tile");
};

// raw dot products of rows r0 + ty*4 .. +3 with keys tx*KPT .. +KPT-1
template <int RB>
__device__ inline void logits_tile(const float *qs, const float *ks, int d, int r_pad, int r0, int ty, int tx,
                                   float (&acc)[4][TileMap<RB>::KPT])
{
    constexpr int KPT = TileMap<RB>::KPT;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < KPT; ++b) acc[a][b] = 0.f;
    const float *qp = qs + r0 + ty * 4;
    const float *kp = ks + tx * KPT;
#pragma unroll 8
    for (int c = 0; c < d; ++c) {
        const float4 qv = *reinterpret_cast<const float4 *>(qp + c * r_pad);
        const float qa[4] = {qv.x, qv.y, qv.z, qv.w};
        float ka[KPT];
        if constexpr (KPT == 4) {
            const float4 kv = *reinterpret_cast<const float4 *>(kp + c * kKPad);
            ka[0] = kv.x, ka[1] = kv.y, ka[2] = kv.z, ka[3] = kv.w;
        } else if constexpr (KPT == 2) {
            const float2 kv = *reinterpret_cast<const float2 *>(kp + c * kKPad);
            ka[0] = kv.x, ka[1] = kv.y;
        } else {
            ka[0] = kp[c * kKPad];
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < KPT; ++b) acc[a][b] = fmaf(qa[a], ka[b], acc[a][b]);
    }
}

// (max, sum) pairs of exponentials, to base 2: the pair of the union
__device__ inline void merge_stats(float &m, float &l, float m2, float l2)
{
    const float mn = fmaxf(m, m2);
    const float safe = mn == -INFINITY ? 0.f : mn;
    l = l * exp2f(m - safe) + l2 * exp2f(m2 - safe);
    m = mn;
}

__device__ __forceinline__ float2 ld_cluster(const float2 *p, int rank)
{
    uint32_t addr;
    float2 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}

// Grid: x = statistics chunk x blocks per chunk (the blocks of a chunk are one cluster), y = unit.
template <typename T, int RB>
__global__ void __launch_bounds__(kThreads)
score_stats_simt(const __grid_constant__ KShape s, const T *__restrict__ q, const T *__restrict__ k,
                 float2 *__restrict__ stats, int n_chunks, int r_pad, int r_tile, int tiles_per_block)
{
    constexpr int KPT = TileMap<RB>::KPT, TX = TileMap<RB>::TX;
    extern __shared__ __align__(16) float smem[];
    float *qs = smem;                                                   // [d][r_tile]
    float *ks = qs + s.d * r_tile;                                      // [d][kKPad]
    float2 *rows = reinterpret_cast<float2 *>(ks + s.d * kKPad);        // [r_pad] this block's (max, sum) ...
    float2 *half = rows + (tiles_per_block < kChunkTiles ? r_pad : 0);  // ... and, 16-row tiles: the second warps'
    int *last = reinterpret_cast<int *>(half + (RB == 16 ? r_pad : 0)); // [r_tile] last key of each row

    pdl_wait();
    pdl_trigger();      // the score kernel may read Q and K from here on: what wrote them has completed
    const int unit = blockIdx.y, cs = kChunkTiles / tiles_per_block;
    const int chunk = blockIdx.x / cs, rank = blockIdx.x - chunk * cs;
    const int b = unit / s.hkv, h = unit % s.hkv;
    const SeqInfo si = seq_info(s, b);
    const int n = si.n, n_r = n - s.alpha;
    const int j_begin = chunk * kStatChunk + rank * tiles_per_block * kKT;
    const int j_end = min(n, j_begin + tiles_per_block * kKT);
    const bool idle = n_r <= 0 || j_begin >= n;
    float2 *out = stats + ((size_t)unit * n_chunks + chunk) * r_pad;
    if (cs == 1) rows = out;      // nothing to combine: the rows are kept where they go
    for (int r = threadIdx.x; r < r_pad; r += kThreads) rows[r] = make_float2(-INFINITY, 0.f);
    if (!idle) {
        load_q_transposed<T, RB>(s, q + b * s.qsb + (long long)h * s.G * s.qsh, qs, last, n_r, r_tile);
        const T *k_unit = k + (si.off * s.st + b * s.sb + h * s.sh);
        const int ty = threadIdx.x / TX, tx = threadIdx.x % TX;
        for (int j0 = j_begin; j0 < j_end; j0 += kKT) {
            __syncthreads();
            load_k_transposed(s, k_unit, ks, j0, n);
            __syncthreads();
            for (int r0 = 0; r0 < r_tile; r0 += RB) {
                float acc[4][KPT];
                logits_tile<RB>(qs, ks, s.d, r_tile, r0, ty, tx, acc);
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const int r = r0 + ty * 4 + a;
                    const int jl = last[r] - j0 - tx * KPT;      // of this thread's keys, those up to jl count
                    float x[KPT], m = -INFINITY;
#pragma unroll
                    for (int c = 0; c < KPT; ++c) {
                        x[c] = c <= jl ? acc[a][c] * s.scale_log2 : -INFINITY;
                        m = fmaxf(m, x[c]);
                    }
#pragma unroll
                    for (int o = 1; o < (TX < 32 ? TX : 32); o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                    const float safe = m == -INFINITY ? 0.f : m;
                    float l = 0.f;
#pragma unroll
                    for (int c = 0; c < KPT; ++c) l += exp2f(x[c] - safe);
#pragma unroll
                    for (int o = 1; o < (TX < 32 ? TX : 32); o <<= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
                    // one thread per row adds the tile to the block's running pair
                    if (TX <= 32) {
                        if (tx == 0) {
                            float2 p = rows[r];
                            merge_stats(p.x, p.y, m, l);
                            rows[r] = p;
                        }
                    } else if (tx % 32 == 0) {
                        float2 *mine = tx == 0 ? rows : half;
                        float2 p = j0 == j_begin ? make_float2(-INFINITY, 0.f) : mine[r];
                        merge_stats(p.x, p.y, m, l);
                        mine[r] = p;
                    }
                }
            }
        }
        if (TX > 32) {
            __syncthreads();
            for (int r = threadIdx.x; r < r_tile; r += kThreads) {
                float2 p = rows[r];
                merge_stats(p.x, p.y, half[r].x, half[r].y);
                rows[r] = p;
            }
        }
    }
    if (cs == 1) return;
    // the chunk's rows: the blocks of the cluster share them out, each combines its rows over all blocks in order
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    for (int r = rank * kThreads + threadIdx.x; r < r_pad; r += cs * kThreads) {
        float m = -INFINITY, l = 0.f;
        for (int c = 0; c < cs; ++c) {
            const float2 p = ld_cluster(rows + r, c);
            merge_stats(m, l, p.x, p.y);
        }
        out[r] = make_float2(m, l);
    }
    // no block leaves while another may still read its rows
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Eq. 4 for one window: the sorting network where there is one for its length, else the serial form
__device__ inline float pool_window(const float *w, int omega, int size, int p)
{
    switch (omega) {
    case 4: return pool_window_sorted<4>(w, size, p, threadIdx.x & 31);
    case 8: return pool_window_sorted<8>(w, size, p, threadIdx.x & 31);
    case 16: return pool_window_sorted<16>(w, size, p, threadIdx.x & 31);
    case 32: return pool_window_sorted<32>(w, size, p, threadIdx.x & 31);
    default: return pool_top_p(w, size, p);
    }
}

// ---------------------------------------------------------------------------------------------
// one launch for statistics, scores and selection
// ---------------------------------------------------------------------------------------------
struct FusedArgs {
    KShape s;
    StatEntry *stats;       // [units][n_chunks][r_pad]: published statistics of 512 keys
    StatEntry *entries;     // [units][kw_max]: published window scores, for the block that selects
    float *window_scores, *token_scores;
    int *window_idx, *kept_len;     // null: no selection
    int *status;
    LaunchCount *count;
    unsigned salt;
    int n_chunks, r_pad, r_tile;
};

// Where all blocks are resident at once (cooperative launch) the logits of a block's one tile stay in its registers
// while the unit's statistics are put together: the tiles of Q and K are transposed and multiplied once instead of twice,
// and two kernel boundaries go.  The blocks of 512 keys are a cluster and combine their rows through distributed shared
// memory; chunks and window scores are handed over as self-validating words; the block of the unit's last review
// keys selects.  Windows must not straddle tiles.  Bounded, like the other kernels that wait: status bit 0.
// Grid: x = tiles rounded up to whole clusters, y = unit.
template <typename T, int RB, int PASSES>
__global__ void __launch_bounds__(kThreads, 4)
score_fused_simt(const __grid_constant__ FusedArgs a, const T *__restrict__ q, const T *__restrict__ k)
{
    constexpr int KPT = TileMap<RB>::KPT, TX = TileMap<RB>::TX, TY = kThreads / TX;
    constexpr int kSharers = TX < 32 ? TX : 32;              // neighbouring lanes that share a row
    extern __shared__ __align__(16) float smem[];
    const KShape &s = a.s;
    float *qs = smem;                                        // [d][r_tile]
    float *ks = qs + s.d * a.r_tile;                         // [d][kKPad]
    float2 *rows = reinterpret_cast<float2 *>(ks + s.d * kKPad);   // [2][r_pad] this block's (max, sum) per row
    float *lse2 = reinterpret_cast<float *>(rows + 2 * a.r_pad);   // [r_pad]
    float *part = lse2 + a.r_pad;                            // [TY][kKT]
    float *t_tile = part + TY * kKT;                         // [kKT]
    int *last = reinterpret_cast<int *>(t_tile + kKT);       // [r_tile]
    TopkSmem &topk_sm = *reinterpret_cast<TopkSmem *>(smem); // the selection comes when all of these are done with
    __shared__ int abort_s;
    __shared__ unsigned long long tag_s;

    const int unit = blockIdx.y, chunk = blockIdx.x / kChunkTiles, rank = blockIdx.x - chunk * kChunkTiles;
    const int b = unit / s.hkv, h = unit - b * s.hkv;
    const SeqInfo si = seq_info(s, b);
    const int n = si.n, n_r = n - s.alpha, j0 = blockIdx.x * kKT;
    const int ty = threadIdx.x / TX, tx = threadIdx.x % TX;
    unsigned long long launches = 0;
    if (threadIdx.x == 0) launches = launches_so_far(a.count);
    const bool idle = n_r <= 0 || j0 >= n;
    float acc[PASSES][4][KPT];
    if (!idle) {
        load_q_transposed<T, RB>(s, q + b * s.qsb + (long long)h * s.G * s.qsh, qs, last, n_r, a.r_tile);
        load_k_transposed(s, k + (si.off * s.st + b * s.sb + h * s.sh), ks, j0, n);
    }
    if (threadIdx.x == 0) {
        abort_s = 0;
        tag_s = launch_tag(launches, a.salt);
    }
    for (int r = threadIdx.x; r < 2 * a.r_pad; r += kThreads) rows[r] = make_float2(-INFINITY, 0.f);
    __syncthreads();
    if (threadIdx.x == 32) count_launch(a.count, launch_of(tag_s), gridDim.x * gridDim.y);
    if (!idle) {
#pragma unroll
        for (int p = 0; p < PASSES; ++p) {
            logits_tile<RB>(qs, ks, s.d, a.r_tile, p * RB, ty, tx, acc[p]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = p * RB + ty * 4 + i, jl = last[r] - j0 - tx * KPT;      // of this thread's keys, those up to jl count
                float m = -INFINITY;
#pragma unroll
                for (int c = 0; c < KPT; ++c) {
                    acc[p][i][c] *= s.scale_log2;
                    if (c <= jl) m = fmaxf(m, acc[p][i][c]);
                }
#pragma unroll
                for (int o = 1; o < kSharers; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                const float safe = m == -INFINITY ? 0.f : m;
                float l = 0.f;
#pragma unroll
                for (int c = 0; c < KPT; ++c)
                    if (c <= jl) l += exp2f(acc[p][i][c] - safe);
#pragma unroll
                for (int o = 1; o < kSharers; o <<= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
                if (tx % kSharers == 0) rows[(tx / kSharers) * a.r_pad + r] = make_float2(m, l);
            }
        }
    }
    // the chunk's rows: each block of the cluster combines a share of them over all blocks, a lane per block
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    const int share = a.r_pad / kChunkTiles;
    if ((int)threadIdx.x < share * kChunkTiles) {            // whole warps: r_pad is a multiple of 64
        const int r = rank * share + threadIdx.x / kChunkTiles, from = threadIdx.x % kChunkTiles;
        float2 v = ld_cluster(rows + r, from);
        if (TX > 32) {
            const float2 second = ld_cluster(rows + a.r_pad + r, from);
            merge_stats(v.x, v.y, second.x, second.y);
        }
#pragma unroll
        for (int o = 1; o < kChunkTiles; o <<= 1)
            merge_stats(v.x, v.y, __shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
        if (from == 0 && r < s.R && chunk * kStatChunk < n)
            publish_entry(a.stats + ((size_t)unit * a.n_chunks + chunk) * a.r_pad + r,
                          (unsigned long long)__float_as_uint(v.x) | (unsigned long long)__float_as_uint(v.y) << 32, tag_s);
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");      // this block has read its peers' rows

    const int j_end = min(n_r, j0 + kKT);
    if (j0 < n_r) {
        // log2 of every row's normaliser from the unit's chunks: neighbouring threads share a row
        const int used = (n + kStatChunk - 1) / kStatChunk;
        const int tpr = a.r_pad <= 64 ? 4 : 2;
        {
            const int r = threadIdx.x / tpr, of = threadIdx.x - r * tpr;
            float M = -INFINITY, L = 0.f;
            if (r < s.R) {
                const StatEntry *st = a.stats + (size_t)unit * a.n_chunks * a.r_pad + r;
                for (int c0 = of; c0 < used; c0 += 4 * tpr) {
                    unsigned wanted = 0u;
#pragma unroll
                    for (int u = 0; u < 4; ++u) wanted |= (c0 + u * tpr < used ? 1u : 0u) << u;
                    StatEntry e[4];
                    wait_entries<4>(st + (size_t)c0 * a.r_pad, (size_t)tpr * a.r_pad, wanted, tag_s, e, &abort_s);
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (wanted >> u & 1u)
                            merge_stats(M, L, __uint_as_float((unsigned)e[u].value), __uint_as_float((unsigned)(e[u].value >> 32)));
                }
            }
            __syncwarp();
            for (int o = 1; o < tpr; o <<= 1) {
                const float m2 = __shfl_xor_sync(0xffffffffu, M, o), l2 = __shfl_xor_sync(0xffffffffu, L, o);
                merge_stats(M, L, m2, l2);
            }
            if (of == 0 && r < a.r_pad) lse2[r] = r < s.R && L > 0.f ? M + log2f(L) : INFINITY;
        }
        __syncthreads();
        float col[KPT];
#pragma unroll
        for (int c = 0; c < KPT; ++c) col[c] = 0.f;
#pragma unroll
        for (int p = 0; p < PASSES; ++p)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float ls = lse2[p * RB + ty * 4 + i];
#pragma unroll
                for (int c = 0; c < KPT; ++c) col[c] += exp2f(acc[p][i][c] - ls);
            }
#pragma unroll
        for (int c = 0; c < KPT; ++c) part[ty * kKT + tx * KPT + c] = col[c];
        __syncthreads();
        if (threadIdx.x < kKT) {
            float t = 0.f;
#pragma unroll
            for (int y = 0; y < TY; ++y) t += part[y * kKT + threadIdx.x];
            t_tile[threadIdx.x] = t;
            if (a.token_scores && j0 + (int)threadIdx.x < n_r) a.token_scores[(size_t)unit * s.nr_max + j0 + threadIdx.x] = t;
        }
        __syncthreads();
        // Eq. 3-4: the tile's windows
        const int n_win = (j_end - j0 + s.omega - 1) / s.omega;
        if ((int)threadIdx.x < n_win) {
            const int lo = threadIdx.x * s.omega;
            const float r = pool_window(t_tile + lo, s.omega, min(s.omega, j_end - j0 - lo), s.p);
            const size_t w = (size_t)unit * s.kw_max + j0 / s.omega + threadIdx.x;
            a.window_scores[w] = r;
            if (a.window_idx) publish_entry(a.entries + w, __float_as_uint(r), tag_s);
        }
    }
    // no block leaves, or overwrites its rows, while another may still read them
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (a.window_idx) {
        if (n_r <= 0) {
            // a unit without review context still gets its (empty) selection
            if (blockIdx.x == 0) {
                for (int x = threadIdx.x; x < s.k_max; x += kThreads) a.window_idx[(size_t)unit * s.k_max + x] = -1;
                if (threadIdx.x == 0) a.kept_len[unit] = min(n, s.alpha);
            }
        } else if (j0 < n_r && j_end == n_r) {
            __syncthreads();
            select_topk_block<kThreads>((int)threadIdx.x, topk_sm,
                                        PublishedScores<4>{a.entries + (size_t)unit * s.kw_max, tag_s, &abort_s, topk_hint(s.R, n)},
                                        num_windows(n, s.alpha, s.omega), num_selected_capped(n, s.alpha, s.omega, si.budget, s.k_max),
                                        s.k_max, a.window_idx + (size_t)unit * s.k_max, a.kept_len + unit, n, s.alpha, s.omega);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && abort_s) atomicOr(a.status, kStatusWaitExpired);
}

// the selection that the score kernel's last block of a unit runs (window_idx null: none)
struct SimtSelect {
    int *window_idx, *kept_len, *status, *sync;
    bool release_early;     // the gather behind it waits before it looks at the indices
};

template <typename T, int RB>
// (five blocks per SM: the sorting network of long windows would take it beyond 48 registers, which costs the beginning
// of the kernel its place beside the statistics kernel's blocks: 44.6 us instead of 42.1 us for 4 heads x 6,000 keys)
__global__ void __launch_bounds__(kThreads, 5)
score_pool_simt(const __grid_constant__ KShape s, const T *__restrict__ q, const T *__restrict__ k, const float2 *stats,
                const float *lse_obs, float *window_scores, float *__restrict__ token_scores, int n_chunks,
                int r_pad, int r_tile, int chunk_keys, const __grid_constant__ SimtSelect sel)
{
    constexpr int KPT = TileMap<RB>::KPT, TX = TileMap<RB>::TX, TY = kThreads / TX;
    extern __shared__ __align__(16) float smem[];
    float *qs = smem;                          // [d][r_tile]
    float *ks = qs + s.d * r_tile;             // [d][kKPad]
    float *lse2 = ks + s.d * kKPad;            // [r_pad]
    float *part = lse2 + r_pad;                // [TY][kKT]
    float *t_chunk = part + TY * kKT;          // [chunk_keys rounded up to kKT]
    TopkSmem &topk_sm = *reinterpret_cast<TopkSmem *>(smem);   // the selection comes when all of these are done with

    if (sel.release_early) pdl_trigger();
    // with given normalisers there is no statistics kernel in front that has waited for Q and K
    if (lse_obs) pdl_wait();
    const int unit = blockIdx.y;
    const int b = unit / s.hkv, h = unit % s.hkv;
    const SeqInfo si = seq_info(s, b);
    const int n = si.n, n_r = n - s.alpha;
    const int j_begin = blockIdx.x * chunk_keys;
    if (n_r <= 0 || j_begin >= n_r) {
        if (!lse_obs) pdl_wait();
        // a unit without review context still gets its (empty) selection
        if (sel.window_idx && n_r <= 0 && blockIdx.x == 0)
            select_topk_block<kThreads>((int)threadIdx.x, topk_sm, WrittenScores{window_scores, -1}, 0, 0, s.k_max, sel.window_idx + (size_t)unit * s.k_max,
                                        sel.kept_len + unit, n, s.alpha, s.omega);
        return;
    }
    const int j_end = min(n_r, j_begin + chunk_keys);
    const T *k_unit = k + (si.off * s.st + b * s.sb + h * s.sh);
    load_q_transposed<T, RB>(s, q + b * s.qsb + (long long)h * s.G * s.qsh, qs, nullptr, n_r, r_tile);

    const int ty = threadIdx.x / TX, tx = threadIdx.x % TX;
    for (int j0 = j_begin; j0 < j_end; j0 += kKT) {
        __syncthreads();
        load_k_transposed(s, k_unit, ks, j0, n_r);
        __syncthreads();
        float col[KPT];
#pragma unroll
        for (int c = 0; c < KPT; ++c) col[c] = 0.f;
        for (int r0 = 0; r0 < r_tile; r0 += RB) {
            float acc[4][KPT];
            logits_tile<RB>(qs, ks, s.d, r_tile, r0, ty, tx, acc);
            if (j0 == j_begin && r0 == 0) {
                // Only now are the statistics needed.  lse2 = log2 of the row normaliser: the threads of a row
                // (kThreads / r_pad of them, neighbours) merge every that-many-th chunk, then one another; or the
                // caller's value (natural log) in base 2
                if (!lse_obs) pdl_wait();
                const int tpr = r_pad <= 64 ? 4 : (r_pad <= 128 ? 2 : 1);
                const int used = (n + kStatChunk - 1) / kStatChunk;
                for (int rr = threadIdx.x; rr < r_pad * tpr; rr += kThreads) {
                    const int r = rr / tpr, part_of = rr - r * tpr;
                    float v = INFINITY;
                    if (lse_obs) {
                        const int g = r / s.alpha, i = r - g * s.alpha;
                        if (r < s.R) v = lse_obs[((size_t)b * s.hq + (size_t)h * s.G + g) * s.alpha + i] * 1.4426950408889634f;
                    } else {
                        const float2 *st = stats + (size_t)unit * n_chunks * r_pad + r;
                        float M = -INFINITY, L = 0.f;
                        for (int c0 = part_of; c0 < used; c0 += 4 * tpr) {
                            float2 p[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                p[u] = c0 + u * tpr < used ? __ldcg(st + (size_t)(c0 + u * tpr) * r_pad) : make_float2(-INFINITY, 0.f);
#pragma unroll
                            for (int u = 0; u < 4; ++u) merge_stats(M, L, p[u].x, p[u].y);
                        }
                        for (int o = 1; o < tpr; o <<= 1) {
                            const float m2 = __shfl_xor_sync(0xffffffffu, M, o), l2 = __shfl_xor_sync(0xffffffffu, L, o);
                            merge_stats(M, L, m2, l2);
                        }
                        if (r < s.R && L > 0.f) v = M + log2f(L);
                    }
                    if (part_of == 0) lse2[r] = v;
                }
                __syncthreads();
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const float ls = lse2[r0 + ty * 4 + a];
#pragma unroll
                for (int c = 0; c < KPT; ++c) col[c] += exp2f(fmaf(acc[a][c], s.scale_log2, -ls));
            }
        }
#pragma unroll
        for (int c = 0; c < KPT; ++c) part[ty * kKT + tx * KPT + c] = col[c];
        __syncthreads();
        if (threadIdx.x < kKT) {
            float t = 0.f;
#pragma unroll
            for (int y = 0; y < TY; ++y) t += part[y * kKT + threadIdx.x];
            const int j = j0 + threadIdx.x;
            t_chunk[j - j_begin] = t;
            if (token_scores && j < n_r) token_scores[(size_t)unit * s.nr_max + j] = t;
        }
    }
    __syncthreads();
    // Eq. 3-4: windows of this chunk (chunk_keys is a multiple of omega)
    const int w_begin = j_begin / s.omega;
    const int n_win = (j_end - j_begin + s.omega - 1) / s.omega;
    for (int lw = threadIdx.x; lw < n_win; lw += kThreads) {
        const int lo = lw * s.omega;
        window_scores[(size_t)unit * s.kw_max + w_begin + lw] =
            pool_window(t_chunk + lo, s.omega, min(s.omega, (j_end - j_begin) - lo), s.p);
    }
    if (!sel.window_idx) return;
    // The block that counts itself last on the unit's ticket word selects for the unit and clears the word.
    __syncthreads();
    if (threadIdx.x == 0) {
        const int used = (n_r + chunk_keys - 1) / chunk_keys;
        int *ticket = sel.sync + kSyncTickets + kSyncWordsPerUnit * unit;
        __threadfence();                 // publishes the window scores the whole block wrote
        const int before = atomicAdd(ticket, 1);
        if (before == used - 1) atomicExch(ticket, 0);
        if (before < 0 || before >= used) atomicOr(sel.status, kStatusWaitExpired);   // the workspace was not cleared
        __threadfence();
        topk_sm.remaining = before == used - 1;
    }
    __syncthreads();
    const bool selects = topk_sm.remaining != 0;
    __syncthreads();                     // the word is the selection's own from here on
    if (selects)
        select_topk_block<kThreads>((int)threadIdx.x, topk_sm, WrittenScores{window_scores + (size_t)unit * s.kw_max, topk_hint(s.R, n)}, num_windows(n, s.alpha, s.omega),
                                    num_selected_capped(n, s.alpha, s.omega, si.budget, s.k_max), s.k_max,
                                    sel.window_idx + (size_t)unit * s.k_max, sel.kept_len + unit, n, s.alpha, s.omega);
}

}  // namespace

// The opt-in to more than 48 KB of dynamic shared memory is a property of (kernel, device): it is
// raised once per device and kernel to the largest size asked for so far, not on every launch.
static cudaError_t allow_dynamic_smem(const void *fn, int dev, int slot, size_t bytes)
{
    static std::mutex mu;
    static size_t allowed[kMaxDevices][12] = {};
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (bytes <= allowed[dev][slot]) return cudaSuccess;
    const cudaError_t err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (err == cudaSuccess) allowed[dev][slot] = bytes;
    return err;
}

// Tiles of 64 keys per block: one while the blocks fit the GPU once or twice (latency), two and four when they fill it
// more often, since every block transposes the whole of Q first.  A wave is 740 blocks, five per SM (the score kernel's
// bound; at d = 128 shared memory leaves three).  Select call, fp32, R = 64, d = 64 / 128, us with 1, 2, 4, 8 tiles:
//     376 tiles   36  42  52  85   /   54  65  73 140       1,504 tiles   97  93 110 167  /  179 151 146 206
//   4,096 tiles  222 196 181 218   /  450 372 366 458      16,384 tiles  851 732 669 652  /  1709 1416 1269 1300
// R = 16, 32 and 128 lie alike.
constexpr int kBlocksPerWave = 740;
constexpr int kMaxBlockTiles = 4;
static int simt_tiles_per_block(const KShape &ks)
{
    const long long tiles = (long long)ks.batch * ks.hkv * ((ks.max_seqlen + kKT - 1) / kKT);
    if (ks.R > 1024) return kChunkTiles;     // the rows of a cluster's blocks would not fit shared memory beside Q
    int t = 1;
    while (t < kMaxBlockTiles && tiles / (2 * t) >= kBlocksPerWave) t *= 2;
    return t;
}

// keys per block of the score kernel: whole windows
static int simt_chunk_keys(const KShape &ks, int tiles_per_block)
{
    int per = tiles_per_block * kKT / ks.omega;
    if (per < 1) per = 1;
    return per * ks.omega;
}

static int simt_row_tile(const KShape &ks) { return ks.R <= 16 ? 16 : (ks.R <= 32 ? 32 : 64); }

static void simt_smem(const KShape &ks, int r_pad, size_t &stats_bytes, size_t &pool_bytes)
{
    const int rb = simt_row_tile(ks), r_tile = rb < 64 ? rb : r_pad;
    const int tpb = simt_tiles_per_block(ks), chunk_keys = simt_chunk_keys(ks, tpb);
    const size_t tiles = (size_t)ks.d * r_tile + (size_t)ks.d * kKPad;
    stats_bytes = sizeof(float) * (tiles + (tpb < kChunkTiles ? 2 * (size_t)r_pad : 0) + (rb == 16 ? 2 * (size_t)r_pad : 0) + (size_t)r_tile);
    pool_bytes = sizeof(float) * (tiles + (size_t)r_pad + (size_t)(rb / 4) * kKT + (size_t)((chunk_keys + kKT - 1) / kKT) * kKT);
    if (pool_bytes < sizeof(TopkSmem)) pool_bytes = sizeof(TopkSmem);
}

template <typename T, int RB>
static cudaError_t launch_simt_tile(const KShape &ks, int slot, const void *q, const void *k, float *window_scores,
                                    float *token_scores, float2 *stats, const Workspace &ws, cudaStream_t stream,
                                    const float *lse_obs, const SimtSelect &sel)
{
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    const int units = ks.batch * ks.hkv, r_pad = ws.r_pad, r_tile = RB < 64 ? RB : r_pad;
    const int tpb = simt_tiles_per_block(ks), chunk_keys = simt_chunk_keys(ks, tpb);
    size_t smem1, smem2;
    simt_smem(ks, r_pad, smem1, smem2);
    if (!lse_obs) {
        auto fn = score_stats_simt<T, RB>;
        err = allow_dynamic_smem(reinterpret_cast<const void *>(fn), dev, slot, smem1);
        if (err != cudaSuccess) return err;
        const int cs = kChunkTiles / tpb, chunks = (ks.max_seqlen + kStatChunk - 1) / kStatChunk;
        err = launch_pdl(fn, dim3(chunks * cs, units), kThreads, smem1, stream, cs, ks, (const T *)q, (const T *)k, stats,
                         ws.n_stat_chunks, r_pad, r_tile, tpb);
        if (err != cudaSuccess) return err;
    }
    auto fn = score_pool_simt<T, RB>;
    err = allow_dynamic_smem(reinterpret_cast<const void *>(fn), dev, slot + 1, smem2);
    if (err != cudaSuccess) return err;
    const int n_r_max = ks.max_seqlen - ks.alpha;
    err = launch_pdl(fn, dim3((n_r_max + chunk_keys - 1) / chunk_keys, units), kThreads, smem2, stream, 1, ks, (const T *)q,
                     (const T *)k, (const float2 *)stats, lse_obs, window_scores, token_scores, ws.n_stat_chunks, r_pad, r_tile,
                     chunk_keys, sel);
    if (err == cudaSuccess) count_launches(lse_obs ? 1 : 2);
    return err;
}

// Launches the fused kernel where its clusters are all resident at once, else leaves `taken` false: more blocks than that
// would wait for blocks that cannot start.  Wherever they fit it is the faster way; select call, fp32, us, two launches /
// one: 2 heads x 600 keys, 16 rows, d = 64 12.4 / 10.6; 8 heads x 4,000, 16 rows 24.1 / 17.0; 4 heads x 6,000, 64 rows
// 30.9 / 20.6 (d = 128: 48.2 / 30.8); 2 heads x 6,000, 128 rows 33.6 / 24.3 (d = 128: 49.8 / 34.9).
template <typename T, int RB, int PASSES>
static cudaError_t launch_fused_tile(const KShape &ks, const void *q, const void *k, float *window_scores, float *token_scores,
                                     void *workspace, const Workspace &ws, cudaStream_t stream, int *window_idx, int *kept_len,
                                     bool &taken)
{
    FusedArgs a;
    char *base = static_cast<char *>(workspace);
    a.s = ks;
    a.stats = reinterpret_cast<StatEntry *>(base + ws.stats_off);
    a.entries = reinterpret_cast<StatEntry *>(base + ws.entries_off);
    a.window_scores = window_scores;
    a.token_scores = token_scores;
    a.window_idx = window_idx;
    a.kept_len = kept_len;
    a.status = reinterpret_cast<int *>(base + ws.status_off);
    a.count = reinterpret_cast<LaunchCount *>(base + ws.count_off);
    a.salt = ws.salt;
    a.n_chunks = (ks.max_seqlen + kStatChunk - 1) / kStatChunk;
    a.r_pad = ws.r_pad;
    a.r_tile = RB * PASSES;
    size_t smem = sizeof(float) * ((size_t)ks.d * (a.r_tile + kKPad) + 5 * (size_t)a.r_pad + (RB / 4 + 1) * kKT + a.r_tile);
    if (smem < sizeof(TopkSmem)) smem = sizeof(TopkSmem);

    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    const auto fn = score_fused_simt<T, RB, PASSES>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.n_chunks * kChunkTiles, ks.batch * ks.hkv);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kChunkTiles;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeCooperative;
    attr[1].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    {
        // clusters that are resident at once: a property of device, kernel and shared-memory size, asked for once each.
        // None where a block is refused that much shared memory: with long rows the two kernels need 1.3 to 2.6 KB less
        // than this one (head dimension 288 with 65-128 rows: 225.25 and 227.75 KB of the 227 there are).
        static std::mutex mu;
        static size_t allowed[kMaxDevices] = {};
        static size_t asked[kMaxDevices][4] = {};
        static int resident[kMaxDevices][4] = {};
        if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> lock(mu);
        int slot = 0;
        while (slot < 4 && asked[dev][slot] != smem && asked[dev][slot] != 0) ++slot;
        int fits = slot < 4 ? resident[dev][slot] : 0;
        if (slot == 4 || asked[dev][slot] == 0) {
            if (smem > 48u * 1024u && smem > allowed[dev]) {
                err = cudaFuncSetAttribute(reinterpret_cast<const void *>(fn), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
                if (err == cudaSuccess) allowed[dev] = smem;
            }
            if (err == cudaSuccess) err = cudaOccupancyMaxActiveClusters(&fits, fn, &cfg);
            if (err != cudaSuccess) {
                (void)cudaGetLastError();      // too much shared memory, or a device without such clusters: the two kernels
                fits = 0;
            }
            if (slot < 4) {
                asked[dev][slot] = smem;
                resident[dev][slot] = fits;
            }
        }
        if (a.n_chunks * ks.batch * ks.hkv > fits) return cudaSuccess;
    }
    cfg.numAttrs = 2;
    err = cudaLaunchKernelEx(&cfg, fn, a, (const T *)q, (const T *)k);
    if (err == cudaErrorCooperativeLaunchTooLarge) {
        (void)cudaGetLastError();              // fewer SMs than the query answers for: the two kernels wait for nobody
        return cudaSuccess;
    }
    if (err != cudaSuccess) return err;
    taken = true;
    count_launches(1);
    return cudaSuccess;
}

template <typename T>
static cudaError_t launch_fused_type(const KShape &ks, const void *q, const void *k, float *window_scores, float *token_scores,
                                     void *workspace, const Workspace &ws, cudaStream_t stream, int *window_idx, int *kept_len,
                                     bool &taken)
{
    if (ks.R <= 16) return launch_fused_tile<T, 16, 1>(ks, q, k, window_scores, token_scores, workspace, ws, stream, window_idx, kept_len, taken);
    if (ks.R <= 32) return launch_fused_tile<T, 32, 1>(ks, q, k, window_scores, token_scores, workspace, ws, stream, window_idx, kept_len, taken);
    if (ks.R <= 64) return launch_fused_tile<T, 64, 1>(ks, q, k, window_scores, token_scores, workspace, ws, stream, window_idx, kept_len, taken);
    return launch_fused_tile<T, 64, 2>(ks, q, k, window_scores, token_scores, workspace, ws, stream, window_idx, kept_len, taken);
}

template <typename T>
static cudaError_t launch_simt_type(const KShape &ks, int slot, const void *q, const void *k, float *window_scores,
                                    float *token_scores, float2 *stats, const Workspace &ws, cudaStream_t stream,
                                    const float *lse_obs, const SimtSelect &sel)
{
    switch (simt_row_tile(ks)) {
    case 16: return launch_simt_tile<T, 16>(ks, slot, q, k, window_scores, token_scores, stats, ws, stream, lse_obs, sel);
    case 32: return launch_simt_tile<T, 32>(ks, slot + 2, q, k, window_scores, token_scores, stats, ws, stream, lse_obs, sel);
    default: return launch_simt_tile<T, 64>(ks, slot + 4, q, k, window_scores, token_scores, stats, ws, stream, lse_obs, sel);
    }
}

cudaError_t launch_score_simt(const KShape &ks, int dtype, const void *q, const void *k,
                              float *window_scores, float *token_scores,
                              void *workspace, const Workspace &ws, cudaStream_t stream, const float *lse_obs,
                              int *window_idx, int *kept_len, bool group)
{
    float2 *stats = reinterpret_cast<float2 *>(static_cast<char *>(workspace) + ws.stats_off);
    if (ks.max_seqlen <= ks.alpha) return window_idx ? launch_topk(ks, window_scores, window_idx, kept_len, stream) : cudaSuccess;
    if (!lse_obs && simt_fused_shape(ks)) {
        bool taken = false;
        const cudaError_t err = dtype == WKV_F32 ? launch_fused_type<float>(ks, q, k, window_scores, token_scores, workspace, ws,
                                                                            stream, window_idx, kept_len, taken)
                                                 : launch_fused_type<__nv_bfloat16>(ks, q, k, window_scores, token_scores, workspace,
                                                                                    ws, stream, window_idx, kept_len, taken);
        if (err != cudaSuccess || taken) return err;
    }
    // The selection inside the score kernel where a block keeps the unit's window scores in registers (eight per
    // thread): one launch less.  Longer lists go to the kernel with four times the threads.
    const bool inside = window_idx && ks.kw_max <= 8 * kThreads;
    SimtSelect sel = {};
    sel.release_early = group;
    if (inside) {
        sel.window_idx = window_idx;
        sel.kept_len = kept_len;
        sel.status = reinterpret_cast<int *>(static_cast<char *>(workspace) + ws.status_off);
        sel.sync = reinterpret_cast<int *>(static_cast<char *>(workspace) + ws.sync_off);
    }
    const cudaError_t err =
        dtype == WKV_F32
            ? launch_simt_type<float>(ks, 0, q, k, window_scores, token_scores, stats, ws, stream, lse_obs, sel)
            : launch_simt_type<__nv_bfloat16>(ks, 6, q, k, window_scores, token_scores, stats, ws, stream, lse_obs, sel);
    if (err != cudaSuccess || !window_idx || inside) return err;
    return launch_topk(ks, window_scores, window_idx, kept_len, stream);
}

// shared-memory need of the CUDA-core kernels, for the host-side support check
size_t score_simt_smem_bytes(const KShape &ks, int r_pad)
{
    size_t a, b;
    simt_smem(ks, r_pad, a, b);
    return a > b ? a : b;
}

}  // namespace wkv
