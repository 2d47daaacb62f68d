// Tensor-core score kernel (tcgen05 + tensor memory + TMA) for bf16 inputs: Eq. 1-4 of the leader
// and, when asked, the budgeted selection, in ONE launch.
//
// The token score of Eq. 2, t_j = sum_i exp(s_ij) / Z_i, needs every row's softmax normaliser
// Z_i (a reduction over all keys) before any column sum can be finished, so the keys are swept
// twice; a block starts normalising a unit's keys once all chunks of that unit have delivered their
// sweep-1 statistics (published words that say themselves whether they are there, no grid-wide barrier):
//   sweep 1  D[rows, keys] = Q K^T per 128-key tile with the observation rows on the tensor-memory
//            lanes: one thread owns one row and keeps its running (max, sum exp2) without any
//            cross-thread traffic (Eq. 1's normaliser, causal mask on the tiles that touch the
//            observation window).  K comes from HBM.
//   sweep 2  D[keys, rows] = K Q^T with the keys on the lanes: one thread owns one key and sums
//            exp2(x_ij - lse2_i) over the rows (Eq. 2); the block then pools its windows (Eq. 3-4).
//            The block re-reads the keys it streamed in sweep 1, as far as they fit from L2.
//   select   the block of a unit's last chunk waits for the unit's other blocks and runs the selection.
// Units are taken in waves of as many as the blocks can share (tc_plan).  A work item is (unit, chunk of <= 37 key
// tiles); the persistent blocks (at most one per SM) take the items of a wave round-robin.
//
// Warp roles: warp 0 issues the TMA tile loads (4-stage ring), warp 1 issues the MMAs (each as a whole
// converged warp, one elected lane acting) into four
// accumulator buffers of 128 columns in tensor memory, and four compute groups of four warps (one
// warp per 32-lane quarter of tensor memory) take the accumulators round-robin, each with its own
// buffer, 32 columns at a time.  With more than 128 observation rows (up to 256) every key tile
// gives two accumulators, one per 128-row block of Q, which go through the same buffers and groups; the four warps that share an SM sub-partition cover each other's load latency.  The
// contraction is the only tensor-core work; exponentials, sums and pooling are fp32 on the CUDA
// cores in a fixed order, so results are bit-identical from run to run.
//
// Every wait is bounded (mbarriers and the wait for a unit's statistics): on expiry the block sets bit 0 of the
// status word, drains its own TMA loads, frees its tensor memory and returns.
//
// Where the whole problem is one wave (ONE) the launch is a programmatic dependent and guarantees nothing about which
// blocks run together: a block looks for what others publish for a while and then does without them
// (stand_in, late_selection), with the same results.  With several waves the launch is cooperative.
#include "tc_common.cuh"
#include "score_math.cuh"
#include "topk_block.cuh"
#include "wkv_internal.cuh"

#include <cuda.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

namespace wkv {
namespace {

using namespace tc;

constexpr int kMaxStages = 4;
// Ring depth: two 128-row blocks of Q and their two buffers of token scores leave room for three stages (a key tile
// lasts twice as long there; the fourth stage made no difference)
__host__ __device__ constexpr int stages_for(int mb) { return mb == 2 ? 3 : kMaxStages; }
constexpr int kEarlyTiles = 2;                           // key tiles requested ahead of the Q image at the start of an item
constexpr int kMaxGroups = 4;
__host__ __device__ constexpr int groups_for(int) { return 4; }
__host__ __device__ constexpr int block_threads(int mb) { return 64 + groups_for(mb) * 128; }
constexpr int kTile = kTcTileKeys;                       // keys per tile
constexpr int kRegion = kTile * 128;                     // bytes of one 64-column block of a key tile
constexpr uint32_t kTmemCols = 512;                      // all of tensor memory: four accumulator buffers,
constexpr uint32_t kTmemBase = 0;                        // which therefore begin with its first column
constexpr uint32_t kNoTmem = ~0u;
constexpr int kChunkCap = kTcChunkCap;                   // token scores a block may hold

struct TcArgs {
    KShape s;
    StatEntry *stats;       // [units][n_stat_chunks][r_pad]: published statistics of sweep 1
    StatEntry *scores;      // [units][kw_max]: published window scores, for the block that selects
    float *window_scores;
    float *token_scores;
    const float *lse_obs;   // [B, H_q, alpha] natural log of Eq. 1's normalisers from the caller, or null
    int *window_idx;        // fused selection when non-null
    int *kept_len;
    int *status;
    int *sync;
    LaunchCount *count;
    unsigned salt;          // part of the launch's tag
    int n_stat_chunks, r_pad;
    int chunks_per_unit, units_per_wave;
    int kblocks;            // head_dim / 64
    int slot_tok, slot_h, slot_b;   // which tensor-map coordinate (1..3) carries token / head / batch
    unsigned alpha_inverse; // ceil(2^16 / alpha): r * alpha_inverse >> 16 is r / alpha for r, alpha <= 256
    int r16;                // observation rows rounded up to a multiple of 16
    int looks;              // ONE: how often a block looks for another's words before it does without
    int alone;              // ONE: it does without all statistics but its own, whether they have come or not
};

__device__ __forceinline__ uint8_t *align_1024(uint8_t *p)
{
    return reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(p) + 1023u) & ~uintptr_t(1023u));
}

struct Barriers {
    uint64_t full[kMaxStages];        // TMA -> MMA: the stage holds a key tile
    uint64_t empty[kMaxStages];       // MMA -> TMA: the MMAs that read the stage have completed
    uint64_t tfull[kMaxGroups];    // MMA -> compute group: the accumulator buffer is complete
    uint64_t tempty[kMaxGroups];   // compute group -> MMA: the accumulator buffer has been read
};

__device__ __forceinline__ void init_barriers(Barriers &bar)
{
    for (int i = 0; i < kMaxStages; ++i) {
        mbar_init(&bar.full[i], 1);
        mbar_init(&bar.empty[i], 1);
    }
    for (int i = 0; i < kMaxGroups; ++i) {
        mbar_init(&bar.tfull[i], 1);
        mbar_init(&bar.tempty[i], 4);      // one arrival per warp of the group
    }
    fence_barrier_init();
}

// A compute warp waits through its lane 0 only (fewer threads hammering the barrier word leaves the
// shared-memory / special-function issue queue to the real work); the result is broadcast.
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag, int lane)
{
    int ok = 1;
    if (lane == 0) ok = mbar_wait(bar, parity, abort_flag) ? 1 : 0;
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}
// every lane has finished reading the accumulator buffer: hand it back to the MMA warp
__device__ __forceinline__ void warp_release(uint64_t *bar, int lane)
{
    tc_fence_before_sync();
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
}

// Hand-over between blocks: every partial statistic and, where the launch
// selects, every window score is published as one 16-byte word of value and tag, written and read as a whole, so that
// it says itself whether it is there: no fence, no counter, and the data arrives with the answer.  The tag holds the
// number of this launch on the workspace (LaunchCount), which what an earlier launch has left behind, of whatever
// shape, cannot equal.  8 heads x 4,096 keys: 2.3 us from the end of sweep 1 to the normalisers and 3.3 us from the pooled
// windows to the selection; with counters raised by a release and polled it was 3.7 and 4.6 us.
// No block waits before it has finished all its sweep-1 work, so every wait among running blocks ends; ONE does without
// blocks that do not run, and in a cooperative launch all do.  Bounded there: a thread that looks for longer than two
// seconds gives up and sets the block's abort flag.

// The value, but nothing that is computed from it before this point: what only the ends of an item need would otherwise
// be computed ahead of the tile loops and take their registers.
__device__ __forceinline__ int late(int x)
{
    asm volatile("" : "+r"(x));
    return x;
}

// geometry of one work item
struct Item {
    int unit, chunk, b, h;
    int n, n_r;
    long long off;
    int j_begin, j_end, n_tiles;
    int reuse;   // sweep 2: the stage ring still holds the item's last tiles from sweep 1
};
template <bool EARLY = false>
__device__ __forceinline__ void set_item(const TcArgs &a, int unit, int chunk, int review_only, Item &im)
{
    const KShape &s = a.s;
    im.unit = unit;
    im.chunk = chunk;
    im.b = unit / s.hkv;
    im.h = unit - im.b * s.hkv;
    if (s.cu) {
        const int from = length_word<EARLY>(s.cu + im.b), to = length_word<EARLY>(s.cu + im.b + 1), lo = min(max(from, 0), s.total_rows);
        im.n = min(min(max(to - from, 0), s.n_cap), s.total_rows - lo);
        im.off = lo;
    } else {
        im.n = s.max_seqlen;
        im.off = 0;
    }
    im.n_r = im.n - s.alpha;
    const int n_keys = review_only ? im.n_r : im.n;
    const int len = tc_chunk_len(n_keys > 0 ? n_keys : 1, a.chunks_per_unit, review_only ? s.omega : 1);
    im.j_begin = chunk * len;
    im.j_end = min(n_keys, im.j_begin + len);
    im.n_tiles = im.j_end > im.j_begin ? (im.j_end - im.j_begin + kTile - 1) / kTile : 0;
    im.reuse = 0;
}
// Tile taken at step u of an item.  Sweep 1 and a sweep 2 that has to load everything go through the
// tiles in ascending order.  A block that scores the item it has just taken statistics of still holds
// that item's last STAGES tiles in the ring, in ring order: it scores those first, without
// loading them again, and then walks down through the rest.
template <int STAGES>
__device__ __forceinline__ int tile_at(bool reuse, int n_tiles, int u)
{
    if (!reuse) return u;
    return u < STAGES ? n_tiles - STAGES + u : n_tiles - 1 - u;
}

// The compute groups' part of the two sweeps.  Accumulators are numbered v = tile * MB + row half across the block's tile
// stream, `it` tiles lie before the item's, and group `grp` of NG takes those with v mod NG = grp.  Shared memory is passed
// by its 32-bit addresses, so that it is known as such in the calls below too.
struct GroupBarriers {
    uint32_t tfull, tempty, abort_flag;
};
template <typename T>
__device__ __forceinline__ T *shared_at(uint32_t addr)
{
    return static_cast<T *>(__cvta_shared_to_generic(addr));
}
struct StatsSweep {
    int nslot, col0;        // 32-column slots of an accumulator this thread reduces, and the first one's column
    int limit;              // last key the thread's row may attend to
    int j_begin, j_plain;   // first key of the item; tiles that end before j_plain need no masking
};
template <int MB>
__device__ __forceinline__ float2 stats_sweep(GroupBarriers gb, StatsSweep w, uint32_t taddr, uint32_t it, int n_tiles, int grp, float c)
{
    constexpr int NG = groups_for(MB);
    uint64_t *const tfull = shared_at<uint64_t>(gb.tfull), *const tempty = shared_at<uint64_t>(gb.tempty);
    volatile int *const abort_flag = shared_at<volatile int>(gb.abort_flag);
    const int lane = threadIdx.x & 31;
    float m = -INFINITY, l = 0.f;
    for (uint32_t v = it * MB; v < (it + n_tiles) * MB; ++v) {
        if ((int)(v % NG) != grp) continue;
        const int tile0 = w.j_begin + (int)(v / MB - it) * kTile;
        if (!warp_wait(tfull, (v / NG) & 1, abort_flag, lane)) break;
        tc_fence_after_sync();
        const bool fast = tile0 + kTile - 1 < w.j_plain;     // no masking
        for (int sl = 0; sl < w.nslot; ++sl) {
            float x[32];
            tmem_ld32(taddr + sl * 32, x);
            if (sl + 1 == w.nslot) warp_release(tempty, lane);   // the buffer may be overwritten now
            stats_update<true>(x, fast, tile0 + w.col0 + sl * 32, w.limit, c, m, l);
        }
    }
    return make_float2(m, l);
}
struct ScoreSweep {
    int rows;               // of the group's half: 32-row slices; a 16-row tail follows if their number has bit 4 set
    uint32_t neg_lse2, t_out;
    int n_keys;
    bool reuse;
    float *token_out;       // or null
};
template <int MB>
__device__ __forceinline__ void score_sweep(GroupBarriers gb, ScoreSweep w, uint32_t taddr, uint32_t it, int n_tiles, int grp, int L, float c)
{
    constexpr int NG = groups_for(MB);
    uint64_t *const tfull = shared_at<uint64_t>(gb.tfull), *const tempty = shared_at<uint64_t>(gb.tempty);
    volatile int *const abort_flag = shared_at<volatile int>(gb.abort_flag);
    const float *const neg_lse2 = shared_at<const float>(w.neg_lse2);
    float *const t_out = shared_at<float>(w.t_out);
    const int lane = threadIdx.x & 31;
    const int n32 = w.rows >> 5;
    const bool tail = (w.rows & 16) != 0;
    for (uint32_t v = it * MB; v < (it + n_tiles) * MB; ++v) {
        if ((int)(v % NG) != grp) continue;
        if (!warp_wait(tfull, (v / NG) & 1, abort_flag, lane)) break;
        tc_fence_after_sync();
        unsigned long long a01 = 0ull, a23 = 0ull;
        for (int sl = 0; sl < n32; ++sl) {
            float x[32];
            tmem_ld32(taddr + sl * 32, x);
            if (sl + 1 == n32 && !tail) warp_release(tempty, lane);   // the buffer may be overwritten now
            score_accumulate<32, true>(x, neg_lse2 + sl * 32, c, a01, a23);
        }
        if (tail) {
            float x[16];
            tmem_ld16(taddr + n32 * 32, x);
            warp_release(tempty, lane);
            score_accumulate<16, true>(x, neg_lse2 + n32 * 32, c, a01, a23);
        }
        const float2 s01 = halves_of(a01), s23 = halves_of(a23);
        const float tj = (s01.x + s01.y) + (s23.x + s23.y);
        const int j = tile_at<stages_for(MB)>(w.reuse, n_tiles, (int)(v / MB - it)) * kTile + L;
        if (j < w.n_keys) {
            t_out[j] = tj;
            if (w.token_out) w.token_out[j] = tj;
        }
    }
}
// Eq. 1's normaliser of every row from the published statistics of a unit's `used` chunks (row r's of chunk c at
// st[c * r_pad + r]) -> -log2 of it in neg_lse2.  `tl`: number of the compute thread; MERGERS neighbouring ones share a row.
// LOOK of a thread's words are looked at together, `looks` times, or (PATIENT) until they come or the wait expires.
template <int MERGERS, int LOOK, bool PATIENT>
__device__ __forceinline__ void merge_stats(const StatEntry *st, int used, int rows, int r_pad, unsigned long long tag, int tl,
                                            float *neg_lse2, volatile int *flag, int looks)
{
    const int r = tl / MERGERS, mp = tl % MERGERS;
    float M = -INFINITY, sum = 0.f;
    if (r < rows) {
        for (int c0 = mp; c0 < used; c0 += LOOK * MERGERS) {
            unsigned wanted = 0u;
#pragma unroll
            for (int u = 0; u < LOOK; ++u) wanted |= (c0 + u * MERGERS < used ? 1u : 0u) << u;
            StatEntry e[LOOK];
            if (PATIENT) wait_entries<LOOK>(st + r + (size_t)c0 * r_pad, (size_t)MERGERS * r_pad, wanted, tag, e, flag);
            else look_for_entries<LOOK>(st + r + (size_t)c0 * r_pad, (size_t)MERGERS * r_pad, wanted, tag, e, flag, looks);
            float2 p[LOOK];
            float Mn = M;
#pragma unroll
            for (int u = 0; u < LOOK; ++u) {
                p[u] = make_float2(wanted >> u & 1u ? __uint_as_float((unsigned)e[u].value) : -INFINITY,
                                   wanted >> u & 1u ? __uint_as_float((unsigned)(e[u].value >> 32)) : 0.f);
                Mn = fmaxf(Mn, p[u].x);
            }
            if (Mn > -INFINITY) {
                sum *= fast_exp2(M - Mn);
#pragma unroll
                for (int u = 0; u < LOOK; ++u)
                    if (p[u].y > 0.f) sum += p[u].y * fast_exp2(p[u].x - Mn);
                M = Mn;
            }
        }
    }
    __syncwarp();
    float Ma = M;
#pragma unroll
    for (int o = 1; o < MERGERS; o <<= 1) Ma = fmaxf(Ma, __shfl_xor_sync(0xffffffffu, Ma, o));
    sum = sum > 0.f ? sum * fast_exp2(M - Ma) : 0.f;
#pragma unroll
    for (int o = 1; o < MERGERS; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (mp == 0) neg_lse2[r] = sum > 0.f ? -(Ma + log2f(sum)) : -INFINITY;
}

// ---------------------------------------------------------------------------------------------
// the kernel
// ---------------------------------------------------------------------------------------------
// A block's state in shared memory, beside the images of Q and of the key tiles
// what a block takes from wave to wave
struct Carry {
    uint32_t it;          // key tiles it has pushed through the pipeline so far
    uint32_t issued;      // tiles whose loads have been issued
    int q_unit_loaded;    // unit whose Q image is in shared memory, -1: none
};
template <int MB>
struct Shared {
    int counted;                               // the block is among the launch's counted blocks
    __align__(8) Barriers bar;
    uint32_t tmem_base;                        // kNoTmem until tensor memory has been taken
    int abort;
    int late;                                  // ONE: a statistic has not come in time
    int left_over;                             // ONE: a window score has not, or another block's selection is left to this one
    unsigned last_chunk;                       // ONE: the unit's last chunk that holds review keys
    unsigned long long tag;                    // what this launch marks its published words with
    float2 part[groups_for(MB)][128 + 8];      // sweep 1: a group's (max, sum) of the rows on its lanes
    __align__(16) float neg_lse2[256];         // -log2 of the row normaliser; -inf for padding rows
    __align__(16) float t_chunk[MB][kChunkCap];   // sweep 2: per half, the key's sum over that half's rows
    TopkSmem topk;
};
template <int MB>
__device__ __forceinline__ Shared<MB> &shared_state()
{
    __shared__ Shared<MB> state;
    return state;
}
extern __shared__ uint8_t smem_raw[];

// The selection as a call, where a block goes through several waves: its registers would otherwise be laid over what
// lives from wave to wave.
template <int MB>
__device__ __noinline__ void select_call(PublishedScores<1> src, int kw, int k, int k_max, int *out, int *kept_len, int n, int alpha, int omega)
{
    select_topk_block<block_threads(MB)>((int)threadIdx.x, shared_state<MB>().topk, src, kw, k, k_max, out, kept_len, n, alpha, omega);
}

// What a block of ONE does when words have not come in time.  The blocks that should publish them may not have started,
// and may be unable to before this one ends (another stream's kernel, of this library or not, holds their SMs).
//
// Window scores: the selection is left to the block that counts itself last on the unit's ticket, by when all blocks are
// publishing.  `ticket[1]` says so.  By the whole block, at its end: the one that has waited in vain (the last may have
// counted itself meanwhile: then it selects after all), or the one that has found it gone.
template <int MB>
__device__ __noinline__ void late_selection(const TcArgs &a)
{
    Shared<MB> &sh = shared_state<MB>();
    const KShape &s = a.s;
    const int unit = blockIdx.x / a.chunks_per_unit, chunk = blockIdx.x - unit * a.chunks_per_unit;
    if (chunk == (int)sh.last_chunk) {
        if (threadIdx.x == 0) {
            int *const ticket = a.sync + kSyncTickets + kSyncWordsPerUnit * unit;
            __threadfence();                        // what this block has written of a selection comes before the other's
            atomicExch(ticket + 1, 1);
            __threadfence();
            sh.topk.remaining = atomicAdd(ticket, 0) == 0 && atomicExch(ticket + 1, 0) != 0;
            __threadfence();
            atomicAdd(&a.count->left_over, 1u);
        }
        __syncthreads();
        if (!sh.topk.remaining) return;
        __syncthreads();
    }
    Item im;
    set_item(a, unit, 0, 1, im);
    const int budget = s.budgets ? s.budgets[im.b] : s.budget;
    const int kw = num_windows(im.n, s.alpha, s.omega), k = num_selected_capped(im.n, s.alpha, s.omega, budget, s.k_max);
    const PublishedScores<1> src = {a.scores + (size_t)unit * s.kw_max, sh.tag, &sh.abort, topk_hint(s.R, im.n)};
    select_topk_block<block_threads(MB)>((int)threadIdx.x, sh.topk, src, kw, k, s.k_max, a.window_idx + (size_t)unit * s.k_max,
                                         a.kept_len + unit, im.n, s.alpha, s.omega);
    __syncthreads();
}

// One wave of a block.  The sweeps have no registers to spare, and inside a loop over waves or items everything that
// lives on counts: 8 heads x 65,536 keys, 128 rows, one wave, take 58.1 us as ONE and 61.0 us as the form with a
// loop (65.2 us where that looks at five published words at a time and has the selection inlined, as ONE does).  MB: 128-row blocks of observation rows, 1 (R <= 128) or 2 (R <= 256).  SINGLE: no block has more
// than one item of a wave.  ONE: and there is one wave, so that nothing is kept from item to item.  STAND_IN: with the
// statistics that others have not published (stand_in).
template <int MB, bool ONE, bool SINGLE, bool STAND_IN>
__device__ __forceinline__ void take_wave(const CUtensorMap *tmap, const TcArgs &a, const __nv_bfloat16 *__restrict__ q, int u0,
                                          Carry &carry)
{
    constexpr int NG = groups_for(MB), kStages = stages_for(MB);
    constexpr int kThreads = block_threads(MB);
    constexpr int q_rows = MB * 128;
    constexpr int q_region = q_rows * 128;                // bytes of one 64-column block of the Q image
    // A key tile gives one accumulator of 128 columns per 128-row block of Q ("half" rh = 0, 1 with
    // two row blocks); accumulators are numbered v = tile * MB + rh across the block's whole tile
    // stream, and buffers and compute groups take them round-robin (v mod NG).  With two row blocks a
    // group therefore always works on the same half (NG is even).
    constexpr uint32_t buf_cols = kTmemCols / NG;         // accumulator buffer stride in tensor memory
    static_assert(buf_cols >= kTile, "accumulator buffers exceed tensor memory");

    Shared<MB> &sh = shared_state<MB>();
    Barriers &bar = sh.bar;
    const KShape &s = a.s;
    // (Computed anew in every wave where there are several: kept across the steps at the end of an item it would cost the
    // sweeps their registers.)
    const int tid = ONE ? (int)threadIdx.x : late((int)threadIdx.x);
    const int warp = tid >> 5, lane = tid & 31;
    const int units = ONE ? a.units_per_wave : s.batch * s.hkv;
    const int cpu = a.chunks_per_unit;
    const float c = s.scale_log2;

    uint8_t *q_img = align_1024(smem_raw);
    uint8_t *k_stage0 = q_img + a.kblocks * q_region;
    const int stage_bytes = a.kblocks * kRegion;
    const int ksteps = s.d / 16;
    const uint32_t leader = elect_one();     // lane that acts for its warp where a whole warp issues

    constexpr uint32_t tmem_base = kTmemBase;
    uint32_t &it = carry.it, &p_issued = carry.issued;
    int &q_unit_loaded = carry.q_unit_loaded;

    // Row layout of the Q image: image row r holds observation row (r mod Rp); with Rp < 128 the rows
    // repeat so that all 128 lanes work in sweep 1, each copy taking its own slice of a tile's columns.
    // Rows [0, r16) of the image are the B operand of sweep 2.
    const int Rp = MB == 2 ? 256 : (s.R <= 32 ? 32 : (s.R <= 64 ? 64 : 128));

    // the query head, within the unit's G, that observation row r < 256 belongs to: r / alpha
    auto head_of = [&](int r) { return (int)((unsigned)r * a.alpha_inverse >> 16); };
    auto make_item = [&](int unit, int chunk, int review_only, Item &im) { set_item(a, unit, chunk, review_only, im); };

    // Called by every warp except the producer; ends with a barrier among those warps.  The compute warps load, four loads
    // in flight per thread.  The producer starts streaming key tiles once these small loads
    // have been ISSUED (go_producer): a tile burst issued first would sit in front of them in the
    // SM's memory pipeline for microseconds.
    constexpr int kLoaders = kThreads - 64;               // the compute warps
    auto go_producer = [&]() { asm volatile("bar.arrive 2, %0;" ::"n"(kThreads) : "memory"); };
    auto load_q_image = [&](const Item &im, bool signal) {
        if (ONE ? q_unit_loaded < 0 : q_unit_loaded != im.unit) {
            unsigned long long launches = 0;
            const bool first = q_unit_loaded < 0;      // the number is raised while the launch runs: it is read once
            if (first && threadIdx.x == 32) launches = launches_so_far(a.count);
            const __nv_bfloat16 *q_unit = q + im.b * s.qsb + (long long)im.h * s.G * s.qsh;
            const int vshift = s.d == 128 ? 4 : 3;            // log2(16-byte vectors per row)
            const int total = q_rows << vshift;
            const int loader = warp == 1 ? total : late((int)threadIdx.x) - 64;
            if (warp == 1) {
                if (signal) go_producer();
                // The warp that issues the MMAs takes tensor memory meanwhile, at the block's first item and so behind the wait for
                // the kernel in front: a block of that kernel which shares the SM and has yet to take its own would wait for
                // this one, which waits for that kernel.  That takes as long as the loads, so it comes first: groups of 8 heads, us,
                // ahead of the wait / so / behind a share of the loads / behind the barrier below: 4,096 keys 16.35 / 16.29 / 16.40 /
                // 16.50, 8,192 23.98 / 23.80 / 23.99 / -, selection and four gathers of 32,768 keys, given normalisers 49.3 / 49.4 / 49.5 / -.
                if (first) {
                    __syncwarp();
                    tmem_alloc(&sh.tmem_base, kTmemCols);
                    asm volatile("bar.arrive 4, 64;" ::: "memory");
                }
            }
            for (int base = loader; base < total; base += kLoaders * 4) {
                int4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int idx = base + u * kLoaders;
                    v[u] = make_int4(0, 0, 0, 0);
                    if (idx < total) {
                        const int rq = (idx >> vshift) & (Rp - 1), cc = idx & ((1 << vshift) - 1);
                        if (rq < s.R) {
                            const int g = head_of(rq), i = rq - g * s.alpha;
                            v[u] = __ldg(reinterpret_cast<const int4 *>(q_unit + g * s.qsh + i * s.qst + cc * 8));
                        }
                    }
                }
                if (signal && base == loader) go_producer();
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int idx = base + u * kLoaders;
                    if (idx < total) {
                        const int r = idx >> vshift, cc = idx & ((1 << vshift) - 1);
                        *reinterpret_cast<int4 *>(q_img + (cc >> 3) * q_region + swz128_offset(r, cc & 7)) = v[u];
                    }
                }
            }
            if (signal && warp != 1 && loader >= total) go_producer();   // a thread without a share of the image
            fence_proxy_async_smem();
            if (first && threadIdx.x == 32) sh.tag = launch_tag(launches, a.salt);
            asm volatile("bar.sync 1, %0;" ::"n"(kLoaders + 32) : "memory");
        } else if (signal) {
            go_producer();
        }
    };

    // producer: the item's key tiles into the stage ring (the block-wide tile counter `it` keeps the phases)
    auto produce = [&](const Item &im, int t_begin, int t_end) {
        const int tok0 = (int)im.off + im.j_begin;
        const int bcoord = s.cu ? 0 : im.b;
        for (int t = t_begin; t < t_end; ++t) {
            const uint32_t g = it + t;
            const int st = g % kStages;
            // (the limit of the waits counts from when tensor memory has been had: another kernel on the SM may hold it)
            if (g == kStages) asm volatile("bar.sync 4, 64;" ::: "memory");
            if (g >= kStages && !mbar_wait(&bar.empty[st], ((g / kStages) - 1) & 1, &sh.abort)) return;
            if (im.reuse && t < kStages) {
                // the stage holds this tile already: complete the phase without a load
                if (leader) mbar_arrive(&bar.full[st]);
                ++p_issued;
                continue;
            }
            mbar_arrive_expect_tx_if(leader, &bar.full[st], (uint32_t)stage_bytes);
            const int tok = tok0 + tile_at<kStages>(im.reuse, im.n_tiles, t) * kTile;
            const int c1 = a.slot_tok == 1 ? tok : (a.slot_h == 1 ? im.h : bcoord);
            const int c2 = a.slot_tok == 2 ? tok : (a.slot_h == 2 ? im.h : bcoord);
            const int c3 = a.slot_tok == 3 ? tok : (a.slot_h == 3 ? im.h : bcoord);
            for (int kb = 0; kb < a.kblocks; ++kb)
                tma_load_4d_if(leader, k_stage0 + st * stage_bytes + kb * kRegion, tmap, &bar.full[st], kb * 64, c1, c2, c3);
            ++p_issued;
        }
    };

    // MMA issue for one item.  sweep 1: D[rows, keys] = Q K^T; sweep 2: D[keys, rows] = K Q^T; per key
    // tile one accumulator per 128-row block of Q.
    // One warp issues everything, so its instruction count per tile is on the critical path: the
    // matrix descriptors of Q and of stage 0 are built once, and every k-step only adds a
    // compile-time constant to the address field (the fields above it never change).
    const uint64_t q_desc0 = umma_desc_sw128(smem_u32(q_img));
    const uint64_t k_desc0 = umma_desc_sw128(smem_u32(k_stage0));
    auto issue_tile = [&](auto ksteps_tag, uint32_t d_tmem, uint64_t k_desc, uint64_t q_desc, uint32_t idesc,
                          bool sweep2) {
        constexpr int KSTEPS = decltype(ksteps_tag)::value;
#pragma unroll
        for (int ks = 0; ks < KSTEPS; ++ks) {
            const uint32_t qo = (uint32_t)((ks >> 2) * q_region + (ks & 3) * 32) >> 4;
            const uint32_t ko = (uint32_t)((ks >> 2) * kRegion + (ks & 3) * 32) >> 4;
            if (sweep2) umma_bf16_if(leader, d_tmem, k_desc + ko, q_desc + qo, idesc, ks > 0);
            else umma_bf16_if(leader, d_tmem, q_desc + qo, k_desc + ko, idesc, ks > 0);
        }
    };
    auto issue_mma = [&](const Item &im, auto sweep2_tag) {
        constexpr bool sweep2 = decltype(sweep2_tag)::value;
        const uint32_t stage_step = (uint32_t)stage_bytes >> 4;
        for (int t = 0; t < im.n_tiles; ++t) {
            const uint32_t g = it + t;
            const int st = g % kStages;
            if (!mbar_wait(&bar.full[st], (g / kStages) & 1, &sh.abort)) return;
            const uint64_t k_desc = k_desc0 + (uint64_t)(st * stage_step);
#pragma unroll
            for (int rh = 0; rh < MB; ++rh) {
                const uint32_t v = g * MB + rh;
                const int buf = v % NG;
                if (v >= NG && !mbar_wait(&bar.tempty[buf], ((v / NG) - 1) & 1, &sh.abort)) return;
                tc_fence_after_sync();
                // sweep 2: the rows of this half are the N dimension (a multiple of 16)
                const int n_rows = rh == 0 ? min(a.r16, 128) : a.r16 - 128;
                const uint32_t idesc = sweep2 ? umma_idesc_bf16(128, n_rows) : umma_idesc_bf16(128, kTile);
                const uint64_t q_desc = q_desc0 + (uint64_t)((rh * kRegion) >> 4);
                const uint32_t d_tmem = tmem_base + buf * buf_cols;
                if (ksteps == 8) issue_tile(std::integral_constant<int, 8>{}, d_tmem, k_desc, q_desc, idesc, sweep2);
                else issue_tile(std::integral_constant<int, 4>{}, d_tmem, k_desc, q_desc, idesc, sweep2);
                umma_commit_if(leader, &bar.tfull[buf]);
            }
            umma_commit_if(leader, &bar.empty[st]);
        }
    };

    const int grp = warp >= 2 ? (warp - 2) >> 2 : 0, quarter = warp & 3;
    const int L = quarter * 32 + lane;
    const uint32_t taddr_grp = tmem_base + ((uint32_t)(quarter * 32) << 16) + grp * buf_cols;

    const GroupBarriers gb = {smem_u32(&bar.tfull[grp]), smem_u32(&bar.tempty[grp]), smem_u32(&sh.abort)};
    // sweep-1 compute: the row's partial (max, sum exp2) over the item's keys -> part[grp][L]
    auto compute_stats = [&](const Item &im) {
        StatsSweep w;
        w.nslot = MB == 2 ? kTile / 32 : Rp >> 5;
        w.col0 = MB == 2 ? 0 : L & ~(Rp - 1);               // warp-uniform: Rp is a multiple of 32
        const int row = MB == 2 ? (grp & 1) * 128 + L : L & (Rp - 1);
        w.limit = row < s.R ? min(im.n_r + row - head_of(row) * s.alpha, im.j_end - 1) : -1;
        w.j_begin = im.j_begin;
        w.j_plain = min(im.n_r + 1, im.j_end);
        const uint32_t taddr = taddr_grp + w.col0;
        // (STAND_IN: to the place of the group that has these tiles where they are the block's first)
        sh.part[STAND_IN ? (grp - (int)(it * MB)) & (NG - 1) : grp][L] = stats_sweep<MB>(gb, w, taddr, it, im.n_tiles, grp, c);
    };

    // kMergers neighbouring threads share an observation row when partial statistics are merged, within the block and
    // between the chunks; both in a fixed order
    constexpr int kComputeThreads = kThreads - 64;
    constexpr int kMergers = kComputeThreads / q_rows;
    constexpr int kLook = ONE ? 5 : 2;         // (the rounding of a normaliser depends on it)
    auto compute_barrier = [&]() { asm volatile("bar.sync 3, %0;" ::"n"(kComputeThreads) : "memory"); };

    // combines the compute groups and the column slices of each row and publishes the item's statistics
    auto publish_stats = [&](const Item &im) {
        const int tl = late((int)threadIdx.x) - 64, r = tl / kMergers, mp = tl % kMergers;
        // with two row blocks a row lives in the groups of its half (group index odd or even)
        const float2 *mine = MB == 2 ? &sh.part[(r >> 7) + 2 * mp][r & 127] : &sh.part[mp][r];
        float2 p[4];
#pragma unroll
        for (int cp = 0; cp < 4; ++cp) p[cp] = (MB == 2 ? cp == 0 : (r < Rp && cp * Rp < 128)) ? mine[cp * Rp] : make_float2(-INFINITY, 0.f);
        float M = fmaxf(fmaxf(p[0].x, p[1].x), fmaxf(p[2].x, p[3].x));
#pragma unroll
        for (int o = 1; o < kMergers; o <<= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
        float sum = 0.f;
#pragma unroll
        for (int cp = 0; cp < 4; ++cp)
            if (p[cp].y > 0.f) sum += p[cp].y * fast_exp2((p[cp].x - M) * c);
#pragma unroll
        for (int o = 1; o < kMergers; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (mp == 0 && r < s.R && !*static_cast<volatile int *>(&sh.abort))
            publish_entry(a.stats + ((size_t)im.unit * a.n_stat_chunks + im.chunk) * a.r_pad + r,
                          (unsigned long long)__float_as_uint(M * c) | (unsigned long long)__float_as_uint(sum) << 32, sh.tag);
    };

    // sweep-2 compute: token score of key L of every tile of the item -> t_chunk (and token_scores)
    auto compute_scores = [&](const Item &im) {
        const int rh = MB == 2 ? (grp & 1) : 0;
        ScoreSweep w;
        w.rows = rh == 0 ? min(a.r16, 128) : a.r16 - 128;
        w.neg_lse2 = smem_u32(sh.neg_lse2 + rh * 128);
        w.t_out = smem_u32(sh.t_chunk[rh]);
        w.n_keys = im.j_end - im.j_begin;
        w.reuse = im.reuse;
        w.token_out = MB == 1 && a.token_scores ? a.token_scores + (size_t)im.unit * s.nr_max + im.j_begin : nullptr;
        score_sweep<MB>(gb, w, taddr_grp, it, im.n_tiles, grp, L, c);
    };

    auto block_barrier = [&]() {
        tc_fence_before_sync();
        __syncthreads();
        tc_fence_after_sync();
    };
    const int n_items = ONE ? (int)gridDim.x : min(a.units_per_wave, units - u0) * cpu;
    int item;

    if constexpr (STAND_IN) {
        static_assert((NG & (NG - 1)) == 0, "groups are numbered modulo a power of two");
        Item im;
        const int unit = (int)blockIdx.x / cpu, own = (int)blockIdx.x - unit * cpu;
        make_item(unit, 0, 0, im);
        const int used1 = (im.n + im.j_end - 1) / im.j_end;     // chunks of the unit that hold keys in sweep 1
        const StatEntry *const words = a.stats + (size_t)unit * a.n_stat_chunks * a.r_pad;
        unsigned taken = 0;
        for (int x = 1; x <= used1; ++x) {
            const int chunk = (own + x) % used1;
            const int lacks = tid < s.R && (a.alone ? chunk != own : read_entry(words + (size_t)chunk * a.r_pad + tid).tag != sh.tag);
            if (!__syncthreads_or(lacks)) continue;
            make_item(unit, chunk, 0, im);
            if (warp == 0) {
                produce(im, 0, im.n_tiles);
            } else if (warp == 1) {
                issue_mma(im, std::false_type{});
            } else {
                compute_stats(im);
                compute_barrier();
                publish_stats(im);
            }
            it += im.n_tiles;
            ++taken;
            block_barrier();
            if (*static_cast<volatile int *>(&sh.abort)) return;
        }
        if (threadIdx.x == 0 && taken) atomicAdd(&a.count->stood_in, taken);
    }

    // ------------------------------------------------------------------ sweep 1
    // (not needed when the caller supplies the normalisers: sweep 2 then reads the keys from HBM)
    item = blockIdx.x;
    if (!STAND_IN && !a.lse_obs && (ONE || item < n_items)) do {
        Item im;
        const int nth = item / cpu;
        make_item(u0 + nth, item - nth * cpu, 0, im);
        if (im.n_r <= 0 || im.n_tiles == 0) continue;
        if (!ONE && q_unit_loaded != im.unit && q_unit_loaded >= 0) block_barrier();   // the image is still being read
        if (warp == 0) {
            // the first tiles leave before the loads of the Q image (they land while those are
            // being issued); the rest of the ring's burst follows once the Q loads are on their way
            const int early = min(kEarlyTiles, im.n_tiles);
            produce(im, 0, early);
            asm volatile("bar.sync 2, %0;" ::"n"(kThreads) : "memory");
            produce(im, early, im.n_tiles);
        } else {
            load_q_image(im, true);
            if (warp == 1) {
                issue_mma(im, std::false_type{});
            } else {
                compute_stats(im);
                compute_barrier();
                publish_stats(im);
            }
        }
        // No barrier of the whole block here: the TMA and MMA warps run on into the second sweep, whose first
        // accumulators fill as the last ones of this one are read.
        q_unit_loaded = im.unit;
        it += im.n_tiles;
        if (!SINGLE && item + (int)gridDim.x < n_items) block_barrier();   // `part` is rewritten by the next item
    } while (!SINGLE && (item += gridDim.x) < n_items);

    // ------------------------------------------------------------------ sweep 2 (+ selection)
    item = blockIdx.x;
    if (ONE || item < n_items) do {
        Item im;
        const int nth = item / cpu;
        make_item(u0 + nth, item - nth * cpu, 1, im);
        // read now, needed only by the block that selects: the load is long done by then
        const int budget = a.window_idx ? (s.budgets ? __ldg(s.budgets + im.b) : s.budget) : 0;
        if (im.n_r <= 0 || im.n_tiles == 0) {
            // a unit without review context still gets its (empty) selection, from its first item
            if (a.window_idx && im.n_r <= 0 && im.chunk == 0) {
                for (int x = threadIdx.x; x < s.k_max; x += kThreads) a.window_idx[(size_t)im.unit * s.k_max + x] = -1;
                if (threadIdx.x == 0) a.kept_len[im.unit] = min(im.n, s.alpha);
            }
            __syncthreads();   // as at the end of every item: what made the block give up has been seen by all
            continue;
        }
        if (!SINGLE && q_unit_loaded != im.unit && q_unit_loaded >= 0) block_barrier();   // the image is still being read
        const int len1 = tc_chunk_len(im.n, cpu, 1);
        // the ring holds the last tiles of the block's one item of the wave, if they are this sweep's tiles too
        const int keys1 = min(im.n - im.chunk * len1, len1);
        im.reuse = !STAND_IN && !a.lse_obs && (SINGLE || (item == (int)blockIdx.x && item + (int)gridDim.x >= n_items)) &&
                   im.n_tiles >= kStages && im.chunk * len1 == im.j_begin && (keys1 + kTile - 1) / kTile == im.n_tiles;
        if (warp == 0) {
            // ahead of the small loads of this item: the tiles the ring still holds (no traffic), or
            // the first tiles as in sweep 1
            const int ahead = im.reuse ? kStages : min(kEarlyTiles, im.n_tiles);
            produce(im, 0, ahead);
            asm volatile("bar.sync 2, %0;" ::"n"(kThreads) : "memory");
            produce(im, ahead, im.n_tiles);
        } else {
            load_q_image(im, false);
            if (warp == 1) {
                // the MMAs do not need the normalisers: the first accumulators fill while the
                // compute warps merge the statistics
                go_producer();
                issue_mma(im, std::true_type{});
                // the block counts itself, once, now that it has read the number of launches
                if (lane == 0 && !STAND_IN && (ONE || !sh.counted)) {
                    count_launch(a.count, launch_of(sh.tag), gridDim.x);
                    sh.counted = 1;
                    if (ONE) {
                        const int len2 = tc_chunk_len(im.n_r, cpu, s.omega);
                        sh.last_chunk = (unsigned)((im.n_r - 1) / len2);
                    }
                }
            } else {
            const int tl = late((int)threadIdx.x) - 64;
            if (a.lse_obs) {
                // the caller's normalisers, to base 2; row r = (query head g of the group, position i)
                if (tl < 256) {
                    float v = -INFINITY;
                    if (tl < s.R) {
                        const int g = head_of(tl), i = tl - g * s.alpha;
                        v = -1.4426950408889634f *
                            __ldg(a.lse_obs + ((size_t)im.b * s.hq + (size_t)im.h * s.G + g) * s.alpha + i);
                    }
                    sh.neg_lse2[tl] = v;
                }
                go_producer();
            } else {
                go_producer();
                const StatEntry *st = a.stats + (size_t)im.unit * a.n_stat_chunks * a.r_pad;
                const int used1 = (im.n + len1 - 1) / len1;    // chunks of the unit that hold keys in sweep 1
                constexpr bool patient = !ONE || STAND_IN;
                merge_stats<kMergers, kLook, patient>(st, used1, s.R, a.r_pad, sh.tag, tl, sh.neg_lse2, patient ? &sh.abort : &sh.late, a.looks);
            }
            compute_barrier();
            compute_scores(im);     // (for nothing if a statistic is late: the accumulators on their way have to be taken)
            }
        }
        q_unit_loaded = im.unit;
        it += im.n_tiles;
        block_barrier();
        if (sh.abort) break;
        if (ONE && !STAND_IN && *static_cast<volatile int *>(&sh.late)) break;     // (stand_in, at the block's end)
        float *t_item = &sh.t_chunk[0][0];
        if (MB == 2) {
            // Eq. 2 sums over all rows: add the two halves' sums of every key
            for (int x = threadIdx.x; x < im.j_end - im.j_begin; x += kThreads) {
                const float tj = sh.t_chunk[0][x] + sh.t_chunk[MB - 1][x];
                t_item[x] = tj;
                if (a.token_scores) a.token_scores[(size_t)im.unit * s.nr_max + im.j_begin + x] = tj;
            }
            __syncthreads();
        }
        const int tid = late((int)threadIdx.x);
        // the unit's ticket counts the blocks that are past all waiting for one another
        int *ticket = a.sync + kSyncTickets + kSyncWordsPerUnit * im.unit;
        const bool last_chunk = im.j_end == im.n_r;     // of those that hold keys in sweep 2
        if (ONE) {
            // Every block of the unit counts itself and the last leaves the ticket at zero.  By a thread of the last warp, which is
            // the last to get windows to pool.
            if (threadIdx.x == kThreads - 32) {
                int left = 0;
                if (a.window_idx) {
                    const unsigned last = sh.last_chunk, before = atomicInc(reinterpret_cast<unsigned *>(ticket), last);
                    if (before > last) atomicOr(a.status, kStatusWaitExpired);   // the workspace was not cleared
                    if (before == last && !last_chunk) {
                        __threadfence();
                        left = atomicExch(ticket + 1, 0);
                        __threadfence();
                    }
                }
                sh.left_over = left;
            }
        } else if (a.window_idx && !a.lse_obs && !last_chunk && threadIdx.x == 0) {
            atomicAdd(ticket, 1);
        }
        // Eq. 3-4: the item's windows (its first key is a multiple of omega)
        {
            const int n_tok = im.j_end - im.j_begin;
            const int omega = late(s.omega);
            const size_t w0 = (size_t)im.unit * s.kw_max + im.j_begin / omega;
            float *ws_out = a.window_scores + w0;
            auto put = [&](int lw, float r) {
                ws_out[lw] = r;
                if (a.window_idx) publish_entry(a.scores + w0 + lw, __float_as_uint(r), sh.tag);
            };
            const int n_win = (n_tok + omega - 1) / omega;
            if (s.omega == 16 || s.omega == 8 || s.omega == 32 || s.omega == 4) {
                // consecutive windows go to different warps so that all four schedulers take part
                for (int lw = tid; lw < n_win; lw += kThreads) {
                    const int lo = lw * s.omega, size = min(s.omega, n_tok - lo);
                    float r;
                    if (s.omega == 16) r = pool_window_sorted<16>(t_item + lo, size, s.p, tid & 31);
                    else if (s.omega == 8) r = pool_window_sorted<8>(t_item + lo, size, s.p, tid & 31);
                    else if (s.omega == 32) r = pool_window_sorted<32>(t_item + lo, size, s.p, tid & 31);
                    else r = pool_window_sorted<4>(t_item + lo, size, s.p, tid & 31);
                    put(lw, r);
                }
            }
            else if (s.omega == 64 || s.omega == 128) {
                // one warp per window
                for (int lw = tid >> 5; lw < n_win; lw += kThreads / 32) {
                    const int lo = lw * s.omega, size = min(s.omega, n_tok - lo);
                    const float r = s.omega == 64 ? pool_window_warp<64>(t_item + lo, size, s.p, tid & 31)
                                                  : pool_window_warp<128>(t_item + lo, size, s.p, tid & 31);
                    if ((tid & 31) == 0) put(lw, r);
                }
            }
            else {
                for (int lw = tid; lw < n_win; lw += kThreads) {
                    const int lo = lw * s.omega;
                    put(lw, pool_top_p(t_item + lo, min(s.omega, n_tok - lo), s.p));
                }
            }
        }
        // The block of the unit's last chunk selects for the unit, from the published scores: that
        // chunk is usually a short one, so its block is done early and the selection does not sit
        // on the path of a block that the next wave is waiting for.
        if (ONE && a.window_idx && last_chunk) {
            __syncthreads();
            const PublishedScores<4, false> src = {a.scores + (size_t)im.unit * s.kw_max, sh.tag, &sh.left_over, topk_hint(s.R, im.n), a.looks};
            const int kw = num_windows(im.n, s.alpha, late(s.omega));
            const int k = num_selected_capped(im.n, s.alpha, late(s.omega), budget, s.k_max);
            select_topk_block<kThreads>((int)threadIdx.x, sh.topk, src, kw, k, s.k_max, a.window_idx + (size_t)im.unit * s.k_max,
                                        a.kept_len + im.unit, im.n, s.alpha, s.omega);
        }
        if constexpr (!ONE) {
            bool selects = last_chunk;
            // With given normalisers nothing else makes a block wait for another, and the selection does not
            // either: the block that counts itself last selects, so the launch need not be cooperative.
            if (a.lse_obs && a.window_idx) {
                if (threadIdx.x == 0) {
                    const int before = atomicAdd(ticket, 1);
                    const int len2 = tc_chunk_len(im.n_r, cpu, late(s.omega)), used2 = (im.n_r + len2 - 1) / len2;
                    if (before == used2 - 1) atomicExch(ticket, 0);
                    if (before < 0 || before >= used2) atomicOr(a.status, kStatusWaitExpired);   // workspace not cleared
                    sh.topk.remaining = before == used2 - 1;
                }
                __syncthreads();
                selects = sh.topk.remaining != 0;
            }
            if (a.window_idx && selects) {
                __syncthreads();                 // a wait that expires from here on is seen by all at the same place
                const PublishedScores<1> src = {a.scores + (size_t)im.unit * s.kw_max, sh.tag, &sh.abort, topk_hint(s.R, im.n)};
                const int kw = num_windows(im.n, s.alpha, late(s.omega));
                const int k = num_selected_capped(im.n, s.alpha, late(s.omega), budget, s.k_max);
                int *const out = a.window_idx + (size_t)im.unit * s.k_max;
                select_call<MB>(src, kw, k, s.k_max, out, a.kept_len + im.unit, im.n, s.alpha, s.omega);
                // the others counted themselves before they published what has just been read: no wait in practice
                if (!a.lse_obs && threadIdx.x == 0 && poll_until_at_least(ticket, im.chunk, &sh.abort)) atomicExch(ticket, 0);
            }
        }
        if (!ONE) __syncthreads();   // t_chunk, neg_lse2 and the selection scratch are reused by the next item
    } while (!SINGLE && (item += gridDim.x) < n_items);
}

// Statistics that have not come in time: the block takes those of every chunk that still lacks some, tile by tile as that
// chunk's block does, in the same order and by the same instructions, so that no bit of the result depends on which of the two
// a normaliser comes from.  By the whole block, at its end; sweep 2, which has taken the accumulators on their way, is repeated.
// Blocks that stand in together begin with different chunks and take what another of them has published.  A launch in which every
// block takes every chunk of the longest unit, 148 of 37 tiles, lasts 5.3 ms (36 us a chunk), 8.6 with 256 rows (59).  Returns the
// number of tiles whose loads the block has issued.
// Inlined, and not called ahead of the pooling: what a call keeps on the stack cost every launch 0.1 to 0.5 us of 16 to 53.
template <int MB>
__device__ __forceinline__ uint32_t stand_in(const CUtensorMap *tmap, const TcArgs &a, const __nv_bfloat16 *q)
{
    const int unit = blockIdx.x / a.chunks_per_unit, chunk = blockIdx.x - unit * a.chunks_per_unit;
    Item first, second;
    set_item(a, unit, chunk, 0, first);
    set_item(a, unit, chunk, 1, second);
    const uint32_t tiles = first.n_tiles + second.n_tiles;      // all that the block has had so far
    Carry carry = {tiles, tiles, unit};
    take_wave<MB, true, true, true>(tmap, a, q, 0, carry);
    return carry.issued;
}

// The unit's Q and the block's first key tile on their way to L2 while the kernel in front drains.  Only a sequence's lengths are
// read here, from L2 and anew behind the wait; lengths that are not the final ones make no more than a wasted fetch inside the tensors.  Passes back to back, us, without / with one tile / two / four / sixteen: 8 heads x 8,192 keys 24.8 /
// 23.8 / 23.9 / 24.2 / 24.2, 16,384 36.3 / 34.6 / 34.6 / 35.0 / 36.0, 32,768 53.5 / 52.0 / 52.2 / 52.5 / 54.8, 3 ragged
// sequences of 2 heads x 12,289 30.1 / 28.5 / 28.7 / 29.1 / 29.2: more only takes bandwidth from the kernel in front.
template <int MB>
__device__ __forceinline__ void fetch_ahead(const CUtensorMap *tmap, const TcArgs &a, const __nv_bfloat16 *q)
{
    const KShape &s = a.s;
    const int unit = blockIdx.x / a.chunks_per_unit;
    Item im;
    set_item<true>(a, unit, blockIdx.x - unit * a.chunks_per_unit, a.lse_obs != nullptr, im);
    if (threadIdx.x < 32) {
        if (im.n_tiles > 0 && elect_one()) {
            const int tok = (int)im.off + im.j_begin, bcoord = s.cu ? 0 : im.b;
            const int c1 = a.slot_tok == 1 ? tok : (a.slot_h == 1 ? im.h : bcoord);
            const int c2 = a.slot_tok == 2 ? tok : (a.slot_h == 2 ? im.h : bcoord);
            const int c3 = a.slot_tok == 3 ? tok : (a.slot_h == 3 ? im.h : bcoord);
            for (int kb = 0; kb < a.kblocks; ++kb) tma_prefetch_4d(tmap, kb * 64, c1, c2, c3);
        }
    } else {
        const int shift = a.kblocks - 1;            // a row is one or two lines of 128 bytes
        const __nv_bfloat16 *const q_unit = q + im.b * s.qsb + (long long)im.h * s.G * s.qsh;
        for (int x = (int)threadIdx.x - 32; x < s.R << shift; x += block_threads(MB) - 32) {
            const int r = x >> shift, g = (int)((unsigned)r * a.alpha_inverse >> 16), i = r - g * s.alpha;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(q_unit + g * s.qsh + i * s.qst + (x & shift) * 64));
        }
    }
}

template <int MB, bool ONE, bool SINGLE>
// 18 warps put five on one SM sub-partition (16K registers): 96 registers per thread at most
__global__ void __launch_bounds__(block_threads(MB), 1)
score_windows_tc(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ TcArgs a,
                 const __nv_bfloat16 *__restrict__ q)
{
    constexpr int kStages = stages_for(MB);
    Shared<MB> &sh = shared_state<MB>();
    Barriers &bar = sh.bar;
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        init_barriers(bar);
        sh.abort = 0;
        sh.tmem_base = kNoTmem;
        sh.late = a.alone;
        sh.left_over = 0;
        sh.counted = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) tma_prefetch_desc(&tmap);
    if (ONE) fetch_ahead<MB>(&tmap, a, q);
    pdl_wait();                 // but for what fetch_ahead says, nothing above touches memory of anybody else

    Carry carry = {0, 0, -1};
    if (ONE) {
        take_wave<MB, true, true, false>(&tmap, a, q, 0, carry);
    } else {
        for (int u0 = 0; u0 < a.s.batch * a.s.hkv && !*static_cast<volatile int *>(&sh.abort); u0 += a.units_per_wave)
            take_wave<MB, false, SINGLE, false>(&tmap, a, q, u0, carry);
    }

    // ------------------------------------------------------------------ teardown
    __syncthreads();
    // (of the blocks that have counted themselves: those with keys to score)
    if (ONE && *static_cast<volatile int *>(&sh.late) && sh.counted && !*static_cast<volatile int *>(&sh.abort)) {
        carry.issued = stand_in<MB>(&tmap, a, q);
        __syncthreads();
    }
    if (ONE && *static_cast<volatile int *>(&sh.left_over) && !*static_cast<volatile int *>(&sh.abort)) late_selection<MB>(a);
    if (threadIdx.x == 32 && !sh.counted) count_launch(a.count, launches_so_far(a.count) + 1, gridDim.x);    // a block without an item
    if (warp == 0 && elect_one()) {
        // nothing of this block may be in flight when it ends: the last MMAs must have released
        // their stages; after a failed wait, the loads already issued must still land.  (The lane that issued
        // them knows how many: the lanes of the warp may give up at different tiles.)
        for (uint32_t g = carry.issued > kStages ? carry.issued - kStages : 0; g < carry.issued; ++g) {
            const int st = g % kStages;
            if (!mbar_wait(&bar.empty[st], (g / kStages) & 1, &sh.abort)) {
                volatile int never = 0;
                mbar_wait(&bar.full[st], (g / kStages) & 1, &never);
            }
        }
        if (sh.abort) atomicOr(a.status, kStatusWaitExpired);
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == 1 && sh.tmem_base != kNoTmem) tmem_dealloc(sh.tmem_base, kTmemCols);
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &qres) ==
                cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// Tensor map of the leader's keys: dimension 0 is the head dimension; token, head and batch follow in
// order of increasing stride.  Box = 64 elements x 128 tokens, 128-byte swizzle, zero fill.
bool make_key_tensor_map(const KShape &ks, const void *k, CUtensorMap *tmap, int slot[3])
{
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc) {
        set_error_detail("cuTensorMapEncodeTiled is not available from the driver");
        return false;
    }
    struct Dim {
        unsigned long long size, stride;
        int which;
    } dims[3] = {
        {(unsigned long long)(ks.cu ? ks.total_rows : ks.max_seqlen), (unsigned long long)ks.st * 2ull, 0},
        {(unsigned long long)ks.hkv, (unsigned long long)ks.sh * 2ull, 1},
        {(unsigned long long)(ks.cu ? 1 : ks.batch), (unsigned long long)ks.sb * 2ull, 2},
    };
    // dimensions of size one carry no address information: place them last with a synthetic stride
    std::stable_sort(dims, dims + 3, [](const Dim &x, const Dim &y) {
        const bool x1 = x.size == 1, y1 = y.size == 1;
        if (x1 != y1) return y1;
        return !x1 && x.stride < y.stride;
    });
    unsigned long long running = (unsigned long long)ks.d * 2ull;
    cuuint64_t gdim[4] = {(cuuint64_t)ks.d, 0, 0, 0}, gstride[3];
    cuuint32_t box[4] = {64, 1, 1, 1}, estr[4] = {1, 1, 1, 1};
    for (int i = 0; i < 3; ++i) {
        if (dims[i].size == 1) dims[i].stride = running;
        if (dims[i].stride == 0 || dims[i].stride % 16 || dims[i].stride >= (1ull << 40) ||
            dims[i].size > 0xffffffffull) {
            set_error_detail("key layout cannot be described by a tensor map (dimension %d: size %llu, stride %llu bytes)",
                             dims[i].which, dims[i].size, dims[i].stride);
            return false;
        }
        gdim[i + 1] = dims[i].size;
        gstride[i] = dims[i].stride;
        if (dims[i].which == 0) box[i + 1] = kTile;
        slot[dims[i].which] = i + 1;
        const unsigned long long span = dims[i].stride * dims[i].size;
        if (span > running) running = span;
    }
    const CUresult r = enc(tmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(k), gdim, gstride, box,
                           estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error_detail("cuTensorMapEncodeTiled failed with code %d", (int)r);
        return false;
    }
    return true;
}

// What the launcher needs to know about a device and its copy of the kernels, looked up on the first
// use of that device: kernel attributes (the shared-memory opt-in) belong to a device, so a process
// that drives several GPUs sets them on each.
struct DeviceInfo {
    bool known = false;
    int cc_major = -1;
    int sm_count = 0;
    int cooperative = 0;
    int blocks_per_sm[2][3] = {{-1, -1, -1}, {-1, -1, -1}};   // resident blocks of each instantiation at its largest footprint
};
std::mutex g_device_mutex;
DeviceInfo g_device_info[kMaxDevices];
// the current device's entry (callers hold no lock: entries are only ever filled in, under the mutex)
DeviceInfo *device_info()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        (void)cudaGetLastError();
        return nullptr;
    }
    std::lock_guard<std::mutex> lock(g_device_mutex);
    DeviceInfo &info = g_device_info[dev];
    if (!info.known) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrComputeCapabilityMajor, dev) == cudaSuccess) info.cc_major = v;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess) info.sm_count = v;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess) info.cooperative = v;
        (void)cudaGetLastError();
        info.known = true;
    }
    return &info;
}

size_t tc_smem_bytes(int kblocks, int mb)
{
    return 1024 + (size_t)kblocks * mb * 128 * 128 + (size_t)stages_for(mb) * kblocks * kRegion;
}

}  // namespace

bool score_tc_supported(const KShape &ks, int dtype)
{
    const DeviceInfo *di = device_info();
    return di && dtype == WKV_BF16 && (ks.d == 64 || ks.d == 128) && ks.R <= 256 && ks.omega <= kTcMaxWindow &&
           di->cc_major == 10 && di->cooperative && di->sm_count > 0;
}

int launch_score_tc(const KShape &ks, const void *q, const void *k, float *window_scores, float *token_scores,
                    int *window_idx, int *kept_len, void *workspace, const Workspace &ws, cudaStream_t stream,
                    const float *lse_obs)
{
    alignas(64) CUtensorMap tmap;
    int slot[3] = {1, 2, 3};
    if (!make_key_tensor_map(ks, k, &tmap, slot)) return WKV_ERR_UNSUPPORTED;
    DeviceInfo *dip = device_info();
    if (!dip) {
        set_error_detail("no current CUDA device, or its ordinal is beyond %d", kMaxDevices - 1);
        return WKV_ERR_CUDA;
    }
    DeviceInfo &di = *dip;

    TcArgs a;
    a.s = ks;
    a.stats = reinterpret_cast<StatEntry *>(static_cast<char *>(workspace) + ws.stats_off);
    a.scores = reinterpret_cast<StatEntry *>(static_cast<char *>(workspace) + ws.entries_off);
    a.count = reinterpret_cast<LaunchCount *>(static_cast<char *>(workspace) + ws.count_off);
    a.salt = ws.salt;
    a.window_scores = window_scores;
    a.lse_obs = lse_obs;
    a.token_scores = token_scores;
    a.window_idx = window_idx;
    a.kept_len = kept_len;
    a.status = reinterpret_cast<int *>(static_cast<char *>(workspace) + ws.status_off);
    a.sync = reinterpret_cast<int *>(static_cast<char *>(workspace) + ws.sync_off);
    a.r_pad = ws.r_pad;
    const int units = ks.batch * ks.hkv;
    const TcPlan plan = tc_plan(units, ks.max_seqlen, ks.omega, ks.R);
    a.n_stat_chunks = plan.chunks_per_unit;
    a.chunks_per_unit = plan.chunks_per_unit;
    a.units_per_wave = plan.units_per_wave;
    a.kblocks = ks.d / 64;
    a.slot_tok = slot[0];
    a.slot_h = slot[1];
    a.slot_b = slot[2];
    a.looks = ws.looks;
    a.alone = ws.alone && !lse_obs;
    a.alpha_inverse = (65536u + ks.alpha - 1) / ks.alpha;
    a.r16 = (ks.R + 15) / 16 * 16;

    const int mb = ks.R > 128 ? 2 : 1;
    const int threads = block_threads(mb);
    const size_t smem = tc_smem_bytes(a.kblocks, mb);
    // persistent blocks, one per SM at most.  With several waves the hand-over of the statistics between the sweeps relies on
    // all being resident, which a cooperative launch sees to; in one wave nothing does.
    int grid = plan.units_per_wave * plan.chunks_per_unit;
    if (grid > di.sm_count) grid = di.sm_count;
    const int form = grid < plan.units_per_wave * plan.chunks_per_unit ? 0 : (plan.units_per_wave < units ? 1 : 2);
    const auto kernel = mb == 1 ? (form == 2 ? score_windows_tc<1, true, true> : form == 1 ? score_windows_tc<1, false, true> : score_windows_tc<1, false, false>)
                                : (form == 2 ? score_windows_tc<2, true, true> : form == 1 ? score_windows_tc<2, false, true> : score_windows_tc<2, false, false>);
    const void *fn = reinterpret_cast<const void *>(kernel);
    int &blocks_per_sm = di.blocks_per_sm[mb - 1][form];
    cudaError_t err = cudaSuccess;
    std::unique_lock<std::mutex> setup_lock(g_device_mutex);
    if (blocks_per_sm < 0) {
        // once per device and instantiation: allow its largest shared-memory request (head_dim 128) and ask how
        // many of its blocks an SM holds at that size
        const size_t smem_max = tc_smem_bytes(2, mb);
        err = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
        if (err == cudaSuccess)
            err = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        int occ = 0;
        if (err == cudaSuccess) err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem_max);
        if (err == cudaSuccess) {
            if (occ < 1) {
                cudaFuncAttributes fa;
                (void)cudaFuncGetAttributes(&fa, fn);
                set_error_detail("tensor-core score kernel does not fit an SM (%d threads, %d registers, %zu + %zu bytes "
                                 "of shared memory)", threads, fa.numRegs, smem_max, fa.sharedSizeBytes);
                return WKV_ERR_CUDA;
            }
            blocks_per_sm = occ;
        }
    }
    setup_lock.unlock();
    const __nv_bfloat16 *qp = static_cast<const __nv_bfloat16 *>(q);
    if (err == cudaSuccess) {
        void *params[3] = {&tmap, &a, &qp};
        // A plain launch may start while the kernel in front drains; a cooperative one may not, and begins on a tick of 2 us
        // behind it.  With given normalisers no block waits for another, and in one wave none depends on it (above).  Group
        // calls back to back, cooperative / plain, us: 8 heads x 4,096 keys 18.4 / 16.6, 8,192 26.7 / 24.8, 16,384 38.9 / 36.2; 3
        // ragged sequences of 2 heads x 12,289 32.8 / 30.0.
        if (lse_obs || form == 2) err = launch_pdl(kernel, dim3(grid), threads, smem, stream, 1, tmap, a, qp);
        else err = cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(threads), params, smem, stream);
    }
    if (err != cudaSuccess) {
        (void)cudaGetLastError();
        set_error_detail("tensor-core score kernel (grid %d x %d threads, %zu bytes of shared memory): %s", grid,
                         threads, smem, cudaGetErrorString(err));
        return WKV_ERR_CUDA;
    }
    count_launches(1);
    return WKV_OK;
}

}  // namespace wkv
