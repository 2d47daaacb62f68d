// Budgeted window selection (sentence after Eq. 4) for one unit by one thread block: the k-th
// largest window score is found with a radix select (9 bits per pass, over the range that scores are expected in or
// else over the bits in which the unit's keys differ, finished by direct ranking once few candidates are left) over an
// order-preserving integer image of the fp32 scores, then the selected window indices are emitted
// in ascending order with one block-wide prefix sum.  Equal scores at the threshold go to the
// lower window index.  Integer arithmetic only after the key mapping, so the result is exact and
// deterministic.  Used by the stand-alone selection kernel and by the fused score kernels.
//
// The whole selection is a chain of short dependent steps, so it is written for latency: block-wide
// reductions go through one word per warp and one warp-reduce instruction per reader (one barrier
// each), the histogram is searched by all warps at once, and the first pass needs no look at the keys' range where
// the caller can say where scores lie.  510 windows on 18 warps: 2.0 us once the keys are there (histogram 0.2, search
// 0.5, ranking 0.5, prefix sum and output 0.6); with a pass over the range first, one warp searching the histogram and a
// prefix sum over the candidates 2.6.
#pragma once

#include "wkv_internal.cuh"

namespace wkv {

constexpr int kTopkDigit = 9;                 // bits resolved per pass
constexpr int kTopkBins = 1 << kTopkDigit;
constexpr int kTopkDirect = 64;               // with at most this many candidates left, rank them directly

struct TopkSmem {
    __align__(16) int hist[kTopkBins];
    __align__(16) unsigned cand[kTopkDirect];
    int warp_sums[2][32];       // two slots: consecutive block scans need no barrier between them
    unsigned warp_min[32], warp_max[32];
    unsigned prefix;
    int remaining;
    int cand_total, n_cand;     // keys in the chosen bin; candidates collected for the direct finish
};

// The NT threads that take part pass their number 0 .. NT - 1 as `tid`.  BAR = 0: they are the
// whole block and synchronise with the block barrier; BAR > 0: they are a subset of the block's warps
// and synchronise on named barrier BAR (the rest of the block runs on independently).
template <int NT, int BAR>
__device__ __forceinline__ void topk_sync()
{
    if (BAR == 0) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"n"(BAR), "n"(NT) : "memory");
}

// larger float <=> larger key; -0 and +0 map to the same key
__device__ __forceinline__ unsigned topk_order_key(float f)
{
    unsigned u = __float_as_uint(f);
    if (u == 0x80000000u) u = 0u;
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ int topk_warp_scan(int v, int lane)   // inclusive
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Exclusive prefix sum of `v` over the NT threads of the block; also returns the total.  One word
// written per warp, one barrier, then every warp adds up the totals of the warps before it with a
// warp-reduce instruction.  `warp_sums` (32 words) must not be in use by a scan that some thread
// of the block may not have left yet: alternate between two slots.
template <int NT, int BAR>
__device__ __forceinline__ int topk_block_scan(int tid, int v, int *warp_sums, int &total)
{
    constexpr int kWarps = NT / 32;
    const int lane = tid & 31, warp = tid >> 5;
    const int incl = topk_warp_scan(v, lane);
    if (lane == 31) warp_sums[warp] = incl;
    topk_sync<NT, BAR>();
    const int wt = lane < kWarps ? warp_sums[lane] : 0;
    total = __reduce_add_sync(0xffffffffu, wt);
    return __reduce_add_sync(0xffffffffu, lane < warp ? wt : 0) + incl - v;
}

// The first pass where scores are token scores' means: a unit's token scores sum to at most its number of observation
// rows R, so they lie around R / n.  512 bins of a sixteenth of an octave cover 12 octaves below and 20 above;
// what lies outside falls into the outer bins, and a threshold there is found the general way.
constexpr int kHintShift = 19;                // bits of a key below a bin: 4 bits of mantissa above them
__device__ __forceinline__ int topk_hint(int rows, int n)
{
    return (int)(topk_order_key((float)rows / (float)n) >> kHintShift) - 12 * 16;
}

// window scores in memory, read through L2: those written by other blocks of the same grid are seen once the caller
// has synchronised with them
struct WrittenScores {
    static constexpr bool kWaits = false;
    const float *scores;
    int hint;            // topk_hint(), or negative: nothing is known about the scores' range
    template <int N>
    __device__ __forceinline__ void keys(unsigned (&key)[N], int lo, int hi) const
    {
#pragma unroll
        for (int e = 0; e < N; ++e) key[e] = lo + e < hi ? topk_order_key(__ldcg(scores + lo + e)) : 0u;
    }
    __device__ __forceinline__ void wait(int, int) const {}
    __device__ __forceinline__ bool gave_up() const { return false; }
    __device__ __forceinline__ unsigned key(int w) const { return topk_order_key(__ldcg(scores + w)); }
};

// The histogram's bin, counted from the top one down, in which the number of keys reaches `remaining`: the thread
// that holds it calls found(bin, what is left of `remaining` inside it, its keys).  Every warp of the first sixteen
// searches a part.  Leaves the histogram zero; begins behind a barrier and ends with one.
template <int NT, int BAR, typename F>
__device__ __forceinline__ void topk_find_bin(int tid, TopkSmem &sm, int remaining, F found)
{
    constexpr int kWarps = NT / 32, kParts = kWarps < 16 ? kWarps : 16, kPer = kTopkBins / (32 * kParts);
    static_assert(kPer * 32 * kParts == kTopkBins, "the warps share the bins evenly");
    const int lane = tid & 31, warp = tid >> 5;
    const int bin0 = (warp * 32 + lane) * kPer;
    int c[kPer], mine = 0;
    if (warp < kParts) {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            c[i] = sm.hist[bin0 + i];
            sm.hist[bin0 + i] = 0;
            mine += c[i];
        }
    }
    int upto = mine;                          // keys in this lane's bins and in higher lanes' bins of the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_down_sync(0xffffffffu, upto, o);
        if (lane + o < 32) upto += t;
    }
    if (lane == 0) sm.warp_sums[1][warp] = upto;
    topk_sync<NT, BAR>();
    int above = __reduce_add_sync(0xffffffffu, lane > warp && lane < kParts ? sm.warp_sums[1][lane] : 0) + upto - mine;
    if (warp < kParts && above < remaining && remaining <= above + mine) {
#pragma unroll
        for (int i = kPer - 1; i >= 0; --i) {
            if (above < remaining && remaining <= above + c[i]) found(bin0 + i, remaining - above, c[i]);
            above += c[i];
        }
    }
    topk_sync<NT, BAR>();
}

// All NT threads of the block call this.  `src.keys(key, lo, hi)` gives the order keys of the unit's windows lo .. hi - 1 (at
// most as many as `key` holds) once they are there; for longer lists `src.wait(lo, hi)` waits for them, `src.gave_up()` tells
// whether a wait of the block's has expired (kWaits: one may) and `src.key(w)` reads one. `out` receives k ascending indices followed by -1 up to k_max.
// Thread t owns the windows [t*E, (t+1)*E), E = ceil(kw / NT).  With E <= REGS (4, 8 or 16) the keys
// are read once and stay in registers through the radix passes and the compaction (one trip to L2
// instead of several); REGS = 0: longer lists are re-read.
template <int NT, int REGS, int BAR, typename Src>
__device__ __forceinline__ void select_topk_impl(int tid, TopkSmem &sm, const Src &src, int kw, int k, int *out,
                                                 int *kept_len_out, int n, int alpha, int omega, int obs_rows)
{
    constexpr int kWarps = NT / 32;
    static_assert(NT % 32 == 0 && NT >= kTopkDirect, "block size");
    const int lane = tid & 31, warp = tid >> 5;
    const int E = (kw + NT - 1) / NT;
    const int w_lo = min(kw, tid * E), w_hi = min(kw, w_lo + E);
    // (the words below are set before the keys are waited for)
    if (tid == 0) sm.n_cand = 0;
    for (int x = tid; x < kTopkBins; x += NT) sm.hist[x] = 0;
    topk_sync<NT, BAR>();
    constexpr bool IN_REGS = REGS > 0;
    constexpr int kTopkRegs = IN_REGS ? REGS : 1;
    unsigned keys[kTopkRegs];
    if (IN_REGS) src.keys(keys, w_lo, w_hi);
    else {
        src.wait(w_lo, w_hi);
        // What is still missing after a wait that expired may come while the passes below read the list, and they write by
        // counts that hold for an unchanged list alone: no selection then.
        if (Src::kWaits) {
            topk_sync<NT, BAR>();
            if (src.gave_up()) return;
        }
    }
    auto key_at = [&](int e) -> unsigned { return IN_REGS ? keys[e] : src.key(w_lo + e); };
    // runs f(e, key) over the thread's own keys
    auto for_own = [&](auto f) {
        if (IN_REGS) {
#pragma unroll
            for (int e = 0; e < kTopkRegs; ++e)
                if (w_lo + e < w_hi) f(e, keys[e]);
        } else {
            for (int e = 0; w_lo + e < w_hi; ++e) f(e, key_at(e));
        }
    };

    // ---- radix select: key of the k-th largest score --------------------------------
    // Bits of a key are resolved 9 at a time from the top until at most kTopkDirect candidates share the prefix; those
    // are ranked against each other directly.
    unsigned kmin = 0u, mask = 0u;    // keys are taken relative to kmin; mask: the bits that are resolved
    int top = 0;                      // ... which are [top, 32)
    bool known = false;
    if (src.hint >= 0) {
        for_own([&](int, unsigned key) {
            atomicAdd(&sm.hist[min(max((int)(key >> kHintShift) - src.hint, 0), kTopkBins - 1)], 1);
        });
        topk_sync<NT, BAR>();
        topk_find_bin<NT, BAR>(tid, sm, k, [&](int bin, int rest, int count) {
            sm.prefix = (unsigned)(src.hint + bin) << kHintShift;
            sm.remaining = rest;
            sm.cand_total = bin == 0 || bin == kTopkBins - 1 ? -1 : count;
        });
        known = sm.cand_total >= 0;
        mask = ~0u << kHintShift;
        top = kHintShift;
    }
    if (!known) {
        // Nothing known: relative to the smallest key, only the bits in which the largest differs from it (scores
        // share sign and most of the exponent: typically one pass).
        unsigned lo = 0xffffffffu, hi = 0u;
        for_own([&](int, unsigned key) {
            lo = min(lo, key);
            hi = max(hi, key);
        });
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_max_sync(0xffffffffu, hi);
        if (lane == 0) {
            sm.warp_min[warp] = lo;
            sm.warp_max[warp] = hi;
        }
        topk_sync<NT, BAR>();
        if (tid == 0) {
            sm.prefix = 0u;
            sm.remaining = k;
            sm.cand_total = kw;
        }
        kmin = __reduce_min_sync(0xffffffffu, lane < kWarps ? sm.warp_min[lane] : 0xffffffffu);
        const unsigned kmax = __reduce_max_sync(0xffffffffu, lane < kWarps ? sm.warp_max[lane] : 0u);
        mask = 0u;
        top = 32 - __clz(kmax - kmin);        // 0 when all keys are equal
        topk_sync<NT, BAR>();
    }
#pragma unroll 1
    while (top > 0) {
        const unsigned prefix = sm.prefix;
        const int remaining = sm.remaining;
        if (sm.cand_total <= kTopkDirect) {
            // direct finish: the candidates are collected, in any order, and each is ranked against the others
            for_own([&](int, unsigned key) {
                const unsigned rk = key - kmin;
                if ((rk & mask) == prefix) sm.cand[atomicAdd(&sm.n_cand, 1)] = rk;
            });
            topk_sync<NT, BAR>();
            // a warp per candidate, two of the others per lane: a handful of votes instead of a loop over all of them
            // (which took 1 us)
            static_assert(kTopkDirect == 64, "two candidates per lane");
            const int n_cand = sm.n_cand;
            const unsigned o0 = sm.cand[lane], o1 = sm.cand[lane + 32];
            const bool in0 = lane < n_cand, in1 = lane + 32 < n_cand;
            for (int c = warp; c < n_cand; c += kWarps) {
                const unsigned my = sm.cand[c];
                const int gt = __popc(__ballot_sync(0xffffffffu, in0 && o0 > my)) + __popc(__ballot_sync(0xffffffffu, in1 && o1 > my));
                const int eq = __popc(__ballot_sync(0xffffffffu, in0 && o0 == my)) + __popc(__ballot_sync(0xffffffffu, in1 && o1 == my));
                if (lane == 0 && gt < remaining && remaining <= gt + eq) {   // all that get here write the same values
                    sm.prefix = my;
                    sm.remaining = remaining - gt;
                }
            }
            topk_sync<NT, BAR>();
            break;
        }
        const int low = top > kTopkDigit ? top - kTopkDigit : 0;
        const unsigned digit_mask = (1u << (top - low)) - 1u;
        for_own([&](int, unsigned key) {
            const unsigned rk = key - kmin;
            if ((rk & mask) == prefix) atomicAdd(&sm.hist[(rk >> low) & digit_mask], 1);
        });
        topk_sync<NT, BAR>();
        topk_find_bin<NT, BAR>(tid, sm, remaining, [&](int bin, int rest, int count) {
            sm.prefix = prefix | ((unsigned)bin << low);
            sm.remaining = rest;   // after the last pass: how many keys equal to the threshold are taken
            sm.cand_total = count;
        });
        mask |= digit_mask << low;
        top = low;
    }
    const unsigned thr = sm.prefix + kmin;
    const int need_eq = sm.remaining;

    // ---- ordered compaction ----------------------------------------------------------
    int n_eq = 0, n_gt = 0;
    if (IN_REGS) {
#pragma unroll
        for (int e = 0; e < kTopkRegs; ++e)
            if (w_lo + e < w_hi) {
                n_eq += keys[e] == thr;
                n_gt += keys[e] > thr;
            }
    } else {
        for (int e = 0; w_lo + e < w_hi; ++e) {
            const unsigned key = key_at(e);
            n_eq += key == thr;
            n_gt += key > thr;
        }
    }
    int eq_rank, pos;   // threshold keys before this thread; output position of its first selected window
    if (IN_REGS) {
        // at most NT * 16 < 2^15 windows: both counts travel through one scan
        int total;
        const int both = topk_block_scan<NT, BAR>(tid, (n_eq << 16) | n_gt, sm.warp_sums[0], total);
        eq_rank = both >> 16;
        pos = (both & 0xffff) + (eq_rank < need_eq ? eq_rank : need_eq);
    } else {
        int eq_total, sel_total;
        eq_rank = topk_block_scan<NT, BAR>(tid, n_eq, sm.warp_sums[0], eq_total);
        int n_eq_taken = need_eq - eq_rank;
        n_eq_taken = n_eq_taken < 0 ? 0 : (n_eq_taken > n_eq ? n_eq : n_eq_taken);
        pos = topk_block_scan<NT, BAR>(tid, n_gt + n_eq_taken, sm.warp_sums[1], sel_total);
    }
    auto emit = [&](int e, unsigned key) {
        bool sel = key > thr;
        if (key == thr) {
            sel = eq_rank < need_eq;
            ++eq_rank;
        }
        if (sel) {
            out[pos++] = w_lo + e;
        }
        if (w_lo + e == kw - 1) {
            const int n_r = n - alpha;
            const int last_size = n_r - (kw - 1) * omega;     // real size of the last window
            *kept_len_out = k * omega - (sel ? omega - last_size : 0) + obs_rows;
        }
    };
    if (IN_REGS) {
#pragma unroll
        for (int e = 0; e < kTopkRegs; ++e)
            if (w_lo + e < w_hi) emit(e, keys[e]);
    } else {
        for (int e = 0; w_lo + e < w_hi; ++e) emit(e, key_at(e));
    }
}

template <int NT, int BAR = 0, typename Src>
__device__ void select_topk_block(int tid, TopkSmem &sm, const Src &src, int kw, int k, int k_max, int *out,
                                  int *kept_len_out, int n, int alpha, int omega)
{
    static_assert(NT % 32 == 0 && NT <= 1024, "block size");
    for (int x = (k > 0 ? k : 0) + tid; x < k_max; x += NT) out[x] = -1;
    const int obs_rows = n < alpha ? n : alpha;
    if (k <= 0) {
        if (tid == 0) *kept_len_out = obs_rows;
        return;
    }
    // Re-reading the list in every pass is a trip to L2 per window and pass: 28 units of 5,945 windows, whole group 311 us
    // against 272 with up to sixteen in registers.
    const int per_thread = (kw + NT - 1) / NT;
    if (per_thread <= 4)
        select_topk_impl<NT, 4, BAR>(tid, sm, src, kw, k, out, kept_len_out, n, alpha, omega, obs_rows);
    else if (per_thread <= 8)
        select_topk_impl<NT, 8, BAR>(tid, sm, src, kw, k, out, kept_len_out, n, alpha, omega, obs_rows);
    else if (per_thread <= 16)
        select_topk_impl<NT, 16, BAR>(tid, sm, src, kw, k, out, kept_len_out, n, alpha, omega, obs_rows);
    else
        select_topk_impl<NT, 0, BAR>(tid, sm, src, kw, k, out, kept_len_out, n, alpha, omega, obs_rows);
}

}  // namespace wkv
