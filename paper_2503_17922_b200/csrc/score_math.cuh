// Device-side pieces shared by the score kernels: the per-element work of the tensor-core kernels' two sweeps
// (Eq. 1's online statistics, Eq. 2's normalised sum), Eq. 4's pooling of one window, and the hand-over between thread
// blocks: published words, acquire / release accesses, bounded waits.
#pragma once

#include "tc_common.cuh"
#include "topk_block.cuh"
#include "wkv_internal.cuh"

namespace wkv {
namespace {

using namespace tc;

__device__ __forceinline__ int ld_acquire_gpu(const int *p)
{
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_gpu_add(int *p, int v)
{
    asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// one thread: polls until the word has reached `target`; false once the block has given up
// (`sleep_ns` > 0: the thread sleeps between looks, for waits that are expected to be long)
__device__ __forceinline__ bool poll_until_at_least(const int *word, int target, volatile int *abort_flag,
                                                    unsigned sleep_ns = 0)
{
    unsigned long long t0 = 0;
    for (uint32_t spin = 1; ld_acquire_gpu(word) < target; ++spin) {
        if (*abort_flag) return false;
        if (sleep_ns) __nanosleep(sleep_ns);
        if ((spin & 255u) == 0u) {
            const unsigned long long now = global_timer_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > 2 * kWaitLimitNs) {
                *abort_flag = 1;
                return false;
            }
        }
    }
    return true;
}

// A published word: value and tag travel together in one 16-byte access (a .b128 access is performed as a whole), so a
// reader that finds the tag has the value, without a fence on either side.
struct __align__(16) StatEntry {
    unsigned long long value, tag;
};
__device__ __forceinline__ void publish_entry(StatEntry *p, unsigned long long value, unsigned long long tag)
{
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p), "l"(value), "l"(tag)
                 : "memory");
}
__device__ __forceinline__ StatEntry read_entry(const StatEntry *p)
{
    StatEntry e;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}" : "=l"(e.value), "=l"(e.tag)
                 : "l"(p)
                 : "memory");
    return e;
}
// Up to N words that are or will be published: word u is at p + u * step, those in the mask `wanted` count.  All that
// are still missing are looked at together, so that each look is one trip.  Bounded like every wait.
template <int N>
__device__ __forceinline__ void wait_entries(const StatEntry *p, size_t step, unsigned wanted, unsigned long long tag,
                                             StatEntry (&e)[N], volatile int *abort_flag)
{
    unsigned long long t0 = 0;
    for (uint32_t spin = 1;; ++spin) {
#pragma unroll
        for (int u = 0; u < N; ++u)
            if (wanted >> u & 1u) e[u] = read_entry(p + u * step);
#pragma unroll
        for (int u = 0; u < N; ++u)
            if ((wanted >> u & 1u) && e[u].tag == tag) wanted &= ~(1u << u);
        if (!wanted || *abort_flag) return;
        if ((spin & 255u) == 0u) {
            const unsigned long long now = global_timer_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > 2 * kWaitLimitNs) {
                *abort_flag = 1;
                return;
            }
        }
    }
}
// The same for a caller that can do without the words: it looks `looks` times (each is a trip to L2, 0.6 us and more), then raises
// the flag, which ends the search of all that share it.
template <int N>
__device__ __forceinline__ void look_for_entries(const StatEntry *p, size_t step, unsigned wanted, unsigned long long tag,
                                                 StatEntry (&e)[N], volatile int *late_flag, int looks)
{
    for (;;) {
#pragma unroll
        for (int u = 0; u < N; ++u)
            if (wanted >> u & 1u) e[u] = read_entry(p + u * step);
#pragma unroll
        for (int u = 0; u < N; ++u)
            if ((wanted >> u & 1u) && e[u].tag == tag) wanted &= ~(1u << u);
        if (!wanted || *late_flag) return;
        if (--looks <= 0) {
            *late_flag = 1;
            return;
        }
    }
}

// Launches on a workspace, counted so that each has a tag of its own.  Every block reads the count before it counts
// itself, and the launch's last block to do so raises it: the blocks of one launch agree on it, the next one's
// find it changed.
struct LaunchCount {
    unsigned blocks;
    unsigned stood_in;      // for diagnosis: chunks whose statistics a block has taken because their block's had not come,
    unsigned left_over;     // and selections left to the block that counts itself last (score_tc.cu)
    unsigned unused;
    unsigned long long launches;
};
// The tag's upper bits make its upper word a NaN with a payload that no arithmetic produces, so that neither numbers
// nor counters that another shape has left at the place of a tag equal one.
constexpr unsigned long long kTagBits = 0xffb5000000000000ull;
__device__ __forceinline__ unsigned long long launches_so_far(const LaunchCount *c)
{
    unsigned long long n;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(n) : "l"(&c->launches) : "memory");
    return n;
}
__device__ __forceinline__ unsigned long long launch_tag(unsigned long long launches, unsigned salt)
{
    return kTagBits | (unsigned long long)(salt & 0xffu) << 40 | ((launches + 1) & 0xffffffffffull);
}
__device__ __forceinline__ unsigned long long launch_of(unsigned long long tag) { return tag & 0xffffffffffull; }
// one thread of each of the launch's `blocks` blocks, `launch` being one more than what it has read
__device__ __forceinline__ void count_launch(LaunchCount *c, unsigned long long launch, unsigned blocks)
{
    if (atomicInc(&c->blocks, blocks - 1) == blocks - 1) c->launches = launch;
}

// The selection reads the published window scores, waiting for those that are still to come: LOOK words at a time.
// PATIENT: until they come or the wait expires, else for `looks` looks.
template <int LOOK, bool PATIENT = true>
struct PublishedScores {
    static constexpr bool kWaits = true;
    const StatEntry *entries;
    unsigned long long tag;
    volatile int *abort_flag;
    int hint;
    int looks = 0;
    template <int N>
    __device__ __forceinline__ void keys(unsigned (&key)[N], int lo, int hi) const
    {
        constexpr int kLook = N < LOOK ? N : LOOK;
#pragma unroll
        for (int e0 = 0; e0 < N; e0 += kLook) {
            StatEntry v[kLook];
            const int left = hi - lo - e0;
            const unsigned wanted = left >= kLook ? (1u << kLook) - 1u : left > 0 ? (1u << left) - 1u : 0u;
            if (PATIENT) wait_entries<kLook>(entries + lo + e0, 1, wanted, tag, v, abort_flag);
            else look_for_entries<kLook>(entries + lo + e0, 1, wanted, tag, v, abort_flag, looks);
#pragma unroll
            for (int e = 0; e < kLook; ++e) key[e0 + e] = e < left ? topk_order_key(__uint_as_float((unsigned)v[e].value)) : 0u;
        }
    }
    __device__ __forceinline__ void wait(int lo, int hi) const
    {
        unsigned unused[LOOK];
        for (int w = lo; w < hi; w += LOOK) keys(unused, w, min(hi, w + LOOK));
    }
    // behind a barrier of all that wait
    __device__ __forceinline__ bool gave_up() const { return *abort_flag != 0; }
    __device__ __forceinline__ unsigned key(int w) const
    {
        return topk_order_key(__ldcg(reinterpret_cast<const float *>(&entries[w].value)));
    }
};

// Two fp32 numbers in one register pair: the packed instructions round each half as the plain ones do and take one issue slot
// for the two.
__device__ __forceinline__ unsigned long long pair_of(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 halves_of(unsigned long long p)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(p));
    return r;
}
__device__ __forceinline__ unsigned long long fma_pair(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ unsigned long long add_pair(unsigned long long a, unsigned long long b)
{
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long exp2_pair(unsigned long long x)
{
    const float2 h = halves_of(x);
    return pair_of(fast_exp2(h.x), fast_exp2(h.y));
}

// acc + 2^x on the FMA pipe: 2^x = 2^t * 2^f with t the nearest integer, and 2^f by a polynomial of degree six
// (a Remez fit of the relative error on [-1/2, 1/2]).  With its coefficients in fp32 it is off by 1.6e-8 at most, evaluated in
// fp32 by 7.9e-8.  From t = -127 on the power of two is zero, so that below -126.5 nothing is added, and at t = 128 it is infinite, so that beyond
// 127.5 the result is; a NaN stays one.  AT_MOST_ZERO: x is not above zero (but for its rounding).
template <bool AT_MOST_ZERO>
__device__ __forceinline__ void add_exp2_fma(unsigned long long &acc, unsigned long long x2)
{
    float2 x = halves_of(x2);
    asm("max.NaN.f32 %0, %0, 0fC2FE0000;" : "+f"(x.x));      // -127
    asm("max.NaN.f32 %0, %0, 0fC2FE0000;" : "+f"(x.y));
    if (!AT_MOST_ZERO) {
        asm("min.NaN.f32 %0, %0, 0f43000000;" : "+f"(x.x));      // 128
        asm("min.NaN.f32 %0, %0, 0f43000000;" : "+f"(x.y));
    }
    auto both = [](float v) { return pair_of(v, v); };
    x2 = pair_of(x.x, x.y);
    const unsigned long long shifted = add_pair(x2, both(12582912.f));                  // 1.5 * 2^23: the integer is in the low bits
    const unsigned long long f = fma_pair(add_pair(shifted, both(-12582912.f)), both(-1.f), x2);
    unsigned long long p = both(1.5345812e-4f);
    p = fma_pair(p, f, both(1.3399931e-3f));
    p = fma_pair(p, f, both(9.618489e-3f));
    p = fma_pair(p, f, both(5.5503286e-2f));
    p = fma_pair(p, f, both(2.4022646e-1f));
    p = fma_pair(p, f, both(6.931472e-1f));
    p = fma_pair(p, f, both(1.f));
    const float2 t = halves_of(shifted);
    acc = fma_pair(p, pair_of(__int_as_float((__float_as_int(t.x) << 23) + 0x3f800000), __int_as_float((__float_as_int(t.y) << 23) + 0x3f800000)), acc);
}
constexpr int kFmaEveryStats = 8, kFmaEveryScore = 16;      // two of so many neighbouring exponentials
// FMA_SHARE: one exponential in four of the statistics sweep and one in eight of the scoring sweep go that way, two neighbours as a
// pair.  The special-function pipe is what bounds the sweeps where keys come fast enough, and the FMA pipe is half idle.  Whole
// pass, us, plain instructions with one in eight in launches of one wave only / packed, none / one in eight / one in four: 4
// layers of 8 heads x 16,384 keys, 128 rows, 36.7 / 37.7 / 36.2 / 36.0; 4 ragged sequences of 16-32 K keys, 128 rows, 176 / 179 /
// 175 / 176; of 20-40 K, 256 rows, 343 / 348 / 339 / 335; 8 of 32-64 K, 256 rows, 1,005 / 1,006 / 981 / 992.
// The two shares differ for precision's sake: ex2.approx lies 5e-8 too low on average (1.6e-8 near zero), the polynomial has no bias,
// and the accumulators' rounding makes scores 1-2e-7 too high; a normaliser with more of the polynomial's terms makes up for the
// terms of the score.  Window scores against 64 bits, rms over 24 inputs, before and now: 128 rows 3.01 and 2.99e-7, 256 rows 2.59 and
// 2.57e-7, in several waves 2.493 and 2.490e-7, 2.049 and 2.045e-7 (one in eight of both there: 2.510 and 2.062e-7).

// ---------------------------------------------------------------------------------------------
// per-element work of the two sweeps
// ---------------------------------------------------------------------------------------------
// sweep 1: online-softmax update of one row with 32 more logits (raw dot products; c = log2(e)/sqrt(d))
template <bool FMA_SHARE = false>
__device__ __forceinline__ void stats_update(float (&v)[32], bool fast, int jb, int limit, float c, float &m,
                                             float &l)
{
    if (!fast) {
#pragma unroll
        for (int x = 0; x < 32; ++x)
            if (jb + x > limit) v[x] = -INFINITY;
    }
    float g0 = fmaxf(v[0], v[1]), g1 = fmaxf(v[2], v[3]);
#pragma unroll
    for (int x = 4; x < 32; x += 4) {
        g0 = fmaxf(g0, fmaxf(v[x], v[x + 1]));
        g1 = fmaxf(g1, fmaxf(v[x + 2], v[x + 3]));
    }
    const float m_new = fmaxf(m, fmaxf(g0, g1));
    if (m_new > -INFINITY) {
        const float mc = m_new * c;
        const unsigned long long c2 = pair_of(c, c), mc2 = pair_of(-mc, -mc);
        unsigned long long a01 = 0ull, a23 = 0ull;
#pragma unroll
        for (int x = 0; x < 32; x += 4) {
            a01 = add_pair(a01, exp2_pair(fma_pair(pair_of(v[x], v[x + 1]), c2, mc2)));
            const unsigned long long y = fma_pair(pair_of(v[x + 2], v[x + 3]), c2, mc2);
            if (FMA_SHARE && x % kFmaEveryStats == 0) add_exp2_fma<true>(a23, y);
            else a23 = add_pair(a23, exp2_pair(y));
        }
        const float2 s01 = halves_of(a01), s23 = halves_of(a23);
        const float add = (s01.x + s01.y) + (s23.x + s23.y);
        l = m_new == m ? l + add : l * fast_exp2((m - m_new) * c) + add;
        m = m_new;
    }
}
// sweep 2: adds exp2(x*c - lse2) of 32 (or 16) rows to the four partial sums of a key
template <int N, bool FMA_SHARE = false>
__device__ __forceinline__ void score_accumulate(const float (&v)[N], const float *nl_base, float c, unsigned long long &a01,
                                                 unsigned long long &a23)
{
    const unsigned long long c2 = pair_of(c, c);
#pragma unroll
    for (int x = 0; x < N; x += 4) {
        const ulonglong2 nl = *reinterpret_cast<const ulonglong2 *>(nl_base + x);
        a01 = add_pair(a01, exp2_pair(fma_pair(pair_of(v[x], v[x + 1]), c2, nl.x)));
        const unsigned long long y = fma_pair(pair_of(v[x + 2], v[x + 3]), c2, nl.y);
        if (FMA_SHARE && x % kFmaEveryScore == 0) add_exp2_fma<false>(a23, y);   // (a caller's normaliser may be too low)
        else a23 = add_pair(a23, exp2_pair(y));
    }
}

// Eq. 4 for one window of compile-time length (a power of two) by one thread: a bitonic sorting
// network in registers (every compare-exchange of a stage is independent of the others, so the
// thread is not latency-bound), then the p largest are summed in descending order.  Positions
// beyond `size` (ragged last window) hold -inf and sort to the end.  `w` is 16-byte aligned shared memory that holds
// omega values.
template <int omega>
__device__ __forceinline__ float pool_window_sorted(const float *w, int size, int p, int lane)
{
    // Neighbouring lanes take neighbouring windows, so a lane starts with another 16-byte piece of its window than the
    // lanes it would share banks with; the network does not care in which register an element starts.
    constexpr int kPieces = omega / 4;
    const int turn = (lane * kPieces) >> 3;
    float v[omega];
#pragma unroll
    for (int i = 0; i < kPieces; ++i) {
        const int c = (i + turn) % kPieces;
        const float4 x = *reinterpret_cast<const float4 *>(w + 4 * c);
        v[4 * i] = 4 * c < size ? x.x : -INFINITY;
        v[4 * i + 1] = 4 * c + 1 < size ? x.y : -INFINITY;
        v[4 * i + 2] = 4 * c + 2 < size ? x.z : -INFINITY;
        v[4 * i + 3] = 4 * c + 3 < size ? x.w : -INFINITY;
    }
#pragma unroll
    for (int k = 2; k <= omega; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1)
#pragma unroll
            for (int i = 0; i < omega; ++i) {
                const int l = i ^ j;
                if (l > i) {
                    const float hi = fmaxf(v[i], v[l]), lo = fminf(v[i], v[l]);
                    const bool descending = (i & k) == 0;
                    v[i] = descending ? hi : lo;
                    v[l] = descending ? lo : hi;
                }
            }
    const int p_eff = p < size ? p : size;
    float acc = 0.f;
#pragma unroll
    for (int x = 0; x < omega; ++x) acc += x < p_eff ? v[x] : 0.f;
    return acc / (float)p_eff;
}

// Eq. 4 for one window of 64 or 128 tokens by one warp: lane l holds elements l, l + 32, ... in
// registers; a bitonic sorting network over (register, lane) orders them descending (partners 32 or
// more apart are registers of the same lane, closer ones are exchanged by shuffle), then the p largest
// are summed: per lane in ascending rank, across lanes by a fixed butterfly, so the result is the same
// from run to run.  Positions beyond `size` hold -inf.  Every lane returns the window score.
template <int omega>
__device__ __forceinline__ float pool_window_warp(const float *w, int size, int p, int lane)
{
    constexpr int NR = omega / 32;
    static_assert(omega == 64 || omega == 128, "window length");
    float v[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) v[r] = r * 32 + lane < size ? w[r * 32 + lane] : -INFINITY;
#pragma unroll
    for (int k = 2; k <= omega; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= 32) {
                const int jj = j >> 5;
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    if ((r & jj) == 0) {
                        const float hi = fmaxf(v[r], v[r | jj]), lo = fminf(v[r], v[r | jj]);
                        const bool descending = ((r * 32 + lane) & k) == 0;
                        v[r] = descending ? hi : lo;
                        v[r | jj] = descending ? lo : hi;
                    }
                }
            } else {
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    const float other = __shfl_xor_sync(0xffffffffu, v[r], j);
                    const bool lower = (lane & j) == 0;
                    const bool descending = ((r * 32 + lane) & k) == 0;
                    v[r] = (lower == descending) ? fmaxf(v[r], other) : fminf(v[r], other);
                }
            }
        }
    }
    const int p_eff = p < size ? p : size;
    float acc = 0.f;
#pragma unroll
    for (int r = 0; r < NR; ++r) acc += (r * 32 + lane < p_eff) ? v[r] : 0.f;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc / (float)p_eff;
}

}  // namespace
}  // namespace wkv
