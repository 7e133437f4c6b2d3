// Steps 4 and 5a from ranked lists, in one launch.
//
// Pivot i's picks are among the Q_i = q_0 + ... + q_i smallest (dup, index) pairs of its row (dart_staged.cuh), whatever the
// other pivots take.  One CTA per (sample, pivot) puts those Q_i into order; the CTA of a sample that finishes last takes the
// pivots' turns over the ranked lists, in rank order, and writes the packed index list.  What bounded the other forms:
//   - ordering: a radix select and a sort are some twenty block-wide steps (16 us for 128 lists of 312 out of 2880 values).
//     Here: the row stays in registers; a threshold guessed from its smallest value and its mean lets through a few more
//     entries than the list needs (counted, and guessed again until it does: 1 to 3 counts); those alone go into a histogram of
//     equal bins, its prefix sums are the bins' places, and every entry counts the smaller ones among the few that share its bin.
//     (With the row in shared memory, two passes over all of it and bins over [min, 2 mean - min] one sample took 1 to 4 us more;
//     a queue of the entries below the threshold, so that only they meet the atomics, was no faster at 32768 rows (402 us for
//     389) and slower where half of a row is kept: 190 for 146.)
//   - the turns: a walk 32 entries at a time, one dependent vote after the other (1.4 us per turn).  Here a lane holds eight
//     consecutive entries (16 bytes), their eight flags are read at once, and four votes over the bits of the lanes' counts
//     give every lane its rank among 256 entries: 0.45 us per turn.
// Measured (us, before: the bands or sorted lists): 1 x 2880 tokens, 8 pivots 39 -> 19; 4 x 4608, 32 pivots 70 -> 29; 8 x 1500
// keeping half 60 -> 18; 256 x 2880, 8 pivots 60 -> 38, 128 pivots 488 -> 389.  Of the last, reading the rows is 80 (at the
// memory's rate it would be 57), minimum and mean 25, the counts 30, the atomics' two passes 100, the places 40; what remains is
// the last samples' turns.  For one sample all of it is a chain of short steps.
// A list of nearly all tokens cannot wait for a guess that lets all of them through: once few are left the bins reach to the largest
// value (8 x 2880 keeping everything, 8 pivots 237 us -> 27; 256 x 576 125 -> 31).
// Rows whose values the bins do not separate (many equal values, a value that is not finite) are ranked by an exact radix
// select, then by counting or, as that grows with the square of the length, a sort (8 x 2880 equal rows, 8 pivots, keeping half
// 82 us -> 50, everything 238 -> 70; 256 x 1000, 64 pivots, half 533 -> 470).  The result equals retain_kernel's exactly.
//
// With independent pivots (DART_RULE_UNION) the lists are the q_i smallest and the last CTA only merges them.
#pragma once
#include "dart_staged.cuh"

namespace dart {

constexpr int kRankMaxThreads = 512;
constexpr int kRankMaxP = 1024;       // a context's most pivots
constexpr int kRankMaxVis = 16384;    // 512 threads x 8 x 4 values in registers
constexpr int kRankMaxList = 4096;    // longest list
constexpr int kRankLongList = 1000;   // lists that take more threads
constexpr uint32_t kRankMaxBin = 192; // entries of one bin that are ranked by counting
constexpr int kRankTries = 10;        // guesses at the threshold
constexpr int kRankMaxRest = 144;     // tokens beyond a threshold that a list of nearly all takes along
constexpr int kRankMaxCount = 1000;   // steps per thread up to which the exact route orders a list by counting (their number grows with the square)

// one flag per token and one more that is never free
__host__ __device__ inline size_t rank_flag_bytes(int n_vis) { return ((size_t)n_vis + 16) / 16 * 16; }
// values per thread in registers: 4 R
inline int rank_regs(int n_vis, int threads) { return n_vis <= 8 * threads ? 2 : n_vis <= 16 * threads ? 4 : n_vis <= 24 * threads ? 6 : 8; }
// shared memory of the ranking: the entries of the bins a list needs, 4 bins per thread, one bit per token
inline size_t rank_phase1_bytes(int n_vis, int m, int threads)
{
    return ((size_t)m + kRankMaxBin + 1) / 2 * 16 + (size_t)threads * 16 + ((size_t)n_vis + 127) / 128 * 16;
}
// places of the lists in the sample's part of the workspace, in entries of 16 bits: list i starts at rank_place(i), a multiple of 8
__host__ __device__ inline int rank_place(int i, int q, int r, bool each)
{
    // sum over k < i of (Q_k or q_k), every list rounded up by at most 7
    const int n = i < r ? i : r;
    const int sum = each ? i * q + n : q * (i * (i + 1) / 2) + n * (n + 1) / 2 + r * (i - n);
    return ((sum + 7) & ~7) + 8 * i;
}
__host__ __device__ inline int rank_length(int i, int q, int r, bool each) { return each ? q + (i < r ? 1 : 0) : quota_prefix(i, q, r); }

struct RankParams {
    const float *sim;          // [B][P][n_vis]
    const int32_t *pivot_idx;  // [B][P]
    uint16_t *lists;           // [B][sample_entries]
    size_t sample_entries;
    int *arrived;              // [B] lists written; zero on entry and on exit
    const int64_t *pos_in;
    int S, vis_offset, n_vis, P, n_keep, m; // m: the longest list (n_keep - P, or n_keep when pivots may be text tokens)
    int each;                  // 1: independent pivots (lists of q_i, merged)
    int stage_entries;         // entries of 16 bits per staging buffer of the turns
    int32_t *out_idx;          // quotas: [B][S_out]; independent pivots: unused
    int64_t *out_pos;
    uint8_t *keep_out;         // [B][n_vis]; NULL unless wanted
    int32_t *owner_out;        // [B][n_vis]; NULL unless wanted
    float *eps_out;            // [B][P]; NULL unless wanted
    int32_t *len_out;          // independent pivots: [B] packed length
    int32_t *row_word;         // [B][S_out] the kept vision rows' indices as the gather waits for them; -1 on entry, put back by the gather; may be NULL
    const int *status;
};

struct RankShared {
    SelectSmem sel;
    float red_lo[kRankMaxThreads / 32], red_hi[kRankMaxThreads / 32], red_sum[kRankMaxThreads / 32];
    uint32_t scan[kRankMaxThreads / 32];
    int32_t piv[kRankMaxP];
    uint32_t n_pivots, biggest, n_list, n_below[kRankTries], last;
};

constexpr int kRankStaticSmem = 8192;
static_assert(sizeof(RankShared) + 64 <= kRankStaticSmem, "static shared memory exceeds its reserve");

// Inclusive sum over the CTA's threads (two barriers)
__device__ __forceinline__ uint32_t cta_scan(uint32_t v, uint32_t *per_warp)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) per_warp[warp] = v;
    __syncthreads();
    uint32_t x = lane < nwarp && lane < warp ? per_warp[lane] : 0u;
    return v + __reduce_add_sync(0xffffffffu, x);
}

// n distinct entries of `list` in ascending order: a bitonic sort of any length (every comparison puts the smaller entry at the
// lower place, so that what is missing up to a power of two would never move).
__device__ __forceinline__ void cta_sort(unsigned long long *list, int n)
{
    auto order = [&](int i, int l) {
        if (l >= n) return;
        const unsigned long long x = list[i], y = list[l];
        if (x > y) list[i] = y, list[l] = x;
    };
    __syncthreads();
    for (int k = 1; k < n; k <<= 1) { // sorted runs of k to runs of 2 k
        const int pairs = (n + 2 * k - 1) / (2 * k) * k;
        for (int e = threadIdx.x; e < pairs; e += blockDim.x) {
            const int at = e & (k - 1), run = 2 * (e - at);
            order(run + at, run + 2 * k - 1 - at);
        }
        __syncthreads();
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int e = threadIdx.x; e < pairs; e += blockDim.x) {
                const int i = 2 * e - (e & (j - 1));
                order(i, i + j);
            }
            __syncthreads();
        }
    }
}

// A NaN that no arithmetic produces (its NaN is 0x7fffffff): below no threshold.  The row's values are results of arithmetic, and so
// are their negatives (flipping the sign bit of a NaN would give this one): one NaN makes their sum a NaN, and the row takes the
// exact route.
constexpr uint32_t kNotAToken = 0xffffffffu;

// A row's values into registers, or (kNegate) minus them if sign is -1
template <bool kNegate, int R>
__device__ __forceinline__ void load_row(const float *row, int n, float sign, float4 (&v)[R])
{
    const int t = threadIdx.x, T = blockDim.x;
    const float none = __uint_as_float(kNotAToken);
    auto value = [&](float x) { return kNegate ? fmaf(x, sign, 0.0f) : x; };
    if (((uintptr_t)row & 15u) == 0 && (n & 3) == 0) {
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const int j = 4 * (T * k + t);
            if (j < n) {
                const float4 f = *reinterpret_cast<const float4 *>(row + j);
                v[k] = make_float4(value(f.x), value(f.y), value(f.z), value(f.w));
            } else {
                v[k] = make_float4(none, none, none, none);
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const int j = 4 * (T * k + t);
            v[k].x = j < n ? value(row[j]) : none;
            v[k].y = j + 1 < n ? value(row[j + 1]) : none;
            v[k].z = j + 2 < n ? value(row[j + 2]) : none;
            v[k].w = j + 3 < n ? value(row[j + 3]) : none;
        }
    }
}

// The C smallest (value, index) pairs of a row of which n_in tokens take part, ranked, into out[0 .. C).  v: the thread's values (tokens
// 4 (T k + t) ...), tokens that do not take part and what lies behind the row as kNotAToken; list, hist (4 T words), skip (a bit per token that does not
// take part): shared memory.  flip: 0, or all ones if v holds the row's values with the opposite sign.
template <int R, bool kOutliers, typename Out>
__device__ __forceinline__ void rank_row(const float *row, uint32_t flip, const uint32_t *skip, const float4 (&v)[R], int n, int n_in, Out *out, int C,
                                         unsigned long long *list, uint32_t *hist, RankShared &sh)
{
    const int t = threadIdx.x, T = blockDim.x, lane = t & 31, warp = t >> 5, nwarp = T >> 5;
    // smallest and largest value, and the mean (NaN if a token's value is)
    float lo = __int_as_float(0x7f800000), hi = __int_as_float(0xff800000), sum = 0.f;
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const float f[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) lo = fminf(lo, f[e]), hi = fmaxf(hi, f[e]), sum += __float_as_uint(f[e]) != kNotAToken ? f[e] : 0.f;
    }
    lo = order_key_inv(__reduce_min_sync(0xffffffffu, order_key(lo)));
    hi = order_key_inv(__reduce_max_sync(0xffffffffu, order_key(hi)));
    sum = warp_sum(sum);
    if (lane == 0) sh.red_lo[warp] = lo, sh.red_hi[warp] = hi, sh.red_sum[warp] = sum;
    __syncthreads();
    lo = lane < nwarp ? sh.red_lo[lane] : __int_as_float(0x7f800000);
    hi = lane < nwarp ? sh.red_hi[lane] : hi;
    sum = lane < nwarp ? sh.red_sum[lane] : 0.f;
    // The first threshold: normal values whose smallest is at its expected place; the quantile by Tukey's approximation
    // 4.91 (u^0.14 - (1 - u)^0.14).  The next ones move on by what the count says.  Only the number of guesses depends on it.
    float low, mid; // the minimum and the mean above it
    int n_of = n;   // of how many values
    if constexpr (kOutliers) {
        // ... of the warp with the largest minimum: over all values a few outliers (a sample's largest norms) move them by more than
        // the others' spread, and 6 to 9 guesses were needed instead of 1 or 2.
        int n_warp = 0; // values of warp `lane`
#pragma unroll
        for (int k = 0; k < R; ++k) n_warp += min(max(n - 4 * (T * k + 32 * lane), 0), 128);
        const uint32_t high = lo < __int_as_float(0x7f800000) ? order_key(lo) : 0u;
        const int from = __ffs((int)__ballot_sync(0xffffffffu, high == __reduce_max_sync(0xffffffffu, high))) - 1;
        low = __shfl_sync(0xffffffffu, lo, from), mid = __shfl_sync(0xffffffffu, sum / (float)n_warp, from) - low;
        n_of = __shfl_sync(0xffffffffu, n_warp, from);
        if (__any_sync(0xffffffffu, sum != sum)) mid = __uint_as_float(kNotAToken);
        lo = order_key_inv(__reduce_min_sync(0xffffffffu, order_key(lo)));
    } else {
        low = lo = order_key_inv(__reduce_min_sync(0xffffffffu, order_key(lo)));
        mid = warp_sum(sum) / (float)n - low;
    }
    hi = order_key_inv(__reduce_max_sync(0xffffffffu, order_key(hi)));
    auto quantile = [](float u) { return 4.91f * (__powf(u, 0.14f) - __powf(1.0f - u, 0.14f)); };
    const float inv_n = 1.0f / (float)n, least = -quantile(fminf(0.5f / (float)n_of, 0.25f)), wanted = quantile(fminf((1.3f * (float)C + 40.f) * inv_n, 0.97f));
    float part = 1.0f + wanted / least, few = 0.f, many = 0.f, top = 0.f;
    bool has_few = false, has_many = false, exact = !(hi > lo) || !(hi - lo < 3.0e38f) || !(mid > 0.0f);
    int m = 0;
    reinterpret_cast<uint4 *>(hist)[t] = make_uint4(0, 0, 0, 0);
    for (int guess = 0; !exact; ++guess) {
        top = low + part * mid;
        if (!(top < hi)) top = hi;
        uint32_t c = 0;
#pragma unroll
        for (int k = 0; k < R; ++k) c += (v[k].x <= top) + (v[k].y <= top) + (v[k].z <= top) + (v[k].w <= top);
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) atomicAdd(&sh.n_below[guess], c);
        __syncthreads();
        m = (int)sh.n_below[guess];
        if (m >= C && m <= 3 * C + 256) break;
        if (m < C && n_in - m <= kRankMaxRest) { // the list takes nearly all tokens: let all of them through
            m = n_in, top = hi;
            break;
        }
        exact = guess + 1 == kRankTries || (m < C && top == hi);
        (m < C ? few : many) = part;
        (m < C ? has_few : has_many) = true;
        part += (wanted - quantile(fminf(((float)m + 0.5f) * inv_n, 0.97f))) / least;
        if (has_few && has_many && !(part > 0.9f * few + 0.1f * many && part < 0.1f * few + 0.9f * many)) part = 0.5f * (few + many);
    }
    // bins: the low bits of 2^23 + (x - base) scale, never below 0 or above 4 T - 1; outliers go to the first one
    const float base = kOutliers && low - lo > top - low && top > low ? low : lo, scale = ((float)(4 * T) - 1.0f) / (top - base);
    if (!exact && scale < 3.0e38f) {
        auto bin_of = [&](float x) { return (int)(__float_as_uint(fmaf(kOutliers ? fmaxf(x - base, 0.f) : x - base, scale, 8388608.0f)) - 0x4b000000u); };
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const float f[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (f[e] <= top) atomicAdd(&hist[bin_of(f[e])], 1u);
        }
        __syncthreads();
        uint4 *h4 = reinterpret_cast<uint4 *>(hist) + t; // thread t owns bins 4 t ... 4 t + 3
        const uint4 c = *h4;
        const uint32_t incl = cta_scan(c.x + c.y + c.z + c.w, sh.scan);
        uint4 at; // the bins' places
        at.x = incl - (c.x + c.y + c.z + c.w), at.y = at.x + c.x, at.z = at.y + c.y, at.w = at.z + c.z;
        *h4 = at;
        const uint32_t big = max(max(at.x < (uint32_t)C ? c.x : 0u, at.y < (uint32_t)C ? c.y : 0u), max(at.z < (uint32_t)C ? c.z : 0u, at.w < (uint32_t)C ? c.w : 0u));
        if (__reduce_max_sync(0xffffffffu, big) > kRankMaxBin && lane == 0) sh.biggest = 1;
        __syncthreads();
        if (sh.biggest == 0) {
            // entries behind the bin that completes the list have no place in it
#pragma unroll
            for (int k = 0; k < R; ++k) {
                const float f[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (f[e] <= top) {
                        const uint32_t place = atomicAdd(&hist[bin_of(f[e])], 1u);
                        if (place < (uint32_t)C + kRankMaxBin) list[place] = ((unsigned long long)order_key(f[e]) << 32) | (uint32_t)(4 * (T * k + t) + e);
                    }
            }
            __syncthreads();
            // hist[b] is now the end of bin b
            for (int e = t; e < min(m, C + (int)kRankMaxBin); e += T) {
                const unsigned long long x = list[e];
                const int bin = bin_of(order_key_inv((uint32_t)(x >> 32)));
                int k = bin > 0 ? (int)hist[bin - 1] : 0, r = k;
                if (k >= C) continue;
                for (const int end = (int)hist[bin]; k < end; ++k) r += list[k] < x ? 1 : 0;
                if (r < C) out[r] = (Out)(uint32_t)x;
            }
            return;
        }
    }
    // the exact route: many equal values, or one that is not finite
    auto keyfn = [&](int j, uint32_t &key) {
        if ((skip[j >> 5] >> (j & 31)) & 1u) return false;
        key = order_key(row[j]) ^ flip; // (the key of -x is the complement of that of x)
        return true;
    };
    if (t == 0) sh.n_list = 0;
    auto put = [&](int j, uint32_t key) { list[atomicAdd(&sh.n_list, 1u)] = ((unsigned long long)key << 32) | (uint32_t)j; };
    int held = C; // entries of the list
    if (n_in <= C + (int)kRankMaxBin) { // it has room for all tokens
        held = n_in;
        __syncthreads();
        for (int j = t; j < n; j += T) {
            uint32_t key;
            if (keyfn(j, key)) put(j, key);
        }
        __syncthreads();
    } else {
        uint32_t thr, need_eq, cnt_eq;
        block_select_threshold(CtaGroup(), keyfn, n, (uint32_t)C, sh.sel, thr, need_eq, cnt_eq);
        block_select_apply(CtaGroup(), keyfn, n, thr, need_eq, cnt_eq, sh.sel, put);
    }
    if ((held + T - 1) / T * held <= kRankMaxCount) {
        rank_sort(list, held, [&](int r, unsigned long long x) {
            if (r < C) out[r] = (Out)(uint32_t)x;
        });
    } else {
        cta_sort(list, held);
        for (int e = t; e < C; e += T) out[e] = (Out)(uint32_t)list[e];
    }
}

// Step 5a's vision tokens (flags are 0 or 1, 16-byte aligned): every thread has up to eight consecutive words of four flags, so that one
// sum over the CTA places all of them - in shared memory first (list, if it has room for n_keep), so that what is written is written
// side by side; row_word: the same indices once more, word by word for the gather that is waiting for them.  Exactly n_keep tokens are
// flagged: the pivots are distinct, every list is complete, and of pivot i's Q_i entries the pivots before it took at most Q_i - q_i.
// (32 flags of a warp at a time, and the text rows before them, took 1.1 us for 576 tokens and 1.8 for 2880, now 0.8 and 1.0.)
__device__ __forceinline__ void pack_flags(const uint8_t *keep, int vis_offset, int n_vis, int n_keep, const int64_t *__restrict__ pin, int32_t *__restrict__ oi,
                                           int64_t *__restrict__ op, int32_t *row_word, uint16_t *list, bool listed, uint32_t *per_warp)
{
    const int words = (n_vis + 3) / 4, per = (words + (int)blockDim.x - 1) / (int)blockDim.x, w0 = (int)threadIdx.x * per;
    auto flags = [&](int w) { // (what lies behind the last token does not count)
        const uint32_t f = reinterpret_cast<const uint32_t *>(keep)[w];
        return 4 * w + 4 <= n_vis ? f : f & ((1u << (8 * (n_vis - 4 * w))) - 1u);
    };
    uint32_t mine = 0;
    for (int w = w0; w < min(w0 + per, words); ++w) mine += __popc(flags(w));
    int at = (int)(cta_scan(mine, per_warp) - mine);
    auto put = [&](int k, int j) { // kept token number k is token j
        const int s = vis_offset + j;
        if (row_word) asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(row_word + vis_offset + k), "r"(s) : "memory");
        oi[vis_offset + k] = s;
        op[vis_offset + k] = pin ? pin[s] : (int64_t)s;
    };
    for (int w = w0; w < min(w0 + per, words); ++w)
        for (uint32_t f = flags(w); f; f &= f - 1u, ++at) {
            const int j = 4 * w + (__ffs((int)f) - 1) / 8;
            if (listed)
                list[at] = (uint16_t)j;
            else
                put(at, j);
        }
    if (!listed) return;
    __syncthreads();
    for (int k = threadIdx.x; k < n_keep; k += blockDim.x) put(k, list[k]);
}
// ... and its text rows, by threads first, first + threads ...
__device__ __forceinline__ void pack_text(int S, int vis_offset, int n_vis, int n_keep, const int64_t *__restrict__ pin, int32_t *__restrict__ oi,
                                          int64_t *__restrict__ op, int first, int threads)
{
    for (int u = first; u < S - n_vis; u += threads) {
        const int s = u < vis_offset ? u : u + n_vis, k = u < vis_offset ? u : u + n_keep;
        oi[k] = s;
        op[k] = pin ? pin[s] : (int64_t)s;
    }
}

// One pivot's turn, by a warp: the first `want` free entries of its ranked list L[0 .. M) (shared memory, 16-byte aligned) are
// taken.  flags[none] is a place that is never free.  No branch depends on an entry: what a lane does not hold or does not take
// goes to `none` (with a branch per entry a turn took 1.4 us, without 0.45).  kDetail: owners, and the last entry taken is
// returned to every lane (-1 if none).
template <bool kDetail>
__device__ __forceinline__ int take_turn(const uint16_t *L, int M, int want, uint8_t *flags, uint32_t none, int32_t *owner, int i)
{
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    int last = -1;
    for (int s = 0; s < M && want > 0; s += 256) {
        const int at = s + 8 * lane;
        uint4 e = make_uint4(0, 0, 0, 0);
        if (at < M) e = *reinterpret_cast<const uint4 *>(L + at);
        const uint32_t w[4] = {e.x, e.y, e.z, e.w};
        uint32_t j[8], f = 0; // f: which of the lane's entries are free
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            j[k] = (k & 1) ? w[k >> 1] >> 16 : w[k >> 1] & 0xffffu;
            j[k] = at + k >= M ? none : min(j[k], none);
        }
        uint32_t taken[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) taken[k] = flags[j[k]];
#pragma unroll
        for (int k = 0; k < 8; ++k) f |= taken[k] == 0 ? 1u << k : 0u;
        const int c = __popc(f);
        int before = 0, total = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t v = __ballot_sync(0xffffffffu, (c >> k) & 1);
            before += __popc(v & lt) << k;
            total += __popc(v) << k;
        }
        const int may = want - before; // how many of its free entries the lane may take
        uint32_t g = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const bool take = ((f >> k) & 1u) && __popc(f & ((1u << k) - 1u)) < may;
            g |= take ? 1u << k : 0u;
            flags[take ? j[k] : none] = 1;
        }
        if (kDetail) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if ((g >> k) & 1u) {
                    if (owner) owner[j[k]] = i;
                    last = (int)j[k];
                }
            const uint32_t any = __ballot_sync(0xffffffffu, g != 0);
            last = any ? __shfl_sync(0xffffffffu, last, 31 - __clz(any)) : last;
        }
        want -= total;
        __syncwarp(); // the flags are visible to the next block and the next pivot
    }
    return last;
}

// The same for short lists: 32 kGroups entries at a time, an entry of each group per lane, so that a group takes one vote; the first
// entries of the next list (or of this one) are on their way while this turn's flags are read.
template <int kGroups>
__device__ __forceinline__ void turn_entries(const uint16_t *L, int M, int s, uint32_t none, uint32_t (&j)[kGroups])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < kGroups; ++k) {
        const int at = s + 32 * k + lane;
        const uint32_t e = L[min(at, M - 1)];
        j[k] = at < M ? min(e, none) : none;
    }
}
template <int kGroups>
__device__ __forceinline__ void take_short_turns(const uint16_t *buf, int k0, int k1, int q, int r, uint8_t *flags, uint32_t none)
{
    const uint32_t lt = (1u << (threadIdx.x & 31)) - 1u;
    const int from = rank_place(k0, q, r, false);
    const uint16_t *L = buf;
    int M = rank_length(k0, q, r, false);
    uint32_t j[kGroups];
    turn_entries<kGroups>(L, M, 0, none, j);
    for (int i = k0; i < k1; ++i) {
        const int i2 = i + 1 < k1 ? i + 1 : i, M2 = rank_length(i2, q, r, false);
        const uint16_t *L2 = buf + rank_place(i2, q, r, false) - from;
        int want = q + (i < r ? 1 : 0);
        for (int s = 0;;) {
            uint32_t taken[kGroups], next[kGroups];
#pragma unroll
            for (int k = 0; k < kGroups; ++k) taken[k] = flags[j[k]];
            s += 32 * kGroups;
            const bool more = s < M;
            turn_entries<kGroups>(more ? L : L2, more ? M : M2, more ? s : 0, none, next);
            int before = 0;
#pragma unroll
            for (int k = 0; k < kGroups; ++k) {
                const uint32_t free = __ballot_sync(0xffffffffu, taken[k] == 0);
                if (taken[k] == 0 && before + __popc(free & lt) < want) flags[j[k]] = 1;
                before += __popc(free);
            }
            want -= before;
            __syncwarp(); // the flags are visible to the next block and the next pivot
            const bool done = want <= 0 || !more;
            if (done && more) turn_entries<kGroups>(L2, M2, 0, none, next);
#pragma unroll
            for (int k = 0; k < kGroups; ++k) j[k] = next[k];
            if (done) break;
        }
        L = L2, M = M2;
    }
}

// kGroups: 0, or the groups of take_short_turns (then neither owners nor a pivot's last dup are wanted, nor `each`)
template <int R, int kGroups>
__global__ void __launch_bounds__(kRankMaxThreads) rank_kernel(const RankParams p)
{
    extern __shared__ __align__(16) uint8_t rank_smem[];
    __shared__ RankShared sh;
    const int t = threadIdx.x, T = blockDim.x, warp = t >> 5, n = p.n_vis;
    const int i = blockIdx.x, b = blockIdx.y;
    const int32_t *piv = sh.piv;
    const float *rows = p.sim + (size_t)b * p.P * n, *row = rows + (size_t)i * n;
    unsigned long long *list = reinterpret_cast<unsigned long long *>(rank_smem);
    uint32_t *hist = reinterpret_cast<uint32_t *>(list + (p.m + kRankMaxBin + 1) / 2 * 2), *skip = hist + 4 * T;
    for (int k = t; k < (n + 31) / 32; k += T) skip[k] = 0;
    if (t < kRankTries) sh.n_below[t] = 0;
    if (t == 0) sh.n_pivots = 0, sh.biggest = 0;
    __syncthreads();
    wait_for_previous();
    let_next_start();
    if (*p.status != 0) return; // an earlier kernel of this call failed: its outputs are undefined
    float4 v[R];
    load_row<false>(row, n, 1.0f, v);
    const float none = __uint_as_float(kNotAToken);
    uint32_t mine = 0;
    for (int k = t; k < p.P; k += T) {
        const int pv = p.pivot_idx[(size_t)b * p.P + k];
        sh.piv[k] = pv;
        if (pv >= 0 && pv < n) {
            atomicOr(&skip[pv >> 5], 1u << (pv & 31));
            ++mine;
        }
    }
    if (mine) atomicAdd(&sh.n_pivots, mine);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const int j = 4 * (T * k + t);
        if (j >= n) break;
        const uint32_t x = skip[j >> 5] >> (j & 31);
        if (x & 1u) v[k].x = none;
        if (x & 2u) v[k].y = none;
        if (x & 4u) v[k].z = none;
        if (x & 8u) v[k].w = none;
    }
    const int Pv = (int)sh.n_pivots, q = (p.n_keep - Pv) / p.P, r = (p.n_keep - Pv) % p.P;
    const bool each = kGroups == 0 && p.each != 0;
    uint16_t *lists = p.lists + (size_t)b * p.sample_entries;
    if (q + (i < r ? 1 : 0) > 0) // (else this pivot keeps nothing, and so do all later ones)
        rank_row<R, false>(row, 0u, skip, v, n, n - Pv, lists + rank_place(i, q, r, each), rank_length(i, q, r, each), list, hist, sh);
    __syncthreads();
    if (t == 0) { // release: the list; acquire: the other pivots' lists
        int before;
        asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(before) : "l"(p.arrived + b) : "memory");
        sh.last = before == p.P - 1;
        if (before == p.P - 1) p.arrived[b] = 0;
    }
    __syncthreads();
    if (!sh.last) return;
    // ---- the sample's last CTA: the turns
    uint8_t *flags = rank_smem;
    uint16_t *stage = reinterpret_cast<uint16_t *>(rank_smem + rank_flag_bytes(n));
    int32_t *owner = kGroups == 0 && p.owner_out ? p.owner_out + (size_t)b * n : nullptr;
    float *eps = kGroups == 0 && p.eps_out ? p.eps_out + (size_t)b * p.P : nullptr;
    for (int k = t; k < (n + 16) / 16; k += T) reinterpret_cast<uint4 *>(flags)[k] = make_uint4(0, 0, 0, 0);
    if (owner)
        for (int j = t; j < n; j += T) owner[j] = -1;
    __syncthreads();
    if (t == 0) flags[n] = 1;
    for (int k = t; k < p.P; k += T)
        if (piv[k] >= 0 && piv[k] < n) {
            flags[piv[k]] = 1;
            if (owner) owner[piv[k]] = p.P + k;
        }
    const int n_active = q > 0 ? p.P : r; // pivots with a quota
    if (eps)
        for (int k = n_active + t; k < p.P; k += T) eps[k] = __int_as_float(0x7fc00000);
    if (each) { // independent pivots: the lists are what they keep
        for (int k = n_active - 1; k >= 0; --k) {
            const uint16_t *L = lists + rank_place(k, q, r, true);
            const int M = rank_length(k, q, r, true);
            for (int e = t; e < M; e += T) {
                const int j = __ldcg(L + e);
                flags[j] = 1;
                if (owner) owner[j] = k; // the first pivot in rank order that took a token owns it: it writes last
                if (eps && e == M - 1) eps[k] = rows[(size_t)k * n + j];
            }
            if (owner) __syncthreads();
        }
        if (t == 0) sh.n_list = 0;
        __syncthreads();
        uint32_t kept = 0;
        for (int j = t; j < n; j += T) {
            const uint8_t f = flags[j] != 0;
            kept += f;
            p.keep_out[(size_t)b * n + j] = f;
        }
        kept = __reduce_add_sync(0xffffffffu, kept);
        if ((t & 31) == 0) atomicAdd(&sh.n_list, kept);
        __syncthreads();
        if (t == 0) p.len_out[b] = p.S - n + (int)sh.n_list;
        return;
    }
    // rounds: the lists of as many pivots as fit a staging buffer; while warp 0 takes one round's turns the others fetch the next
    auto round_end = [&](int k0) {
        if (rank_place(n_active, q, r, false) - rank_place(k0, q, r, false) <= p.stage_entries) return n_active;
        int k1 = k0;
        while (k1 < n_active && (k1 == k0 || rank_place(k1 + 1, q, r, false) - rank_place(k0, q, r, false) <= p.stage_entries)) ++k1;
        return k1;
    };
    auto fetch = [&](int k0, int k1, uint16_t *buf, int first, int threads) {
        const int from = rank_place(k0, q, r, false), words = k1 > k0 ? (rank_place(k1 - 1, q, r, false) + (rank_length(k1 - 1, q, r, false) + 7) / 8 * 8 - from) / 8 : 0;
        const uint4 *src = reinterpret_cast<const uint4 *>(lists + from);
        for (int e = first; e < words; e += threads) reinterpret_cast<uint4 *>(buf)[e] = __ldcg(src + e);
    };
    const int S_out = p.S - n + p.n_keep;
    const int64_t *pin = p.pos_in ? p.pos_in + (size_t)b * p.S : nullptr;
    int32_t *oi = p.out_idx + (size_t)b * S_out;
    int64_t *op = p.out_pos + (size_t)b * S_out;
    int k0 = 0, k1 = round_end(0);
    fetch(k0, k1, stage, t, T);
    __syncthreads(); // (and the pivots are flagged)
    for (int round = 0; k0 < n_active; ++round) {
        uint16_t *buf = stage + (size_t)(round & 1) * p.stage_entries;
        const int k2 = round_end(k1);
        if (warp == 0) {
            const int from = rank_place(k0, q, r, false);
            if constexpr (kGroups > 0) {
                take_short_turns<kGroups>(buf, k0, k1, q, r, flags, (uint32_t)n);
            } else {
                for (int k = k0; k < k1; ++k) {
                    const uint16_t *L = buf + rank_place(k, q, r, false) - from;
                    const int M = rank_length(k, q, r, false), want = q + (k < r ? 1 : 0);
                    int last = -1;
                    if (owner || eps)
                        last = take_turn<true>(L, M, want, flags, (uint32_t)n, owner, k);
                    else
                        take_turn<false>(L, M, want, flags, (uint32_t)n, nullptr, k);
                    if (eps && t == 0) eps[k] = last >= 0 ? rows[(size_t)k * n + last] : __int_as_float(0x7fc00000);
                }
            }
        } else {
            if (round == 0) pack_text(p.S, p.vis_offset, n, p.n_keep, pin, oi, op, t - 32, T - 32);
            if (k2 > k1) fetch(k1, k2, stage + (size_t)((round + 1) & 1) * p.stage_entries, t - 32, T - 32);
        }
        __syncthreads();
        k0 = k1, k1 = k2;
    }
    if (n_active == 0) pack_text(p.S, p.vis_offset, n, p.n_keep, pin, oi, op, t, T);
    // (the staging buffers, one where all lists fit it, two otherwise, are free again)
    const int room = p.stage_entries >= (int)p.sample_entries ? p.stage_entries : 2 * p.stage_entries;
    pack_flags(flags, p.vis_offset, n, p.n_keep, pin, oi, op, p.row_word ? p.row_word + (size_t)b * S_out : nullptr, stage, p.n_keep <= room, sh.scan);
    if (p.keep_out)
        for (int j = t; j < n; j += T) p.keep_out[(size_t)b * n + j] = flags[j] != 0;
}

// The form for rows of n_vis values; m: the longest list, q: the quota.  Turns by the longest list and the quota (us for the whole
// retention, 256 entries at a time / as here): 128 pivots keeping 4 each of lists up to 512 60 / 46, 100 pivots keeping 2 of up
// to 200 48 / 29, 100 keeping 7 of up to 700 57 / 54, 32 keeping 9 of up to 288 26 / 23; but 36 of up to 1168 33.2 / 35.4, 8 keeping 149 of up to 1192 19 / 21.
// (Kernels of their own: with all four in one the small cases took 1 to 2 us more, for code that is fetched and not used.)
using RankKernel = void (*)(RankParams);
template <int R>
inline RankKernel rank_kernel_of(int groups)
{
    return groups == 0 ? rank_kernel<R, 0> : groups == 1 ? rank_kernel<R, 1> : groups == 2 ? rank_kernel<R, 2> : rank_kernel<R, 4>;
}
inline RankKernel rank_kernel_of(int regs, int groups)
{
    return regs == 2 ? rank_kernel_of<2>(groups) : regs == 4 ? rank_kernel_of<4>(groups) : regs == 6 ? rank_kernel_of<6>(groups) : rank_kernel_of<8>(groups);
}
inline int rank_turn_groups(int m, int q) { return q <= 3 ? 1 : q <= 8 ? 2 : m <= 640 ? 4 : 0; }

// Steps 1 and 2's selection, pivots from scores: the P best tokens of a sample in order of (score, index), one CTA per sample, the
// ranking above over the scores or, where the largest are best, their negatives.  A radix select and a sort
// (pivot_kernel) are some twenty block-wide steps.  Measured (us, with the copy of the pivots' rows, which starts behind it): 1 x 2880
// tokens, 128 pivots 26 -> 18; 16 x 1000, 64 pivots 21 -> 17; 256 x 2880, 32 pivots 30 -> 22; 140 x 2880, 128 pivots 36 -> 28.
template <int R>
__global__ void __launch_bounds__(kRankMaxThreads) pivot_rank_kernel(const float *score, int n, int P, int smallest, int32_t *__restrict__ pivot_idx)
{
    extern __shared__ __align__(16) uint8_t rank_smem[];
    __shared__ RankShared sh;
    const int t = threadIdx.x, T = blockDim.x;
    unsigned long long *list = reinterpret_cast<unsigned long long *>(rank_smem);
    uint32_t *hist = reinterpret_cast<uint32_t *>(list + (P + kRankMaxBin + 1) / 2 * 2), *skip = hist + 4 * T;
    for (int k = t; k < (n + 31) / 32; k += T) skip[k] = 0;
    if (t < kRankTries) sh.n_below[t] = 0;
    if (t == 0) sh.biggest = 0;
    __syncthreads();
    wait_for_previous();
    let_next_start();
    const float *row = score + (size_t)blockIdx.x * n;
    float4 v[R];
    load_row<true>(row, n, smallest ? 1.0f : -1.0f, v);
    rank_row<R, true>(row, smallest ? 0u : 0xffffffffu, skip, v, n, n, pivot_idx + (size_t)blockIdx.x * P, P, list, hist, sh);
}

} // namespace dart
