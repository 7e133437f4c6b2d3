// Flow path: steps 1-3 of a whole batch in ONE persistent launch for up to 32 pivots, built so that a key row's second read
// comes from the L2 cache (or is already waiting in shared memory) instead of HBM.
//
// A row's similarities need the sample's pivots, and those need the norms of all the sample's rows: every row is read twice.
// What decides where the second read is served from is how many bytes of other rows pass between the two reads:
//   (time from a sample's first score to its pivots + time one second-pass item takes) x bandwidth.
// So all of that is kept short here:
//   - the scorers take one row per warp at a time, every SM on the same sample: a sample's rows are scored within a few
//     microseconds of each other;
//   - a row's score and sum of squares are published as ONE 64-bit word, and readers poll the words themselves: no counter,
//     no fence, no second round trip;
//   - a few CTAs do nothing but select pivots from those words: about 3 us a sample (5-6 us on an SM that also streams), and
//     publish them the same way, word by word;
//   - a second-pass item is 64 rows x 1/nsl of the columns: an SM's pivot tile is P x d/nsl (16 KB at 8 pivots, d = 4096, 4
//     slices) instead of P x d, and the item takes about 2.5 us instead of the 20 us of a 128-row tile of full rows;
//   - the item's rows are fetched into a ring before the pivots are known;
//   - the scorers are held back to `window` rows beyond the samples that have their pivots and, in long batches, to `lead` beyond
//     their SM's second pass.
// The slices' shares of a dot product meet in global memory (L2): when a row group's are all there, each of its SMs adds up a part of
// them in slice order and divides by the norms (Eq. 7), so results are bitwise reproducible.
// With the caller's pivots nothing is selected: first and second read then follow each other within the window.
//
// What bounds it: no unit.  32 x 2880 x 4096, 8 pivots (173 us): DRAM 56 % of its peak, L2 41 %, L2 to SM 9.8 TB/s (every key byte crosses
// twice), shared-memory wavefronts 37 %, issue slots 54 %, tensor pipe 7 %; the warps wait for values on their way (long scoreboard 3.7
// of 10.7 cycles per instruction) - the distance between a row's two reads, start and tail.
//
// Per CTA (768 or 896 threads, one CTA per SM, cooperative launch):
//   warps 0-3    pivots of the samples this SM has items of: wait for them, fetch the pivot rows' slice (two buffers)
//   warps 4-7    second pass: mma.sync.m16n8k16, 16 rows each (the tensor pipe is 7 % busy; what the form costs is that every warp
//                reads the pivot tile from shared memory again, which a tcgen05.mma of 64 rows would do once)
//   warp 8       producer: TMA tiles of 64 rows x 64 columns (128-byte swizzle), two per ring stage
//   warps 9-12   combine: count the item, wait for its row group's other slices, add up a part of the shares and write the similarities
//   warps 13-20  scorers: sum |x| (the K-norm of the Sec. 3.3 footnote) and sum x^2 (Eq. 7's denominator) of a row
//   warp 21      watcher: how far the pivots of the batch have got, for the scorers' window
//   warps 22-23  feeders: the scorers' rows into their slots
//   warps 24-27  with more than 16 pivots: second pass for the second half of the pivots
// Every wait is bounded in time; on expiry the kernel records DART_ERR_TIMEOUT in the status word, lets the copies in flight
// land and exits normally.
#pragma once
#include "dart_sweep.cuh"

namespace dart {
namespace flow {

using sweep::Ctl;
using sweep::mbar_arrive;
using sweep::mbar_arrive_expect_tx;
using sweep::mbar_init;
using sweep::Ring;
using sweep::smem_u32;
using sweep::tma_load_2d;

constexpr int kMaxP = 32;
constexpr int kRows = 64;                  // rows of an item
constexpr int kAtomCols = 64;              // 64 bf16 = 128 bytes = one swizzle row
constexpr int kAtomBytes = kRows * 128;    // 8 KB
constexpr int kAps = 2;                    // atoms per ring stage
constexpr int kStageBytes = kAps * kAtomBytes;
constexpr int kMaxStages = 13;
constexpr int kPivWarps = 4;
constexpr int kMulWarp0 = 4, kMulWarps = 4; // 16 rows each; with more than 16 pivots a second group of four takes half of the pivots
constexpr int kProdWarp = 8;
constexpr int kCombWarp0 = 9, kCombWarps = 4; // (an item is counted 2-3 us after its shares were written: two warps held the others up)
constexpr int kScoreWarp0 = kCombWarp0 + kCombWarps, kScoreWarps = 8;
constexpr int kWatchWarp = kScoreWarp0 + kScoreWarps;
constexpr int kFeedWarp = kWatchWarp + 1;
constexpr int kFeedWarps = 2;
constexpr int kMulWarp1 = kFeedWarp + kFeedWarps;
__host__ __device__ constexpr int mul_groups(int NT) { return NT > 2 ? 2 : 1; }
__host__ __device__ constexpr int threads(int NT) { return 32 * (kMulWarp1 + (mul_groups(NT) - 1) * kMulWarps); }
constexpr int kChunk = 8;                  // scorers: 16-byte pieces per lane and chunk
constexpr int kChunkUnits = 32 * kChunk;
constexpr uint32_t kChunkBytes = kChunk * 512; // 4 KB: half a row of 4096 columns
constexpr int kMaxSlots = 6;               // chunks of a row on their way per scorer
constexpr int kSel = 512, kSelGroups = 4;  // threads of a selector CTA that select; at most so many groups of them
__host__ inline int sel_threads(int n_vis) { return n_vis > 1024 ? kSel : kSel / kSelGroups; }
// Longest list that a group of T threads ranks by counting: 3 x 384 or 2 x 640 steps a thread, about what a radix select takes
// (64 x 576 tokens, whole call: lists of 288 111 us, of 576 227, radix select 143; 8 x 2880: lists of 720 108, radix select 101).
__host__ __device__ constexpr int sel_list(int T) { return T == kSel ? 640 : 384; }
constexpr int kPoll = 6;                   // words per selecting thread on their way at once: 3072 tokens
constexpr int kMail = 2;                   // items on their way to each combine warp
constexpr int kPvRing = 16;                // pivot lists kept for the combine warps: 2 pivot buffers + 8 items on their way, and slack
constexpr int kMaxVis = 8192;              // a sample's keys in a selector's shared memory
constexpr int kMaxSlices = 16;
constexpr int kMaxItemAtoms = 16;          // items of at most 128 KB where the batch leaves the choice
constexpr int kStaticSmemReserve = 6144;
constexpr int32_t kNoPivot = -1;           // a pivot's word before it is published
constexpr uint32_t kNoWord = ~0u;
constexpr unsigned long long kNoRec = ~0ull; // a row's word before it is published (no sums produce it)
enum { kWaitRec = 90, kWaitPivots, kWaitPivFree, kWaitPiv, kWaitStage, kWaitStageFree, kWaitMailFree, kWaitMail, kWaitCombRec,
       kWaitWindow, kWaitChunk = 101, kWaitShares }; // (100 is taken by the check of given pivots)
// Selector CTAs: a selection takes about 3 us, a sample streams at about 6 MB per us.  (256 samples of 1 to 4 MB: 8 or 16 CTAs for
// them 360 and 237 us, 6 and 8 CTAs 356 and 229; 2 and 3 are no better and cost large samples 1 %.)
__host__ inline int selectors(long long sample_bytes) { return sample_bytes >= (4 << 20) ? 4 : sample_bytes >= (1 << 20) ? 6 : 8; }

struct Params {
    int B, S, vis_offset, n_vis, P, d8; // d8: row width in 16-byte units
    int n_atoms, n_rg, nsl, na_max;     // atoms per row; row groups per sample; column slices; atoms of the widest slice
    int n_st, n_slot;                   // ring depth; chunks on their way per scorer
    int rows_task, n_chunk;             // scoring: rows per task (2: two rows to a chunk); chunks per task
    int n_stream;                       // CTAs that stream; the others select
    int sel_threads;                    // threads per selection
    int given;                          // the pivots are in pivot_idx already
    int norm_kind, smallest;
    int withhold;                       // test hook: 1 = one row's score is never published, 2 = one item's shares are never counted in
    int window;                         // rows the scorers may be ahead of `pos` (>= n_vis)
    int lead;                           // ... and of their own SM's second pass (>= n_vis: a sample's pivots wait for all of its rows)
    uint32_t pitch;                     // bytes between pivot rows in shared memory
    unsigned long long wait_ns;
    const uint4 *keys;                  // [B][S][d]
    unsigned long long *rec;            // [B][n_vis] (score bits, sum-of-squares bits); kNoRec on entry, put back by the gather
    float *part;                        // [B][n_rg][nsl][8 NT][64] the slices' shares of the dot products
    int *cnt;                           // [B][n_rg] slices that have arrived; zero on entry, put back by the gather
    float *sim;                         // [B][P][n_vis]
    float *l1, *ssq;                    // [B][n_vis], NULL unless the caller wants them
    int32_t *pivot_idx;                 // [B][P]
    int32_t *pv_word;                   // [B][kMaxP] the same, published word by word; kNoPivot on entry, put back by the gather
    const float *text_ssq;              // [B][P] sums of squares of given pivots that are text tokens
    int *status;
};

struct Shared {
    unsigned long long full[kMaxStages], empty[kMaxStages];
    unsigned long long chunk_full[kScoreWarps][kMaxSlots], chunk_empty[kScoreWarps][kMaxSlots];
    unsigned long long piv_full[2], piv_empty[2];
    unsigned long long mail_full[kCombWarps][kMail], mail_empty[kCombWarps][kMail];
    uint32_t set_best[kSelGroups][32]; // selectors: best keys of sets of threads
    uint32_t n_list[kSelGroups];
    int32_t pv[kPvRing][kMaxP];       // pivots of the samples on their way, by the SM's own count of samples
    int abort_flag;
    volatile int at;                  // first row (of the batch) of the SM's own item in the second pass
    volatile int pos;                 // rows (of the batch) whose samples have their pivots; given pivots: rows the second pass is through with
};
static_assert(sizeof(Shared) + 64 <= kStaticSmemReserve, "static shared memory exceeds its reserve");

// shared memory of the two pivot buffers; of a selector: every group's list, histogram and keys
__host__ inline size_t pivot_bytes(int NT, int na_max) { return (size_t)2 * 8 * NT * ((size_t)na_max * 128 + 16); }
__host__ inline size_t selector_bytes(int n_vis)
{
    const int T = sel_threads(n_vis);
    return ((size_t)sel_list(T) * 8 + sizeof(SelectSmem) + (size_t)n_vis * 4) * (kSel / T);
}

// `size` threads of a selector CTA, with a named barrier
struct SelGroup {
    int t, T, barrier;
    __device__ __forceinline__ int tid() const { return t; }
    __device__ __forceinline__ int size() const { return T; }
    __device__ __forceinline__ void sync() const { asm volatile("bar.sync %0, %1;" ::"r"(barrier), "r"(T) : "memory"); }
};

__device__ __forceinline__ unsigned long long ld_rec(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_word(const void *p)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_word(int32_t *p, int32_t v)
{
    asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_rec(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// two fp32 additions / multiply-adds per instruction
__device__ __forceinline__ void add2(unsigned long long &a, unsigned long long x)
{
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(a) : "l"(x));
}
__device__ __forceinline__ void fma2(unsigned long long &a, unsigned long long x)
{
    asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(a) : "l"(x));
}
__device__ __forceinline__ float sum2(unsigned long long a)
{
    return __uint_as_float((uint32_t)a) + __uint_as_float((uint32_t)(a >> 32));
}
__device__ __forceinline__ void ldmatrix4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The items of one SM: slice sl = CTA % nsl, and of that slice every m-th (sample, row group), sample-major, m being the
// number of SMs that share the slice.
struct Items {
    int sl, a0, na; // slice, its first atom and their number
    int b, rg;      // current item
    int n_rg, B, step;
    __device__ explicit Items(const Params &p)
    {
        sl = (int)(blockIdx.x % (unsigned)p.nsl);
        a0 = p.n_atoms * sl / p.nsl;
        na = p.n_atoms * (sl + 1) / p.nsl - a0;
        step = (p.n_stream - sl + p.nsl - 1) / p.nsl;
        n_rg = p.n_rg, B = p.B;
        const int first = (int)blockIdx.x / p.nsl;
        b = first / n_rg, rg = first - b * n_rg;
    }
    __device__ __forceinline__ bool valid() const { return b < B; }
    __device__ __forceinline__ void next()
    {
        rg += step;
        if (rg >= n_rg) {
            const int k = rg / n_rg;
            b += k, rg -= k * n_rg;
        }
    }
};

// The scoring tasks of one scorer (warp w of SM c): of the batch's tasks - p.rows_task rows of one sample, one row where rows are
// wider than half a chunk - every (8 n_stream)-th, sample-major.  The feeder and the scorer walk the same list.
struct Tasks {
    int b, t;       // sample, task within it
    int db, dt, T, B;
    __device__ Tasks(const Params &p, int w)
    {
        T = (p.n_vis + p.rows_task - 1) / p.rows_task, B = p.B;
        const int first = w * p.n_stream + (int)blockIdx.x, step = p.n_stream * kScoreWarps;
        b = first / T, t = first - b * T;
        db = step / T, dt = step - db * T;
    }
    __device__ __forceinline__ bool valid() const { return b < B; }
    __device__ __forceinline__ void next()
    {
        b += db, t += dt;
        if (t >= T) t -= T, ++b;
    }
};

// Feeders: a lane keeps one scorer's p.n_slot slots (4 KB chunks of rows) on their way, as far as the window allows.  Warps of their
// own: a bulk copy takes its thread some 500 cycles to issue (with every scorer refilling its own slots a row of 8 KB took
// 4000 cycles, and the scorers bound the whole path).  Two: a warp that feeds all eight scorers spends 195 cycles per copy and nothing
// else 88 % of the time (whole calls, us, one / two: 64 x 576 118 / 115, 8 x 1500 x 3072 60.5 / 59.3, 256 x 1000 x 3072 514 / 494; 256 x 2880 about
// the same, three there 4 % more than two and four, which costs registers, 7 %).
__device__ __forceinline__ void feed(const Params &p, const Ctl &ctl, Shared &sh, uint32_t slot0)
{
    const int lane = threadIdx.x & 31, w = ((int)(threadIdx.x >> 5) - kFeedWarp) + kFeedWarps * lane; // this lane's scorer
    unsigned long long policy;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(policy));
    const int nc = p.n_chunk;
    Tasks it(p, w < kScoreWarps ? w : 0);
    bool more = w < kScoreWarps && it.valid();
    int c = 0, in = 0;
    uint32_t phase = 1;
    long long issued = 0, since = clock64();
    for (uint32_t spin = 0; __any_sync(0xffffffffu, more);) {
        bool go = false;
        const int far = min(sh.pos + p.window, sh.at + p.lead);
        if (more) {
            const int row = it.b * p.n_vis + it.t * p.rows_task;
            go = (c > 0 || row < far) && sweep::mbar_test(smem_u32(&sh.chunk_empty[w][in]), phase);
            if (go) {
                const int j = it.t * p.rows_task, rows = min(p.rows_task, p.n_vis - j);
                const int from = c * kChunkUnits, n = p.rows_task > 1 ? rows * p.d8 : min(kChunkUnits, p.d8 - from);
                const uint32_t bar = smem_u32(&sh.chunk_full[w][in]);
                mbar_arrive_expect_tx(bar, (uint32_t)n * 16u);
                sweep::bulk_load(slot0 + (uint32_t)(w * p.n_slot + in) * kChunkBytes,
                                 p.keys + ((size_t)it.b * p.S + p.vis_offset + j) * (size_t)p.d8 + from, (uint32_t)n * 16u, bar, policy);
                ++issued;
                if (++in == p.n_slot) in = 0, phase ^= 1u;
                if (++c == nc) {
                    c = 0;
                    it.next();
                    more = it.valid();
                }
            }
        }
        if (__any_sync(0xffffffffu, go)) {
            since = clock64();
            continue;
        }
        __nanosleep(20);
        if ((++spin & 31u) == 0u) {
            bool dead = ctl.aborted();
            if (!dead && (unsigned long long)(clock64() - since) > ctl.limit_cycles) {
                if (lane == 0) ctl.give_up(kWaitWindow, it.b);
                dead = true;
            }
            if (__any_sync(0xffffffffu, dead)) break;
        }
    }
    // the CTA must not exit while a copy is on its way, whatever became of the scorers
    __syncwarp();
    for (long long i = issued > p.n_slot ? issued - p.n_slot : 0; i < issued; ++i)
        ctl.wait_landed(smem_u32(&sh.chunk_full[w][i % p.n_slot]), (uint32_t)((i / p.n_slot) & 1));
}

// The scorers.  A lane adds up the two halves of a chunk apart: they are two rows' (rows_task = 2) or the same row's.
__device__ __forceinline__ void score_rows(const Params &p, const Ctl &ctl, Shared &sh, uint32_t slot0)
{
    const int lane = threadIdx.x & 31, w = (int)(threadIdx.x >> 5) - kScoreWarp0;
    slot0 += (uint32_t)(w * p.n_slot) * kChunkBytes + (uint32_t)lane * 16u;
    int out = 0;
    uint32_t phase = 0;
    for (Tasks it(p, w); it.valid(); it.next()) {
        unsigned long long s[2] = {0ull, 0ull}, q[2] = {0ull, 0ull}; // |x| and x^2, by half of the chunk
        const int j = it.t * p.rows_task, rows = min(p.rows_task, p.n_vis - j);
        int left = rows * p.d8 - lane; // 16-byte pieces from this lane's first on
        for (int c = 0; c < p.n_chunk; ++c, left -= kChunkUnits) {
            const bool ok = ctl.wait_bar(smem_u32(&sh.chunk_full[w][out]), phase, kWaitChunk, it.b);
            if (!__all_sync(0xffffffffu, ok)) return;
            uint4 v[kChunk];
#pragma unroll
            for (int u = 0; u < kChunk; ++u) {
                v[u] = sweep::lds128(slot0 + (uint32_t)out * kChunkBytes + (uint32_t)u * 512u);
                if (u * 32 >= left) v[u] = make_uint4(0, 0, 0, 0); // (what a slot holds beyond the row is left from another one)
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh.chunk_empty[w][out])); // (the values are in registers)
            if (++out == p.n_slot) out = 0, phase ^= 1u;
#pragma unroll
            for (int u = 0; u < kChunk; ++u) {
                const uint32_t x4[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t a = x4[e] & 0x7fff7fffu; // both signs cleared: neither sum looks at them
                    unsigned long long x;
                    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "r"(a << 16), "r"(a & 0xffff0000u));
                    add2(s[u / (kChunk / 2)], x);
                    fma2(q[u / (kChunk / 2)], x);
                }
            }
        }
        float s0 = sum2(s[0]), q0 = sum2(q[0]), s1 = sum2(s[1]), q1 = sum2(q[1]);
        const size_t r = (size_t)it.b * p.n_vis + j;
        float l1, ssq;
        int row = 0;
        if (p.rows_task == 1) {
            // two sums over the warp: the halves of the warp exchange one each, then every half adds up its own
            s0 += s1, q0 += q1;
            float x = lane < 16 ? s0 : q0;
            x += __shfl_xor_sync(0xffffffffu, lane < 16 ? q0 : s0, 16);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            l1 = x, ssq = __shfl_xor_sync(0xffffffffu, x, 16);
        } else {
            // four sums: rows apart by the halves of the warp, then |x| and x^2 by quarters
            const bool up = lane >= 16, odd = (lane & 8) != 0;
            float a = up ? s1 : s0, b = up ? q1 : q0;
            a += __shfl_xor_sync(0xffffffffu, up ? s0 : s1, 16);
            b += __shfl_xor_sync(0xffffffffu, up ? q0 : q1, 16);
            float x = odd ? b : a;
            x += __shfl_xor_sync(0xffffffffu, odd ? a : b, 8);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            l1 = x, ssq = __shfl_xor_sync(0xffffffffu, x, 8);
            row = lane >> 4;
        }
        if ((lane & 15) == 0 && (lane == 0 || p.rows_task == 2) && row < rows && !(p.withhold == 1 && r + row == 0)) {
            st_rec(p.rec + r + row, ((unsigned long long)__float_as_uint(ssq) << 32) | __float_as_uint(l1));
            if (p.l1) p.l1[r + row] = l1, p.ssq[r + row] = ssq;
        }
    }
}

// The end of a selection where many keys pass the floor: the P best by radix select, ranked and published.  (Not inlined, and with a
// publication of its own, so that the code of every other selection stays together: 256 x 2880 1741 us as a branch in it, 1732 so.)
__device__ __noinline__ void select_among_many(const SelGroup group, const uint32_t *skey, int n, int P, SelectSmem &sel, unsigned long long *list, uint32_t *n_list,
                                               int32_t *pv_word, int32_t *pivot_idx)
{
    group.sync(); // everybody has read the list's length
    if (group.t == 0) *n_list = 0;
    auto keyfn = [&](int j, uint32_t &key) {
        key = ~skey[j];
        return true;
    };
    uint32_t thr, need_eq, cnt_eq;
    block_select_threshold(group, keyfn, n, (uint32_t)P, sel, thr, need_eq, cnt_eq);
    block_select_apply(group, keyfn, n, thr, need_eq, cnt_eq, sel, [&](int j, uint32_t key) {
        list[atomicAdd(n_list, 1u)] = ((unsigned long long)key << 32) | (uint32_t)j;
    });
    if (group.t < P) { // P <= 32
        const unsigned long long mine = list[group.t];
        int r = 0;
        for (int u = 0; u < P; ++u) r += list[u] < mine ? 1 : 0;
        st_word(pv_word + r, (int32_t)(uint32_t)mine);
        pivot_idx[r] = (int32_t)(uint32_t)mine;
    }
    group.sync(); // the list may be filled again
}

// The selectors (CTAs that do nothing else).  p.sel_threads threads (512, or four groups of 128 side by side for short samples,
// which come faster than one group takes them) read a sample's words as they appear; the P-th best of 32 sets' best keys is a
// floor that few keys pass; those are ranked by counting.  Where many pass (equal scores: blank patches, padding) a radix select
// finds the P best first, since counting is quadratic (equal rows, pivots alone kept, whole calls, us, counting / so: 64 x 576 227 / 143,
// 8 x 2880 547 / 103, 32 x 2880 1954 / 303, 2 x 8192 1824 / 61).
__device__ __forceinline__ void select_pivots(const Params &p, const Ctl &ctl, Shared &sh, uint8_t *smem)
{
    const int T = p.sel_threads, grp = (int)threadIdx.x / T, n_grp = kSel / T, most = sel_list(T);
    const int t = (int)threadIdx.x - grp * T, lane = t & 31;
    unsigned long long *list = reinterpret_cast<unsigned long long *>(smem) + grp * most;
    SelectSmem &sel = reinterpret_cast<SelectSmem *>(smem + n_grp * most * 8)[grp];
    uint32_t *skey = reinterpret_cast<uint32_t *>(smem + n_grp * (most * 8 + sizeof(SelectSmem))) + (size_t)grp * p.n_vis;
    auto any = [&](bool x) { // OR over the group; doubles as its barrier
        uint32_t r;
        asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 q, %1, 0;\nbar.red.or.pred p, %2, %3, q;\nselp.u32 %0, 1, 0, p;\n}"
                     : "=r"(r)
                     : "r"((uint32_t)x), "r"(1 + grp), "r"(T)
                     : "memory");
        return r != 0;
    };
    const int n_sel = ((int)gridDim.x - p.n_stream) * n_grp;
    for (int b = ((int)blockIdx.x - p.n_stream) * n_grp + grp; b < p.B; b += n_sel) {
        const uint32_t *rec = reinterpret_cast<const uint32_t *>(p.rec + (size_t)b * p.n_vis) + (p.norm_kind == 2 ? 1 : 0);
        const long long t0 = clock64();
        bool dead = false;
        uint32_t best = 0; // larger = better
        for (int j0 = t; j0 < p.n_vis && !dead; j0 += T * kPoll) {
            // all words that are still missing are asked for together (one after the other, a thread that had started early
            // paid a round trip for each of its six)
            uint32_t v[kPoll], miss = 0;
#pragma unroll
            for (int u = 0; u < kPoll; ++u) {
                v[u] = 0;
                if (j0 + u * T < p.n_vis) miss |= 1u << u;
            }
            const uint32_t mine = miss;
            for (uint32_t spin = 1; miss && !dead; ++spin) {
#pragma unroll
                for (int u = 0; u < kPoll; ++u)
                    if ((miss >> u) & 1u) v[u] = ld_word(rec + 2 * (j0 + u * T));
#pragma unroll
                for (int u = 0; u < kPoll; ++u)
                    if (v[u] != kNoWord) miss &= ~(1u << u);
                if (miss) __nanosleep(32);
                if ((spin & 63u) == 0u) {
                    dead = ctl.aborted();
                    if (!dead && (unsigned long long)(clock64() - t0) > ctl.limit_cycles) {
                        ctl.give_up(kWaitRec, b);
                        dead = true;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < kPoll; ++u) {
                uint32_t k = order_key(__uint_as_float(v[u]));
                if (p.smallest) k = ~k;
                if ((mine >> u) & 1u) {
                    skey[j0 + u * T] = k;
                    best = max(best, k);
                }
            }
        }
        uint32_t g = best; // best of a set of T / 32 lanes
        for (int o = T / 64; o > 0; o >>= 1) g = max(g, __shfl_xor_sync(0xffffffffu, g, o));
        if ((t & (T / 32 - 1)) == 0) sh.set_best[grp][t / (T / 32)] = g;
        if (t == 0) sh.n_list[grp] = 0;
        if (any(dead)) return;
        // the floor: the P-th best of the 32 sets' best keys
        const uint32_t x = sh.set_best[grp][lane];
        int gt = 0, ge = 0;
#pragma unroll
        for (int u = 0; u < 32; ++u) {
            const uint32_t y = __shfl_sync(0xffffffffu, x, u);
            gt += y > x, ge += y >= x;
        }
        const uint32_t here = __ballot_sync(0xffffffffu, gt < p.P && ge >= p.P); // (samples of fewer tokens than sets: empty sets hold 0)
        const uint32_t fl = __shfl_sync(0xffffffffu, x, __ffs(here) - 1);
        if (best >= fl)
            for (int j = t; j < p.n_vis; j += T) {
                const uint32_t k = skey[j];
                if (k >= fl) {
                    const uint32_t slot = atomicAdd(&sh.n_list[grp], 1u);
                    if (slot < (uint32_t)most) list[slot] = ((unsigned long long)k << 32) | (0xffffffffu - (uint32_t)j); // equal scores: lower index first
                }
            }
        any(false);
        const int m = (int)sh.n_list[grp];
        if (m > most) {
            select_among_many(SelGroup{t, T, 1 + grp}, skey, p.n_vis, p.P, sel, list, &sh.n_list[grp], p.pv_word + (size_t)b * kMaxP, p.pivot_idx + (size_t)b * p.P);
            continue;
        }
        for (int e = t; e < m; e += T) {
            const unsigned long long mine = list[e];
            int r = 0;
#pragma unroll 8 // (left to the compiler: 4 x 117 x 4096, 31 pivots 45 or 53 us, 25 x 925 x 6144 187 or 208, as it happens to choose)
            for (int u = 0; u < m; ++u) r += list[u] > mine ? 1 : 0;
            if (r < p.P) {
                const int32_t pv = (int32_t)(0xffffffffu - (uint32_t)mine);
                st_word(p.pv_word + (size_t)b * kMaxP + r, pv);
                p.pivot_idx[(size_t)b * p.P + r] = pv;
            }
        }
        any(false); // the list may be filled again
    }
}

// Pivots of the samples this SM has items of: their slice of the columns.
template <int NT>
__device__ __forceinline__ void take_pivots(const Params &p, const Ctl &ctl, Shared &sh, uint32_t piv0)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int seq = 0, last_b = -1;
    for (Items it(p); it.valid(); it.next()) {
        if (it.b == last_b) continue;
        last_b = it.b;
        const int b = it.b, buf = seq & 1;
        bool ok = ctl.wait_bar(smem_u32(&sh.piv_empty[buf]), ((uint32_t)(seq >> 1) & 1u) ^ 1u, kWaitPivFree, b);
        int pv = 0;
        if (lane < p.P && ok) {
            if (p.given) {
                pv = p.pivot_idx[(size_t)b * p.P + lane];
            } else {
                const int32_t *word = p.pv_word + (size_t)b * kMaxP + lane;
                const long long t0 = clock64();
                for (uint32_t spin = 0; (pv = (int)ld_word(word)) == kNoPivot; ++spin) {
                    __nanosleep(32);
                    if ((spin & 31u) == 31u) {
                        ok = !ctl.aborted();
                        if (ok && (unsigned long long)(clock64() - t0) > ctl.limit_cycles) {
                            ctl.give_up(kWaitPivots, b);
                            ok = false;
                        }
                        if (!ok) break;
                    }
                }
            }
        }
        if (!__all_sync(0xffffffffu, ok)) return;
        if (warp == 0 && lane < p.P) sh.pv[seq % kPvRing][lane] = pv;
        // (ranks beyond P repeat the last pivot: their products are not used)
        const int n_ch = it.na * 8;
        for (int i = warp; i < 8 * NT; i += kPivWarps) {
            const int row = __shfl_sync(0xffffffffu, pv, min(i, p.P - 1));
            const uint4 *src = p.keys + ((size_t)b * p.S + p.vis_offset + row) * (size_t)p.d8 + it.a0 * 8;
            const uint32_t dst = piv0 + (uint32_t)(buf * 8 * NT + i) * p.pitch;
            for (int k = lane; k < n_ch; k += 32)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + (uint32_t)k * 16u), "l"(src + k) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        mbar_arrive(smem_u32(&sh.piv_full[buf]));
        ++seq;
    }
}

// Second pass: 16 rows of the item per warp, all columns of the slice, NT of the sample's NTall tiles of 8 pivots (from tile n0 on).
// (32 pivots: one group 2.48, two groups 2.07 ms at 256 x 2880 x 4096: a dependent product returns after some 130 cycles, and a
// warp had 16 per atom to wait for.  16 pivots: one group 1.30, two 1.76 ms: a second group reads the rows from shared memory a
// second time.)
template <int NT, int NTall>
__device__ __forceinline__ void multiply(const Params &p, const Ctl &ctl, Shared &sh, uint32_t ring0, uint32_t piv0, int w, int n0)
{
    const int lane = threadIdx.x & 31;
    const int row = 16 * w + (lane & 15);                     // tile row whose 16 bytes this lane addresses for ldmatrix
    const uint32_t a_row = (uint32_t)row * 128u, a_sw = (uint32_t)(row & 7);
    const uint32_t b_lane = (uint32_t)(lane & 7) * p.pitch + (uint32_t)(lane >> 3) * 16u;
    const size_t part_item = (size_t)8 * NTall * kRows;
    Ring ring(p.n_st);
    int seq = -1, last_b = -1, k = 0;
    for (Items it(p); it.valid(); it.next(), ++k) {
        if (w == 0 && n0 == 0 && lane == 0) sh.at = it.b * p.n_vis + it.rg * kRows;
        if (it.b != last_b) {
            if (seq >= 0 && lane == 0) mbar_arrive(smem_u32(&sh.piv_empty[seq & 1])); // (the warp has converged at the item's end)
            ++seq;
            last_b = it.b;
            const bool ok = ctl.wait_bar(smem_u32(&sh.piv_full[seq & 1]), (uint32_t)(seq >> 1) & 1u, kWaitPiv, it.b);
            if (!__all_sync(0xffffffffu, ok)) return;
        }
        if (p.given && w == 0 && n0 == 0 && lane == 0) sh.pos = it.b * p.n_vis + it.rg * kRows;
        const uint32_t piv = piv0 + (uint32_t)((seq & 1) * 8 * NTall + 8 * n0) * p.pitch + b_lane;
        constexpr int kChains = NT == 1 ? 4 : 2; // independent sums per pivot tile
        float acc[NT][kChains][4];
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int h = 0; h < kChains; ++h)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[n][h][e] = 0.f;
        for (int a = 0; a < it.na; a += kAps) {
            const bool ok = ctl.wait_bar(smem_u32(&sh.full[ring.stage]), ring.phase, kWaitStage, it.b);
            if (!__all_sync(0xffffffffu, ok)) return;
            // All fragments of the stage (of an atom, with more pivots) are asked for before the first is multiplied, and the
            // stage is handed back before that too.
            const uint32_t tile0 = ring0 + (uint32_t)ring.stage * kStageBytes + a_row, pb0 = piv + (uint32_t)a * 128u;
            const bool two = a + 1 < it.na;
            constexpr int kTogether = NT == 1 ? 2 : 1; // atoms
#pragma unroll
            for (int h0 = 0; h0 < kAps; h0 += kTogether) {
                uint32_t af[kTogether][4][4], bf[kTogether][NT][2][4];
#pragma unroll
                for (int h = 0; h < kTogether; ++h) {
                    // (an atom that is not there: the first one again, its products are left out)
                    const uint32_t tile = tile0 + (two ? (uint32_t)(h0 + h) * kAtomBytes : 0u), pb = pb0 + (two ? (uint32_t)(h0 + h) * 128u : 0u);
#pragma unroll
                    for (int u = 0; u < 4; ++u) ldmatrix4(tile + ((((uint32_t)(2 * u) + (uint32_t)(lane >> 4)) ^ a_sw) << 4), af[h][u]);
#pragma unroll
                    for (int n = 0; n < NT; ++n) {
                        ldmatrix4(pb + (uint32_t)n * 8u * p.pitch, bf[h][n][0]);
                        ldmatrix4(pb + (uint32_t)n * 8u * p.pitch + 64u, bf[h][n][1]);
                    }
                }
                if (h0 + kTogether == kAps) {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&sh.empty[ring.stage]));
                }
#pragma unroll
                for (int h = 0; h < kTogether; ++h) {
                    if (h0 + h > 0 && !two) break;
#pragma unroll
                    for (int n = 0; n < NT; ++n) {
                        float (&c0)[4] = acc[n][kChains > 2 ? 2 * h : 0], (&c1)[4] = acc[n][kChains > 2 ? 2 * h + 1 : 1];
                        mma_bf16(c0, af[h][0], bf[h][n][0][0], bf[h][n][0][1]);
                        mma_bf16(c1, af[h][1], bf[h][n][0][2], bf[h][n][0][3]);
                        mma_bf16(c0, af[h][2], bf[h][n][1][0], bf[h][n][1][1]);
                        mma_bf16(c1, af[h][3], bf[h][n][1][2], bf[h][n][1][3]);
                    }
                }
            }
            ring.advance();
        }
        // the slice's share of the dot products: 8 consecutive rows of a pivot per 32 bytes
        float *dst = p.part + (((size_t)it.b * p.n_rg + it.rg) * p.nsl + it.sl) * part_item + (size_t)8 * n0 * kRows + 16 * w + (lane >> 2);
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float *o = dst + (size_t)(8 * n + 2 * (lane & 3) + e) * kRows;
                float v0 = acc[n][0][e] + acc[n][1][e], v1 = acc[n][0][2 + e] + acc[n][1][2 + e];
                if (kChains > 2) v0 += acc[n][kChains - 2][e] + acc[n][kChains - 1][e], v1 += acc[n][kChains - 2][2 + e] + acc[n][kChains - 1][2 + e];
                __stcg(o, v0);
                __stcg(o + 8, v1);
            }
        const int c = k % kCombWarps, slot = k / kCombWarps % kMail;
        const bool ok = ctl.wait_bar(smem_u32(&sh.mail_empty[c][slot]), ((uint32_t)(k / kCombWarps / kMail) & 1u) ^ 1u, kWaitMailFree, it.b);
        if (!__all_sync(0xffffffffu, ok)) return;
        __syncwarp(); // the lanes' stores are ordered before lane 0's release
        if (lane == 0) mbar_arrive(smem_u32(&sh.mail_full[c][slot]));
    }
    if (w == 0 && n0 == 0 && lane == 0) { // nothing holds the scorers back any more
        sh.at = 0x3fffffff;
        if (p.given) sh.pos = 0x3fffffff;
    }
}

// Watcher: how far the batch's pivots have got, for the scorers.  (Held back by the second pass of their own SM instead, the
// scorers of an SM with one item more than the others delayed everybody's pivots: 8 us between the first and the last SM.)  It
// looks at 32 samples at a time: one after the other, a load's 0.45 us per sample held batches of short ones back.
__device__ __forceinline__ void watch(const Params &p, const Ctl &ctl, Shared &sh)
{
    if (p.given) return;
    const int lane = threadIdx.x & 31;
    long long last = clock64();
    for (int b = 0; b < p.B;) {
        const bool there = b + lane >= p.B || (int32_t)ld_word(p.pv_word + (size_t)(b + lane) * kMaxP) != kNoPivot;
        const uint32_t missing = ~__ballot_sync(0xffffffffu, there);
        const int n = missing ? __ffs(missing) - 1 : 32; // samples in a row from b on whose pivots are known
        if (n > 0) {
            b += n;
            if (lane == 0) sh.pos = min(b, p.B) * p.n_vis;
            last = clock64();
        } else {
            __nanosleep(32);
            const bool dead = ctl.aborted() || (unsigned long long)(clock64() - last) > ctl.limit_cycles;
            if (__any_sync(0xffffffffu, dead)) return; // (the scorers' feeder reports it)
        }
    }
}

// Producer: the items' rows into the ring, whether their pivots are known yet or not.
__device__ __forceinline__ void produce(const Params &p, const Ctl &ctl, Shared &sh, uint32_t ring0, const CUtensorMap *tm)
{
    const int lane = threadIdx.x & 31;
    unsigned long long policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    Ring ring(p.n_st);
    long long issued = 0;
    bool ok = true;
    for (Items it(p); ok && it.valid(); it.next()) {
        // (rows beyond the vision block, or beyond the tensor: their products are not used)
        const int y = it.b * p.S + p.vis_offset + it.rg * kRows;
        for (int a = 0; a < it.na; a += kAps) {
            const int nh = min(kAps, it.na - a);
            const uint32_t full = smem_u32(&sh.full[ring.stage]);
            ok = ctl.wait_bar(smem_u32(&sh.empty[ring.stage]), ring.phase ^ 1u, kWaitStageFree, it.b);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            if (lane == 0) mbar_arrive_expect_tx(full, (uint32_t)nh * kAtomBytes);
            __syncwarp();
            if (lane < nh)
                tma_load_2d(ring0 + (uint32_t)ring.stage * kStageBytes + (uint32_t)lane * kAtomBytes, tm, (it.a0 + a + lane) * kAtomCols, y,
                            full, policy);
            ring.advance();
            ++issued;
        }
    }
    if (lane == 0) // the CTA must not exit while a copy is on its way, whatever became of the multipliers
        for (long long i = issued > p.n_st ? issued - p.n_st : 0; i < issued; ++i)
            ctl.wait_landed(smem_u32(&sh.full[i % p.n_st]), (uint32_t)((i / p.n_st) & 1));
}

// Combine: an item is counted once its shares are written; when all slices of its row group are, each of their SMs adds up one part
// in NSL of the group's similarities.  So from four slices on a lane has 16 values per pivot tile to fetch, all at once.
// (With the SM that counted last adding up the whole group, one sample of 576 tokens in 16 slices took 7 us from count to
// similarities, now 2.  Whole calls, us, by number of slices 1 / 2 / 4 / 8 / 16: 16 x 2880 x 1024 51.7 -> 49.3, 54.8 -> 52.4, 63.7 -> 59.4, 94 ->
// 74, 191 -> 117; 8 x 2880 x 4096 with 16 pivots from two on 108 -> 106, 98.2 -> 93.7, 115 -> 94, 202 -> 113; 4 x 1500 x 2048 with 32 55.4 -> 49.2, 53.4 ->
// 47.0, 67.6 -> 49.9, 103 -> 55.6.)
// A warp here waits for the other SMs' shares of its row group, and those for nothing but earlier groups: every SM takes its items
// in the groups' order.
template <int NT, int NSL>
__device__ __forceinline__ void combine(const Params &p, const Ctl &ctl, Shared &sh)
{
    constexpr int V = NSL >= 4 ? 16 / NSL : 4, H = 16 / NSL / V; // consecutive rows per lane and load; blocks of 32 V values per pivot tile
    // Blocks at a time: the same rows, every second pivot.  With one slice and two a lane has several blocks of 4 and 8 values, and one after
    // the other their loads are four and two rounds (whole calls, us, one at a time / all: 6 x 4518 x 1024 49.0 / 47.2, 35 x 1072 51.4 / 49.4, 47 x
    // 4329 172.9 / 169.9, 6 x 609 x 2048 30.0 / 28.8, 16 x 256 30.6 / 29.0, 61 x 1643 158.1 / 157.9; 1 pivot, 128 x 570 118.7 / 120.0).  Two pivot tiles
    // one at a time: 8 x 2880 x 4096 84.0 / 84.7, 39 x 911 x 2048 80.6 / 84.6.
    constexpr int U = NSL <= 2 && NT == 1 ? H : 1;
    constexpr int NTat = NT == 2 && U == 1 ? 2 : 1;              // pivot tiles at a time (registers)
    const int lane = threadIdx.x & 31, c = (int)(threadIdx.x >> 5) - kCombWarp0;
    const size_t part_item = (size_t)8 * NT * kRows;
    int seq = -1, last_b = -1, k = 0;
    auto late = [&](const unsigned long long *rec, int b, unsigned long long &v) { // the word may not be there yet when the pivots were given
        const long long t0 = clock64();
        for (uint32_t spin = 0; (v = ld_rec(rec)) == kNoRec; ++spin) {
            __nanosleep(100);
            if ((spin & 15u) == 15u) {
                if (ctl.aborted()) return false;
                if ((unsigned long long)(clock64() - t0) > ctl.limit_cycles) {
                    ctl.give_up(kWaitCombRec, b);
                    return false;
                }
            }
        }
        return true;
    };
    for (Items it(p); it.valid(); it.next(), ++k) {
        if (it.b != last_b) ++seq, last_b = it.b;
        if (k % kCombWarps != c) continue;
        const int slot = k / kCombWarps % kMail;
        bool ok = ctl.wait_bar(smem_u32(&sh.mail_full[c][slot]), (uint32_t)(k / kCombWarps / kMail) & 1u, kWaitMail, it.b);
        if (!__all_sync(0xffffffffu, ok)) return;
        const size_t group = (size_t)it.b * p.n_rg + it.rg;
        // release: the item's shares, written by the warps that filled the mailbox
        if (NSL > 1 && lane == 0 && !(p.withhold == 2 && group + it.sl == 0)) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p.cnt + group) : "memory");
        bool waited = NSL == 1;
        for (int h = 0; h < H; h += U) {
            const int f = it.sl * (512 / NSL) + (32 * h + lane) * V, i0 = f >> 6, r0 = f & 63; // (first) pivot of a tile and (first) row
            if (NT == 1 && __all_sync(0xffffffffu, i0 >= p.P)) continue; // none of it is wanted
            const int j = it.rg * kRows + r0;
            const unsigned long long *rec = p.rec + (size_t)it.b * p.n_vis;
            unsigned long long w[V], wp[NT][U];
            int pv[NT][U];
#pragma unroll
            for (int e = 0; e < V; ++e) w[e] = j + e < p.n_vis ? ld_rec(rec + j + e) : 0ull;
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = 8 * n + 2 * u + i0;
                    pv[n][u] = i < p.P ? sh.pv[seq % kPvRing][i] : 0;
                    const bool text = pv[n][u] < 0 || pv[n][u] >= p.n_vis;
                    wp[n][u] = text ? (unsigned long long)__float_as_uint(p.text_ssq[(size_t)it.b * p.P + i]) << 32 : ld_rec(rec + pv[n][u]);
                }
            if (!waited) { // acquire: the other slices' shares
                if (lane == 0) ok = ctl.wait_flag(p.cnt + group, kWaitShares, it.b, NSL);
                if (!__all_sync(0xffffffffu, ok)) return;
                __syncwarp(); // (every lane's loads come after lane 0's)
                waited = true;
            }
            const float *src = p.part + group * NSL * part_item + f;
            float *dst = p.sim + ((size_t)it.b * p.P + i0) * p.n_vis + j;
            float nr[V];
#pragma unroll
            for (int n0 = 0; n0 < NT; n0 += NTat) {
                float x[NTat][U][NSL][V];
#pragma unroll
                for (int n = 0; n < NTat; ++n)
#pragma unroll
                    for (int u = 0; u < U; ++u)
#pragma unroll
                        for (int s = 0; s < NSL; ++s) {
                            const float *at = src + s * part_item + (n0 + n) * 512 + u * 128;
                            float (&v)[V] = x[n][u][s];
                            if (8 * (n0 + n) + 2 * u + i0 >= p.P) { // not wanted
#pragma unroll
                                for (int e = 0; e < V; ++e) v[e] = 0.f;
                                continue;
                            }
                            if constexpr (V == 4)
                                asm volatile("ld.relaxed.gpu.global.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "l"(at) : "memory");
                            else if constexpr (V == 2)
                                asm volatile("ld.relaxed.gpu.global.v2.f32 {%0,%1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "l"(at) : "memory");
                            else
                                asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(v[0]) : "l"(at) : "memory");
                        }
                if (n0 == 0) {
#pragma unroll
                    for (int e = 0; e < V; ++e) {
                        if (w[e] == kNoRec) ok = ok && late(rec + j + e, it.b, w[e]);
                        nr[e] = sqrtf(__uint_as_float((uint32_t)(w[e] >> 32)));
                    }
#pragma unroll
                    for (int n = 0; n < NT; ++n)
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (wp[n][u] == kNoRec) ok = ok && late(rec + pv[n][u], it.b, wp[n][u]);
                    if (!__all_sync(0xffffffffu, ok)) return;
                }
#pragma unroll
                for (int n = 0; n < NTat; ++n)
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const float np = sqrtf(__uint_as_float((uint32_t)(wp[n0 + n][u] >> 32)));
#pragma unroll
                        for (int e = 0; e < V; ++e) { // dup = dot / (|pivot| |row|); a zero norm gives 0
                            float a = 0.f;
#pragma unroll
                            for (int s = 0; s < NSL; ++s) a += x[n][u][s][e]; // in slice order
                            const float den = np * nr[e];
                            if (8 * (n0 + n) + 2 * u + i0 < p.P && j + e < p.n_vis)
                                dst[(size_t)(8 * (n0 + n) + 2 * u) * p.n_vis + e] = den > 0.f ? a / den : 0.f;
                        }
                    }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sh.mail_empty[c][slot]));
    }
}

template <int NT>
__global__ void __launch_bounds__(threads(NT), 1) flow_kernel(const __grid_constant__ CUtensorMap tm, const Params p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ Shared sh;
    wait_for_previous();
    if (*p.status != 0) return; // an earlier kernel of this call failed (every CTA sees the same word: nobody waits)
    const uint32_t ring0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t slot0 = ring0 + (uint32_t)p.n_st * kStageBytes;
    const uint32_t piv0 = slot0 + (uint32_t)(kScoreWarps * p.n_slot) * kChunkBytes;
    const int warp = threadIdx.x >> 5;
    // whoever waits for something nearest to what is missing has the shortest limit, so that it is the one that reports it
    const unsigned long long limit = 2ull * p.wait_ns; // ns -> cycles at the highest SM clock: never shorter than asked
    const Ctl ctl{&sh.abort_flag, p.status, warp < kPivWarps ? limit + limit / 8 : warp == kProdWarp ? limit + limit / 2 : limit + limit / 4};
    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(smem_u32(&sh.full[s]), 1);
            mbar_init(smem_u32(&sh.empty[s]), mul_groups(NT) * kMulWarps);
        }
        for (int w = 0; w < kScoreWarps; ++w)
            for (int s = 0; s < kMaxSlots; ++s) mbar_init(smem_u32(&sh.chunk_full[w][s]), 1), mbar_init(smem_u32(&sh.chunk_empty[w][s]), 1);
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&sh.piv_full[s]), kPivWarps * 32);
            mbar_init(smem_u32(&sh.piv_empty[s]), mul_groups(NT) * kMulWarps);
        }
        for (int c = 0; c < kCombWarps; ++c)
            for (int s = 0; s < kMail; ++s) {
                mbar_init(smem_u32(&sh.mail_full[c][s]), mul_groups(NT) * kMulWarps);
                mbar_init(smem_u32(&sh.mail_empty[c][s]), 1);
            }
        sh.abort_flag = 0;
        sh.pos = sh.at = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if ((int)blockIdx.x >= p.n_stream) {
        if (threadIdx.x < kSel) select_pivots(p, Ctl{&sh.abort_flag, p.status, limit}, sh, smem_raw); // (selectors have no ring)
    } else if (warp >= kMulWarp1) {
        multiply<NT / mul_groups(NT), NT>(p, ctl, sh, ring0, piv0, warp - kMulWarp1, NT / mul_groups(NT));
    } else if (warp >= kFeedWarp) {
        feed(p, ctl, sh, slot0);
    } else if (warp == kWatchWarp) {
        watch(p, ctl, sh);
    } else if (warp >= kScoreWarp0) {
        score_rows(p, ctl, sh, slot0);
    } else if (warp < kPivWarps) {
        take_pivots<NT>(p, ctl, sh, piv0);
        // The next kernel may start: every SM is at its last items.  (Let go at the beginning, its CTAs crowded on the SMs that
        // were through first: 8 x 2880 x 4096, 16 pivots 94 -> 97 us.)
        let_next_start();
    } else if (warp < kMulWarp0 + kMulWarps) {
        multiply<NT / mul_groups(NT), NT>(p, ctl, sh, ring0, piv0, warp - kMulWarp0, 0);
    } else if (warp == kProdWarp) {
        produce(p, ctl, sh, ring0, &tm);
    } else {
        switch (p.nsl) {
        case 1: combine<NT, 1>(p, ctl, sh); break;
        case 2: combine<NT, 2>(p, ctl, sh); break;
        case 4: combine<NT, 4>(p, ctl, sh); break;
        case 8: combine<NT, 8>(p, ctl, sh); break;
        default: combine<NT, 16>(p, ctl, sh); break;
        }
    }
    __syncthreads(); // nobody leaves while a copy may still land in the CTA's shared memory
}

} // namespace flow
} // namespace dart
