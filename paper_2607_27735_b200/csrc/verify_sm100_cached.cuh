// Verification attention + Eq. 3 statistic for sm_100a, score-cache variant: one persistent,
// warp-specialised kernel on TMA (no multicast), tcgen05.mma with TMEM accumulators and
// mbarrier pipelines, in which K and V are each read exactly once from memory.
//
// Eq. 3 sums softmax PROBABILITIES over the window rows, so a key's contribution
// exp(s - LSE_row) needs every row's global normaliser, which is known only after all keys
// of the head were seen.  Instead of sweeping K twice, every CTA keeps the score tiles
// S^T = K Q^T of its share of the keys in tensor memory (512 columns per SM hold the output
// accumulator plus (512 - 2N) / N tiles of 128 keys x N rows):
//   P1   stream K, S^T tile -> TMEM (kept), per-row running (max, sum) -> this CTA's partial,
//        published to the CTAs that share the head;
//   P2a  stream V, P~ = exp2(S - lse_local) from the cached tile (needs nothing from other CTAs,
//        so the exchange of the partials hides behind it): O^T += V^T [P~_hi | P~_lo]^T on the
//        tensor cores (bf16 hi + lo split of P~ keeps the 2e-3 bar when one key takes most of the
//        mass); P~ replaces the scores in tensor memory;
//   --   the partials of the head's CTAs are combined into the row LSE (the only cross-CTA
//        dependency), by the publisher warp during P2a when few CTAs share the head;
//   P2b  cached P~ weighted per row with exp2(lse_local - LSE): column sums -> stats;
//   --   the accumulator, rescaled per row the same way, is this CTA's partial output.
// A unit (a group of KV heads of one (layer, sequence)) is cut so that a CTA's share of keys
// fits the cache; larger shares go to the two-sweep variant.
//
// TMEM tile layout: keys on the 128 lanes, the R = n_q * group query rows on the columns, so
// one thread owns one key: the statistic is a thread-local sum and the P1 row max/sum is
// thread-local state reduced once per unit.
//
// Roles (128 + 128 CG threads): warp 0 TMA producer, warp 1 tcgen05.mma issuer (+ TMEM alloc),
// warp 2 publisher (fences, counters, LSE combine), warp 3 reduces the per-CTA O partials (fixed
// order: deterministic), warps 4.. CG softmax warpgroups that split the columns.
//
// All CTAs must become co-resident (they wait on each other's partials): the grid never exceeds
// the SM count at one CTA per SM (see the launcher).  Every wait is bounded; on expiry the kernel
// records SPEC_ERR_TIMEOUT in the status word and drains.
#pragma once

#include <atomic>

#include "sm100_common.cuh"

namespace spec {
namespace sm100 {

namespace {


constexpr int kMaxCache = 32;
constexpr int kLsePubMax = 48;  // CTAs per head up to which the publisher warp alone combines the LSE partials

// Largest of the 32 lanes' values, on every lane.
__device__ __forceinline__ float warp_max_all(float x)
{
    float y;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(y) : "f"(x));
    return y;
}
// Sums over the 32 lanes of n columns per lane.  While the number of columns a lane carries is even, partners exchange
// halves (the lane with bit `o` set keeps the upper half), so the traffic halves at every step; an odd count is
// summed in place on both partners.  Afterwards a lane holds sum_final_n(n) columns starting at `col`, and lanes that
// differ only in the bits of sum_dupmask(n) hold the same ones.
__host__ __device__ constexpr int sum_final_n(int n)
{
    for (int o = 16; o >= 1; o >>= 1)
        if (n % 2 == 0) n /= 2;
    return n;
}
__host__ __device__ constexpr uint32_t sum_dupmask(int n)
{
    uint32_t d = 0;
    for (int o = 16; o >= 1; o >>= 1) {
        if (n % 2 == 0) n /= 2;
        else d |= (uint32_t)o;
    }
    return d;
}
template <int NHT, int n, int o>
__device__ __forceinline__ void sum_step(float (&l)[NHT], int lane, int& col)
{
    if constexpr (o >= 1) {
        if constexpr (n % 2 == 0) {
            constexpr int h = n / 2;
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int j = 0; j < h; ++j) {
                const float give = up ? l[j] : l[j + h], keep = up ? l[j + h] : l[j];
                l[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
            col += up ? h : 0;
            sum_step<NHT, h, o / 2>(l, lane, col);
        } else {
#pragma unroll
            for (int j = 0; j < n; ++j) l[j] += __shfl_xor_sync(0xffffffffu, l[j], o);
            sum_step<NHT, n, o / 2>(l, lane, col);
        }
    }
}

// Which problem a CTA works on in which unit.  A problem is one KV head of one (layer, sequence).  Teams of cph CTAs are
// sized for the longest context the call allows; a sequence whose share still fits the score cache on a half,
// a quarter or an eighth of a team runs on such a part, several problems side by side: a round costs a fixed
// 9-12 us of exchange and drain next to 1.5 us per key tile, so a 10 K sequence on a team sized for 64 K, or a
// 700-token one on a team sized for 6 K, would spend most of its time on the former.  The sequences are taken
// longest first (the lengths are in device memory, so every CTA sorts them for itself), the order of the parts
// alternates from unit to unit, and a class that would not fill half of a round joins the coarser one.
constexpr int kSortMax = 64;  // sequences, two per lane of the warp that sorts them; larger batches keep their order and whole teams
// What a CTA does in one unit.  The first units are worked out in the prologue, by a thread each, and every role reads
// them from shared memory: the arithmetic in each role's loop would be fetched from the instruction cache again every
// unit.  Later units (launches over many layers) take the places of old ones: the publisher warp writes kWorkAhead
// units ahead of its own and moves `limit`, the number of units that may be read.  An entry is neither read before it is
// written nor overwritten before it is read:
//  - the softmax warps keep step with the publisher: they start a unit after its arrival on `lse_ready` for the unit
//    before, when kWorkAhead - 1 units beyond theirs are in the table (they look up to three ahead), and it passes a
//    unit only after all of them have arrived on `pub_o` for it;
//  - the TMA, MMA and reduction warps skip units in which they have nothing to do, so nothing ties them to the
//    publisher: they do not pass `limit`, and say in `at` which unit they read next; the publisher waits for the
//    slowest of them before it overwrites an entry.  (None of them can need the publisher for a unit that far back.)
struct alignas(16) Work {
    int layer, b, h;
    uint16_t n, rank;  // CTAs of the problem (0: nothing to do in this unit), this one's number among them
    int T, t0, t1, prob;
    __device__ bool valid() const { return n != 0; }
    __device__ int cta0() const { return blockIdx.x - rank; }  // first CTA of the part
};
static_assert(sizeof(Work) == 32, "two vector loads");
constexpr int kWorkTab = 32;    // units in the table
constexpr int kWorkAhead = 24;
struct Sched {
    Work work[kWorkTab];
    int n_units, sorted;
    volatile int limit;
    volatile int at[3];         // next unit the TMA, MMA and reduction warps read (kept where n_units > kWorkTab)
    int unit0[kMaxClass + 1];   // first unit of a class
    int seq0[kMaxClass + 1];    // first sequence (in sorted order) of a class
    int len[kSortMax];          // as they come
    uint16_t ord[kSortMax];
};
static_assert(sizeof(Sched) <= 1536, "fits between the histogram and the row partials");

// A sequence's length as it is in memory now, clamped: a length outside [n_q, max_ctx_len] (the launch, the score cache
// and the output rows were sized for that range) is reported once the launch's dependency is resolved.
__device__ __forceinline__ int read_len(const FastParams& p, int b, int* raw = nullptr)
{
    const int t = __ldcg(p.a.ctx_len + b);
    if (raw) *raw = t;
    return min(max(t, p.a.n_q), p.a.max_ctx_len);
}

__device__ __noinline__ void put_work(const FastParams& p, Sched& sc, int unit)
{
    Work w;
    int f = 0;
    while (f + 1 < p.n_cls && unit >= sc.unit0[f + 1]) ++f;
    const int size = p.cls_size[f], subs = p.cls_subs[f], slots = p.HG * subs;
    const int team = fast_div(p, 2, blockIdx.x), local = blockIdx.x - team * p.cph;
    const int sub = div_by(p.cls_mul[f], p.cls_sh[f], local), rank = local - sub * size;
    const int slot = team * subs + sub;
    const int i = (unit - sc.unit0[f]) * slots + ((unit & 1) ? slots - 1 - slot : slot);
    bool valid = sub < subs && i >= 0;
    const int seq = valid ? fast_div(p, 0, i) : 0;
    const int rem = valid ? i - seq * (p.a.kv.n_layers * p.a.kv.n_kv_heads) : 0;
    const int layer = fast_div(p, 1, rem), h = rem - layer * p.a.kv.n_kv_heads;
    valid = valid && seq < sc.seq0[f + 1] - sc.seq0[f];
    const int at = sc.seq0[f] + (valid ? seq : 0);
    const int b = sc.sorted ? sc.ord[at] : at;
    w.T = sc.sorted ? sc.len[b] : read_len(p, b);
    const int nb = (w.T + kTile - 1) / kTile;
    const int n = min(size, nb);  // every CTA of a problem has a tile
    valid = valid && rank < n;
    // shares of nb / n tiles; n < size means a tile each
    w.t0 = !valid ? 0 : (n < size ? rank : div_by(p.cls_mul[f], p.cls_sh[f], rank * nb));
    w.t1 = !valid ? 0 : (n < size ? rank + 1 : div_by(p.cls_mul[f], p.cls_sh[f], (rank + 1) * nb));
    w.layer = layer;
    w.b = b;
    w.h = h;
    w.n = (uint16_t)(valid ? n : 0);
    w.rank = (uint16_t)rank;
    w.prob = (layer * p.a.kv.batch + b) * p.a.kv.n_kv_heads + h;
    sc.work[unit % kWorkTab] = w;
}
// Lengths, their order, classes and this CTA's first units: one warp.
__device__ __noinline__ void make_schedule(const FastParams& p, Sched& sc)
{
    const int lane = threadIdx.x & 31;
    const int B = p.a.kv.batch, LH = p.a.kv.n_layers * p.a.kv.n_kv_heads;
    const bool sorted = B <= kSortMax;
    int cnt[kMaxClass];
#pragma unroll
    for (int f = 0; f < kMaxClass; ++f) cnt[f] = 0;
    if (!sorted) cnt[0] = B;
#pragma unroll 1
    for (int i = 0; i < 2 && sorted; ++i) {
        const int b = lane + 32 * i;
        sc.len[b] = b < B ? read_len(p, b) : 0;
        if (B <= 32) break;
    }
    __syncwarp();
#pragma unroll 1
    for (int i = 0; i < 2 && sorted && 32 * i < B; ++i) {
        const int b = lane + 32 * i, T = sc.len[b];
        int before = 0;
#pragma unroll 1
        for (int j = 0; j < B; ++j) before += (sc.len[j] > T || (sc.len[j] == T && j < b)) ? 1 : 0;
        int f = -1;
        if (b < B) {
            sc.ord[before] = (uint16_t)b;
            const int nb = (T + kTile - 1) / kTile;
            f = p.n_cls - 1;
            while (f > 0 && p.cls_size[f] * p.n_cache < nb) --f;
        }
#pragma unroll
        for (int c = 0; c < kMaxClass; ++c) cnt[c] += __popc(__ballot_sync(0xffffffffu, f == c));
    }
#pragma unroll
    for (int f = kMaxClass - 1; f > 0; --f) {
        if (f < p.n_cls && 2 * cnt[f] * LH <= p.HG * p.cls_subs[f]) {
            cnt[f - 1] += cnt[f];
            cnt[f] = 0;
        }
    }
    // rounds of a class, a class per lane
    int mine = 0;
#pragma unroll
    for (int f = 0; f < kMaxClass; ++f) mine = lane == f ? cnt[f] : mine;
    const int slots = lane < p.n_cls ? p.HG * p.cls_subs[lane] : 1;
    const int rounds = (mine * LH + slots - 1) / slots;
    int u = 0, q = 0;
#pragma unroll
    for (int f = 0; f <= kMaxClass; ++f) {
        if (lane == 0) {
            sc.unit0[f] = u;
            sc.seq0[f] = q;
        }
        u += __shfl_sync(0xffffffffu, rounds, f);
        if (f < kMaxClass) q += cnt[f];
    }
    u -= __shfl_sync(0xffffffffu, rounds, kMaxClass);
    if (lane == 0) {
        sc.n_units = u;
        sc.sorted = sorted ? 1 : 0;
        sc.limit = min(u, kWorkTab);
        sc.at[0] = sc.at[1] = sc.at[2] = 0;
    }
    __syncwarp();
    static_assert(kWorkTab == 32, "a unit per lane");
    if (lane < u) put_work(p, sc, lane);
}

// The schedule of a single sequence whose heads are one round of whole teams (a call per layer of a long context): a unit
// that follows from the length.  The general form takes 5 k cycles from the start of a CTA, most of them first
// instruction fetches, and such a call has nothing to hide them behind: 2 rows over 2 K 14.9 us per launch with it.
__device__ __forceinline__ void one_unit(const FastParams& p, Sched& sc)
{
    int raw;
    Work w;
    w.T = read_len(p, 0, &raw);
    const int team = fast_div(p, 2, blockIdx.x), rank = blockIdx.x - team * p.cph;
    const int layer = fast_div(p, 1, team), h = team - layer * p.a.kv.n_kv_heads;
    const int nb = (w.T + kTile - 1) / kTile, n = min(p.cph, nb);
    const bool valid = rank < n;
    w.t0 = !valid ? 0 : (n < p.cph ? rank : fast_div(p, 2, rank * nb));
    w.t1 = !valid ? 0 : (n < p.cph ? rank + 1 : fast_div(p, 2, (rank + 1) * nb));
    w.layer = layer;
    w.b = 0;
    w.h = h;
    w.n = (uint16_t)(valid ? n : 0);
    w.rank = (uint16_t)rank;
    w.prob = team;
    if ((threadIdx.x & 31) == 0) {
        if (raw != w.T) set_status(p.status, SPEC_ERR_BAD_INDEX);
        sc.work[0] = w;
        sc.n_units = 1;
        sc.limit = 1;
    }
}

__device__ __forceinline__ Work get_work(const Sched& sc, int unit) { return sc.work[unit % kWorkTab]; }
// Waits until a word of the schedule is above `x` (bounded like every wait).
__device__ __noinline__ bool wait_above(const volatile int& word, int x, const Ctl& c)
{
    const long long t0 = clock64();
    while (word <= x) {
        __nanosleep(200);
        if (*c.abort_flag) return false;
        if (clock64() - t0 > c.limit) {
            report_timeout(c, 37);
            return false;
        }
    }
    __threadfence_block();
    return true;
}

// The waits of this kernel poll the abort flag and carry no clock of their own, because each of them ends at a timed one.
// What comes from a copy or the tensor cores passes through the MMA warp, which never blocks and whose idle timer runs
// until it has issued its last product; after that the softmax warps and the publisher wait for one another and,
// through the publisher, for other CTAs' counters, which is timed where it stands (counter_wait, like the waits for
// the work table).  Either raises the flag when the limit runs out.  (The count of tries is no bound in time, the
// hardware may suspend a try: it only ends what a mistake in these lines would leave waiting.)  A clock inlined at each of
// the thirty sites made the function 12 KB longer, and code that does not fit the instruction cache is fetched again
// every unit; a timer in the MMA warp until every other warp is through cost 0.2 us per launch (13.1 -> 13.3 at 2 K).
constexpr uint32_t kMaxTries = 1u << 27;
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, const Ctl& c)
{
    for (uint32_t n = 0; !mbar_try_wait(bar, parity);) {
        if (*c.abort_flag) return false;
        if (++n > kMaxTries) *c.abort_flag = 1;
    }
    return true;
}
// Barrier among the softmax warps, on an mbarrier so that the wait can be abandoned.
__device__ __forceinline__ bool warps_sync(uint32_t bar, uint32_t& n, const Ctl& c)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(bar);
    return bar_wait(bar, n++ & 1, c);
}

struct CBars {  // mbarrier addresses (shared space)
    uint32_t slot_full, slot_empty, q_full, q_empty, s_full, s_free, p_full, p_empty, o_full, o_empty, sm_sync,
        pub_p1, pub_o, lse_ready, raw_full, raw_empty, q_ready;
};

// NC = score columns per softmax warpgroup, CG = number of such warpgroups (R <= NC * CG <= N):
// more, narrower warpgroups hide the latency of the serial softmax sections.
// LP: the publisher warp combines the LSE partials (few CTAs per head); otherwise the softmax warps do.
// PH: one Eq. 3 score per attention head (stats [.., n_q_heads, stride]) instead of per KV head,
// for groups of at most 8 heads (a short statistic pass when the group size divides 8).
// SC: per-(layer, KV head) scales of K and V (an 8-bit cache, expanded to bf16 beforehand or here).
// F8: the cache holds e4m3 bytes.  TMA brings a tile's bytes (16 KB) into a ring of raw stages; the
// softmax warps expand a tile one or two places ahead into the operand slot while the tensor cores
// work on the current one (cvt.rn.f16x2.e4m3x2: every e4m3 value is an fp16 value).  Both products then run on
// fp16 operands: Q is converted once per unit in shared memory, P~ is split into an fp16 rounding of
// 2^14 P~ and the fp16 rounding of 2^11 times its remainder (the two accumulator halves are added with
// that weight in the epilogue); the powers of two join the scales.
// WR: a tile lies in its slot as whole rows, the two 1 KB halves of eight rows side by side (see encode_kv_map_rows); else
// its two 64-wide halves lie 16 KB apart.  A template parameter, since the loops that the distances go into do not bear them
// as run-time values: the MMA warp's descriptors (eight sequences of 9-66 K on 64-token pages 244 -> 248 us, over an 8-bit cache 323 ->
// 330) and the clearing of the ragged tail's rows (80 score columns: 315 -> 350 us for two sequences of 40 K).
template <int NC, int CG, bool LP, bool PH, bool SC, bool F8, bool WR>
__global__ void __launch_bounds__(128 + 128 * CG, 1)
verify_cached_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                     const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ FastParams p)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sgen = smem_raw + (sbase - smem_u32(smem_raw));  // generic pointer to the aligned base

    constexpr int NH = NC;                       // columns per thread
    constexpr int kBlock = 128 + 128 * CG;       // threads per CTA
    constexpr int kSW = 4 * CG;                  // softmax warps
    constexpr int kHalf = WR ? 1024 : 16384;     // bytes from a row's one half to its other
    constexpr int kGroup = WR ? 2048 : 1024;     // and from eight rows to the next eight
    const int N = p.N, R = p.R, G = p.G;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q_bytes = N * 256;                       // one Q buffer: 2 halves x N rows x 128 B
    const int p_bytes = 2 * N * 256;                   // one P buffer: [hi | lo] rows, 8-row blocks x 128 keys x 16 B

    const uint32_t s_slots = sbase;
    const uint32_t s_raw = s_slots + p.n_slots * kSlotBytes;  // F8: n_raw stages of 16 KB
    const uint32_t s_q = s_raw + (F8 ? p.n_raw * 16384 : 0);
    const uint32_t s_p = s_q + q_bytes;                // one Q buffer: the next unit's Q lands after this unit's last QK^T
    const uint32_t s_misc = s_p + p.p_bufs * p_bytes;
    uint8_t* misc = sgen + (s_misc - sbase);
    CBars B;
    {
        uint32_t o = s_misc;
        B.slot_full = o; o += 8 * 8;
        B.slot_empty = o; o += 8 * 8;
        B.q_full = o; o += 16;
        B.q_empty = o; o += 16;
        B.s_full = o; o += 8 * kMaxCache;
        B.s_free = o; o += 8 * kMaxCache;
        B.p_full = o; o += 32;  // up to four P buffers
        B.p_empty = o; o += 32;  // four: indexed by tile sequence number mod 4 (see the P2 loop)
        B.o_full = o; o += 8;
        B.o_empty = o; o += 8;
        B.sm_sync = o; o += 8;
        B.pub_p1 = o; o += 8;   // the last softmax warp stored this CTA's (max, sum) partial
        B.pub_o = o; o += 8;    // every softmax warp stored its share of the output partial
        B.lse_ready = o; o += 8;  // the publisher warp left the row LSE and the rescale factors in shared memory
        B.raw_full = o; o += 32;  // F8: a tile's bytes have landed in a raw stage
        B.raw_empty = o; o += 32; // F8: every softmax warp has expanded its part of the stage
        B.q_ready = o; o += 8;    // F8: Q is fp16 in shared memory
    }
    int* roff_s = reinterpret_cast<int*>(misc + 1024);                    // [128] offset of a row in the output, from row 0
    float* loc_s = reinterpret_cast<float*>(misc + 1024 + 512);           // [128] CTA-local row LSE
    float* fac_s = reinterpret_cast<float*>(misc + 2048);                 // [128] exp2(local - global)
    uint32_t* hist_s = reinterpret_cast<uint32_t*>(misc + 2560);          // [1024] packed 16-bit counts of score bins, 4 KB
    Sched& sc = *reinterpret_cast<Sched*>(misc + 6656);
    float* red_m = reinterpret_cast<float*>(misc + 8192);                 // [kSW warps][NC], <= 2 KB
    float* red_l = red_m + 512;                                           // the same
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(misc + 12288);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    Ctl ctl{abort_flag, p.status, p.wait_limit};

    if (threadIdx.x < kMaxCache) {  // one region's pair of barriers per thread
        mbar_init(B.s_full + 8 * threadIdx.x, 1);
        mbar_init(B.s_free + 8 * threadIdx.x, 4);
    } else if (threadIdx.x < kMaxCache + 8) {
        const int i = threadIdx.x - kMaxCache;
        if (i < p.n_slots) {
            mbar_init(B.slot_full + 8 * i, F8 ? kSW : 1);  // F8: filled by the softmax warps, not by TMA
            mbar_init(B.slot_empty + 8 * i, 1);
        }
        if (F8 && i < 4) {
            mbar_init(B.raw_full + 8 * i, 1);
            mbar_init(B.raw_empty + 8 * i, kSW);
        }
        if (i < 2) {
            mbar_init(B.q_full + 8 * i, 1);
            mbar_init(B.q_empty + 8 * i, 1);
        }
        if (i < 4) {
            mbar_init(B.p_full + 8 * i, kSW);
            mbar_init(B.p_empty + 8 * i, 1);
        }
    } else if (threadIdx.x == kMaxCache + 8) {
        mbar_init(B.o_full, 1);
        mbar_init(B.o_empty, kSW);
        mbar_init(B.sm_sync, kSW);
        mbar_init(B.pub_p1, 1);
        mbar_init(B.pub_o, kSW);
        mbar_init(B.lse_ready, 1);
        if (F8) mbar_init(B.q_ready, kSW);
        *abort_flag = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // zero the Q buffers once: rows R..N-1 are padding the TMA never writes
    for (int i = threadIdx.x; i < q_bytes / 16; i += kBlock)
        *reinterpret_cast<uint4*>(sgen + (s_q - sbase) + 16 * i) = make_uint4(0, 0, 0, 0);
    if (p.a.hist)
        for (int i = threadIdx.x; i < kScoreBins / 2; i += kBlock) hist_s[i] = 0u;
    if (NC * CG < N) {  // row blocks of the P operand that no warpgroup has: zero once (hi and lo part of every buffer)
        const int per = (N - NC * CG) / 8 * 128;  // 16-byte vectors of one part
#pragma unroll 1
        for (int i = threadIdx.x; i < 2 * p.p_bufs * per; i += kBlock) {
            const int part = i / per, k = i - part * per, j = NC * CG / 8 + (k >> 7) + (part & 1) * (N / 8);
            *reinterpret_cast<uint4*>(sgen + (s_p - sbase) + (part >> 1) * p_bytes + j * 2048 + (k & 127) * 16) =
                make_uint4(0u, 0u, 0u, 0u);
        }
    }
    if (p.D == 64) {  // the upper 64-wide half of every tile slot is never loaded: zero rows of V^T (and of K)
        for (int i = threadIdx.x; i < p.n_slots * 1024; i += kBlock)
            *reinterpret_cast<uint4*>(sgen + (s_slots - sbase) + (i >> 10) * kSlotBytes + 16384 + 16 * (i & 1023)) =
                make_uint4(0, 0, 0, 0);
    }
    if (threadIdx.x < R) {
        const int j = fast_div(p, 3, threadIdx.x);
        roff_s[threadIdx.x] = (j * p.a.kv.n_q_heads + (threadIdx.x - j * G)) * p.D;
    }
    for (int r = R + threadIdx.x; r < 128; r += kBlock) {  // padded rows: P = 0
        loc_s[r] = 1.0e30f;
        fac_s[r] = 0.f;
    }
    fence_proxy_async();
    // The schedule is made from the lengths as they are now, before the launch's dependency is resolved (the kernel
    // before may still be writing them: they are read again and compared after the wait below): its latencies and
    // first instruction fetches then hide behind the previous launch's end.
    if (warp == 0 && !p.one_round) make_schedule(p, sc);
    if (warp == 3 && lane < 3)
        asm volatile("prefetch.tensormap [%0];" ::"l"(lane == 0 ? &tm_k : (lane == 1 ? &tm_v : &tm_q)) : "memory");
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // Programmatic dependent launch: this kernel's prologue above may run while the previous
    // kernel in the stream drains; nothing before this point touches global memory the stream
    // produces (the workspace is shared with the previous call).
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;
    if (warp == 0 && p.one_round) {
        one_unit(p, sc);
    } else if (warp == 0) {
        // the schedule stands if the lengths are what they were when it was made; lengths out of range are reported
        const bool sorted = p.a.kv.batch <= kSortMax;
        bool same = sorted;
        for (int b = lane; b < p.a.kv.batch; b += 32) {
            int raw;
            const int T = read_len(p, b, &raw);
            if (raw != T) set_status(p.status, SPEC_ERR_BAD_INDEX);
            if (sorted) same = same && sc.len[b] == T;
        }
        if (!__all_sync(0xffffffffu, same)) make_schedule(p, sc);
    }
    __syncthreads();
    const int U = sc.n_units;
    const uint32_t col_o = 0, col_s = 2 * N;  // O^T (hi | lo) first, then the cached S^T tiles

    if (warp == 0) {
        // =========================== TMA producer ===========================
        uint32_t ring = 0, ring_ph = 0, qn = 0;  // next slot (F8: raw stage), its phase; Q buffers filled
        const int boxes = p.boxes, box_rows = p.box_rows;
        const uint32_t box_bytes = box_rows * (WR ? 256 : 128);
        const int halves = p.D / 64;  // 64-wide halves of the head dimension
        bool ok = true;
        // A tile's boxes, one per lane: at most 16 of 8 whole rows (WR), or that many for either half of the head dimension.
        // F8: the tile's bytes (128 per key) go to a raw stage, and the softmax warps expand them into a slot.
        // The page table is read before the wait for a free slot: its latency (a trip to L2 per tile, which bounded
        // the stream of 16-token pages) hides behind that wait.
        auto load_tile = [&](const CUtensorMap* map, const Work& sg, int tile) -> bool {
            const int key0 = tile * kTile;
            // boxes that hold at least one key < T (pages past the context may not exist)
            const int n_box = min(boxes, (sg.T - key0 + box_rows - 1) / box_rows);
            const int n_ops = F8 || WR ? n_box : halves * n_box;
            const int half = !F8 && !WR && lane >= n_box ? 1 : 0, bx = lane - half * n_box;
            const int pos = key0 + bx * box_rows;
            const int page = page_of(p.a.kv, pos), slot_in_page = pos - page * p.a.kv.page_size;
            int phys = 0;
            if (lane < n_ops) {
                phys = p.a.kv.page_table ? __ldg(p.a.kv.page_table + (int64_t)sg.b * p.a.kv.max_pages + page)
                                         : sg.b * p.a.kv.max_pages + page;
                if (phys < 0 || phys >= p.n_pages) {
                    set_status(p.status, SPEC_ERR_BAD_INDEX);
                    phys = 0;
                }
            }
            const uint32_t s = ring, ph = ring_ph;
            if (++ring == (uint32_t)(F8 ? p.n_raw : p.n_slots)) {
                ring = 0;
                ring_ph ^= 1;
            }
            const uint32_t full = (F8 ? B.raw_full : B.slot_full) + 8 * s;
            bool got = true;
            if (lane == 0) {  // one lane polls
                got = bar_wait((F8 ? B.raw_empty : B.slot_empty) + 8 * s, ph ^ 1, ctl);
                if (got) mbar_expect_tx(full, (uint32_t)n_ops * box_bytes);
            }
            if (!__shfl_sync(0xffffffffu, got ? 1 : 0, 0)) return false;
            if (WR && lane < n_ops)  // (a box is a page: see copy_whole_rows)
                tma_load_5d(s_slots + s * kSlotBytes + bx * box_bytes, map, full, 0, 0, 0, 0,
                            sg.layer * p.row_layer + phys * p.row_page + sg.h * p.row_head, kEvictFirst);
            if (!WR && lane < n_ops)
                tma_load_5d((F8 ? s_raw + s * 16384 : s_slots + s * kSlotBytes + half * 16384) + bx * box_bytes, map, full,
                            half * 64, slot_in_page, sg.h * p.row_head, phys * p.row_page, sg.layer * p.row_layer, kEvictFirst);
            __syncwarp();
            return true;
        };
        for (int u = 0; u < U && ok; ++u) {
            if (U > kWorkTab) {  // (see Sched)
                ok = __all_sync(0xffffffffu, wait_above(sc.limit, u, ctl));
                if (!ok) break;
                if (lane == 0) sc.at[0] = u;
            }
            const Work sg = get_work(sc, u);
            if (!sg.valid()) continue;
            const uint32_t qph = qn & 1;
            ++qn;
            ok = bar_wait(B.q_empty, qph ^ 1, ctl);
            if (!ok) break;
            if (lane == 0) {
                mbar_expect_tx(B.q_full, (uint32_t)halves * R * 128);
                const int row0 = (sg.layer * p.a.kv.batch + sg.b) * p.a.n_q;
                tma_load_3d(s_q, &tm_q, B.q_full, 0, sg.h * G, row0);
                if (halves == 2) tma_load_3d(s_q + N * 128, &tm_q, B.q_full, 64, sg.h * G, row0);
            }
            __syncwarp();
            for (int t = sg.t0; t < sg.t1 && ok; ++t) ok = load_tile(&tm_k, sg, t);
            for (int t = sg.t0; t < sg.t1 && ok; ++t) ok = load_tile(&tm_v, sg, t);
        }
        if (!ok) {  // let copies in flight land before the CTA's shared memory is released
            const long long t0 = clock64();
            while (clock64() - t0 < 400000ll) __nanosleep(1000);
        }
    } else if (warp == 1) {
        // =========================== MMA issuer ===========================
        if (lane == 0) {
            // operand formats (bits 7-9 and 10-12): 1 = bf16, 0 = fp16 (F8: both products on fp16 operands)
            const uint32_t ab_fmt = F8 ? 0u : ((1u << 7) | (1u << 10));
            const uint32_t idesc_qk = (1u << 4) | ab_fmt | ((uint32_t)(N >> 3) << 17) | ((128u >> 4) << 24);
            // O^T += V^T [P_hi | P_lo]^T : A = V^T and B = P^T both MN-major, N = 2 * rows
            const uint32_t idesc_pv = (1u << 4) | ab_fmt | (1u << 15) | (1u << 16) |
                                      ((uint32_t)((2 * N) >> 3) << 17) | ((128u >> 4) << 24);
            // Descriptors of slot 0's tiles: a place further on in shared memory only adds to them.  What this thread does
            // between two products counts: with the descriptors built anew for each, eight sequences of 9-66 K take 242 us
            // instead of 235; with head_dim asked before each of the eight instead of once, 240 (head_dim 64: 238 instead of 222).
            const uint64_t k_desc = desc_kmajor(s_slots, kGroup);
            const uint64_t v_desc = desc_mnmajor(s_slots, kHalf, kGroup);
            // Two independent queues, issued in whichever order their inputs become ready: the
            // QK^T tiles of unit u+1 may overtake the P V tiles of unit u that still wait for P.
            struct Queue {
                int u = -1, c = 0, n_t = 0;   // unit, its tile, its tiles
                uint32_t slot = 0, ph = 0;    // ring position of the tile and the slot's phase
                int at = 0;                   // the tile's number among all tiles, K and V
                bool seek = true, done = false;
            } qq, pq;
            // slots of a unit: its K tiles, then its V tiles
            auto skip = [&](Queue& c, int n) {
                c.slot += n;
                c.at += n;
                while (c.slot >= (uint32_t)p.n_slots) {
                    c.slot -= p.n_slots;
                    c.ph ^= 1;
                }
            };
            auto seek = [&](Queue& c, bool v) {  // on to the next unit with work, as far as the table goes
                skip(c, v ? 0 : c.n_t);          // past the V tiles of the unit left behind
                c.n_t = 0;
                while (c.seek && c.u + 1 < U && c.u + 1 < sc.limit) {
                    __threadfence_block();
                    ++c.u;
                    const Work sg = get_work(sc, c.u);
                    if (sg.valid()) {
                        c.n_t = sg.t1 - sg.t0;
                        c.c = 0;
                        c.seek = false;
                        if (v) skip(c, c.n_t);  // past the K tiles
                    }
                }
                if (U > kWorkTab) sc.at[1] = min(qq.u, pq.u) + 1;
                c.done = c.seek && c.u + 1 >= U;
            };
            uint32_t sfree_par = 0;  // per cache region: parity of the next "region free" phase
            uint32_t region = 0;     // of the next K Q^T tile: regions are taken in turn, across units
            uint32_t pb = 0, pph = 0, pe = 0, o_phase = 0, q_phase = 0;
            bool ok = true;
            auto qk_ready = [&]() -> bool {
                // A slot's phase only tells its last two fills apart, so the tile that had the slot before must have been
                // used: with regions free for the next unit, K Q^T would otherwise take a V tile still in flight
                // for its K tile.
                if (qq.at >= pq.at + p.n_slots) return false;
                if (qq.c == 0 && !mbar_test_wait(F8 ? B.q_ready : B.q_full, q_phase)) return false;
                if (!mbar_test_wait(B.slot_full + 8 * qq.slot, qq.ph)) return false;
                return mbar_test_wait(B.s_free + 8 * region, ((sfree_par >> region) & 1) ^ 1);
            };
            auto issue_qk = [&]() {
                sfree_par ^= 1u << region;
                tc_fence_after();
                const uint64_t k_tile = k_desc + qq.slot * (kSlotBytes >> 4);
                const uint32_t d_s = tmem_base + col_s + region * N;
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    tc_mma(d_s, k_tile + ks * 2, desc_kmajor(s_q + ks * 32), idesc_qk, ks ? 1u : 0u);
                if (WR || p.D == kD) {  // (head_dim 64: the first four 16-wide steps only)
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        tc_mma(d_s, k_tile + ((kHalf >> 4) + ks * 2), desc_kmajor(s_q + N * 128 + ks * 32), idesc_qk, 1u);
                }
                tc_commit(B.s_full + 8 * region);
                tc_commit(B.slot_empty + 8 * qq.slot);
                if (++region == (uint32_t)p.n_cache) region = 0;
                skip(qq, 1);
                if (++qq.c == qq.n_t) {
                    tc_commit(B.q_empty);  // last use of this Q
                    q_phase ^= 1;
                    qq.seek = true;
                }
            };
            auto pv_ready = [&]() -> bool {
                if (!mbar_test_wait(B.p_full + 8 * pb, pph)) return false;
                if (!mbar_test_wait(B.slot_full + 8 * pq.slot, pq.ph)) return false;
                return pq.c != 0 || mbar_test_wait(B.o_empty, o_phase ^ 1);
            };
            auto issue_pv = [&]() {
                tc_fence_after();
                const uint64_t v_tile = v_desc + pq.slot * (kSlotBytes >> 4);
                const uint32_t p_addr = s_p + pb * p_bytes;
                const uint32_t d_o = tmem_base + col_o;
#pragma unroll
                for (int ks = 0; ks < 8; ++ks) {
                    const uint64_t a = v_tile + ks * (2 * kGroup >> 4);
                    const uint64_t b = desc_mnmajor_nosw(p_addr + ks * 256);
                    tc_mma(d_o, a, b, idesc_pv, (pq.c == 0 && ks == 0) ? 0u : 1u);
                }
                tc_commit(B.slot_empty + 8 * pq.slot);
                tc_commit(B.p_empty + 8 * pe);
                pe = (pe + 1) & 3;
                if (++pb == (uint32_t)p.p_bufs) {
                    pb = 0;
                    pph ^= 1;
                }
                skip(pq, 1);
                if (++pq.c == pq.n_t) {
                    tc_commit(B.o_full);
                    o_phase ^= 1;
                    pq.seek = true;
                }
            };
            long long t_idle = clock64();
            uint32_t spins = 0;
            while (ok && !(qq.done && pq.done)) {
                bool progressed = false;
                if (qq.seek && !qq.done) seek(qq, false);
                if (pq.seek && !pq.done) seek(pq, true);
                // a unit's P V tiles can only follow its own K Q^T tiles
                if (!pq.seek && (qq.seek || qq.u > pq.u) && pv_ready()) {
                    issue_pv();
                    progressed = true;
                }
                if (!qq.seek && qk_ready()) {
                    issue_qk();
                    progressed = true;
                }
                if (progressed) {
                    spins = 0;
                    continue;
                }
                // (No sleep here.  With 40 ns between two looks, 25 shapes of 8 to 128 rows on pages of 16 tokens to whole contexts:
                // 0 to 0.9 % slower a launch (85 rows 78.85 -> 79.6 us, 68 rows at 40 K 314.4 -> 316.3, 32 K alone 39.9 -> 40.2), over an
                // 8-bit cache -0.5 to +1.6 %; runs of one side differ by 0.3 %, those of a few thousand keys by 1 %.  On 8-token
                // pages, whose copies bound the launch, -0.3 to +0.8 %.)
                if ((++spins & 63u) == 0) {
                    if (spins == 64) t_idle = clock64();
                    if (*ctl.abort_flag) ok = false;
                    else if (clock64() - t_idle > ctl.limit) {
                        report_timeout(ctl, 16);
                        ok = false;
                    }
                }
            }
        }
        __syncwarp();
    } else if (warp == 2) {
        // =========================== publisher warp ===========================
        // Makes this CTA's partials visible to the other CTAs (device-scope fence + counter), so
        // that no softmax warp ever waits for that round trip: they only arrive on a CTA barrier.
        // It also combines the (max, sum) partials of the CTAs that share the head into the row
        // LSE while the softmax warps are busy with the P V pass.
        bool ok = true;
        for (int unit = 0; unit < U && ok; ++unit) {
            const Work sg = get_work(sc, unit);
            const bool shared = sg.n > 1;  // a problem of one CTA has nothing to exchange
            if (U > kWorkTab && unit + kWorkAhead >= kWorkTab && unit + kWorkAhead < U) {
                if (lane == 0) {  // the place of unit + kWorkAhead - kWorkTab, once everybody is past it
                    for (int r = 0; r < 3 && ok; ++r) ok = wait_above(sc.at[r], unit + kWorkAhead - kWorkTab, ctl);
                    if (ok) {
                        put_work(p, sc, unit + kWorkAhead);
                        __threadfence_block();
                        sc.limit = unit + kWorkAhead + 1;
                    }
                }
                ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                if (!ok) break;
            }
            int* c_p1 = p.counters + sg.prob;
            int* c_o = c_p1 + p.n_counters / 2;
            if (unit >= kRing - 1) {
                // the partials' places are used again by the next unit: their readers must be done (they have been
                // for two units, as a rule)
                const Work old = get_work(sc, unit - (kRing - 1));
                if (old.n > 1) {
                    if (lane == 0)
                        ok = counter_wait(p.counters + old.prob, 2 * old.n, ctl, 36);
                    ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                    if (!ok) break;
                }
            }
            if (lane == 0) {
                ok = bar_wait(B.pub_p1, unit & 1, ctl);
                if (ok && shared) {
                    __threadfence();
                    atomicAdd(c_p1, 1);
                }
            }
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            if (!ok) break;
            if (LP && shared) {
                // ---- row LSE from the partials of the CTAs that share this head ----
                if (lane == 0) ok = counter_wait(c_p1, sg.n, ctl, 31);
                ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;  // lane 0's acquire, then warp-wide
                if (!ok) break;
                const float2* src = p.ml_part + ((int64_t)(unit % kRing) * gridDim.x + sg.cta0()) * R;
                // two lanes per row, 16 rows per pass: each lane folds every other partial, 20 loads in flight
                const int sub = lane & 1;
                for (int r0 = 0; r0 < R; r0 += 16) {
                    const int r = r0 + (lane >> 1);
                    float M = -1.0e30f, Ls = 0.f;
                    if (r < R) {
                        for (int k0 = sub; k0 < sg.n; k0 += 40) {
                            float2 x[20];
                            const float2* q = src + (int64_t)k0 * R + r;
                            const int n_ld = (sg.n - k0 + 1) >> 1;  // partials k0, k0 + 2, ... below n
#pragma unroll
                            for (int u = 0; u < 20; ++u) {
                                x[u] = make_float2(-1.0e30f, 0.f);
                                if (u < n_ld) x[u] = __ldcg(q);
                                q += 2 * R;
                            }
                            float Mn = M;
#pragma unroll
                            for (int u = 0; u < 20; ++u) Mn = fmaxf(Mn, x[u].x);
                            Ls *= ex2(M - Mn);
#pragma unroll
                            for (int u = 0; u < 20; ++u) Ls = fmaf(x[u].y, ex2(x[u].x - Mn), Ls);
                            M = Mn;
                        }
                    }
                    const float M2 = __shfl_xor_sync(0xffffffffu, M, 1);
                    const float L2 = __shfl_xor_sync(0xffffffffu, Ls, 1);
                    const float Mn = fmaxf(M, M2);
                    Ls = Ls * ex2(M - Mn) + L2 * ex2(M2 - Mn);
                    M = Mn;
                    if (sub == 0 && r < R) {
                        const float lse2 = M + log2f(Ls);
                        const float loc = loc_s[r];
                        fac_s[r] = loc < 1.0e29f ? ex2(loc - lse2) : 0.f;  // local -> global normaliser
                        if (sg.rank == 0 && p.a.lse) {
                            const int j = r / G, g = r - j * G;
                            const int64_t row = (((int64_t)sg.layer * p.a.kv.batch + sg.b) * p.a.n_q + j) * p.a.kv.n_q_heads + sg.h * G + g;
                            p.a.lse[row] = lse2 * 0.69314718055994530942f;
                        }
                    }
                }
            }
            // signalled for every unit, empty ones too: the softmax warps wait for it before they go
            // on, so they are never more than one barrier phase ahead of this warp
            __syncwarp();
            if (lane == 0) mbar_arrive(B.lse_ready);
            if (lane == 0) {
                ok = bar_wait(B.pub_o, unit & 1, ctl);
                if (ok && shared) {
                    __threadfence();
                    atomicAdd(c_o, 1);
                }
            }
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
        }
    } else if (warp == 3) {
        // =========================== O reduction warp ===========================
        const int tid = lane;
        bool ok = true;
        for (int unit = 0; unit < U && ok; ++unit) {
            if (U > kWorkTab) {  // (see Sched)
                ok = __all_sync(0xffffffffu, wait_above(sc.limit, unit, ctl));
                if (!ok) break;
                if (lane == 0) sc.at[2] = unit;
            }
            const Work sg = get_work(sc, unit);
            if (sg.n <= 1) continue;  // (a problem of one CTA: the softmax warps store the output)
            int* c_p1 = p.counters + sg.prob;
            int* c_o = c_p1 + p.n_counters / 2;
            if (lane == 0) ok = counter_wait(c_o, sg.n, ctl, 30);
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
            if (!ok) break;
            const int E4 = R * kD / 4;
            const int lo = sg.rank * E4 / sg.n, hi = (sg.rank + 1) * E4 / sg.n;
            const float4* src = reinterpret_cast<const float4*>(
                p.o_part + ((int64_t)(unit % kRing) * gridDim.x + sg.cta0()) * R * kD);
            const int64_t out0 = ((int64_t)sg.layer * p.a.kv.batch + sg.b) * p.a.n_q * p.a.kv.n_q_heads * p.D + sg.h * G * p.D;
            auto store = [&](int e, const float4& v) {
                const int d = 4 * (e & (kD / 4 - 1));
                if (d >= p.D) return;  // head_dim 64: the partial's upper columns are padding
                const int64_t at = out0 + roff_s[e / (kD / 4)] + d;
                if (p.a.out_bf16)
                    *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.a.out) + at) =
                        make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
                else
                    *reinterpret_cast<float4*>(p.a.out + at) = v;
            };
            if (sg.n <= 4) {  // few partials, many elements: three elements of every partial in flight
#pragma unroll 1
                for (int e0 = lo + tid; e0 < hi; e0 += 96) {
                    float4 acc[3];
#pragma unroll
                    for (int u = 0; u < 3; ++u) acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    float4 x[4][3];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
#pragma unroll
                        for (int u = 0; u < 3; ++u) {
                            x[k][u] = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (k < sg.n && e0 + 32 * u < hi) x[k][u] = __ldcg(src + k * E4 + e0 + 32 * u);
                        }
#pragma unroll
                    for (int k = 0; k < 4; ++k)
#pragma unroll
                        for (int u = 0; u < 3; ++u) {
                            acc[u].x += x[k][u].x;
                            acc[u].y += x[k][u].y;
                            acc[u].z += x[k][u].z;
                            acc[u].w += x[k][u].w;
                        }
#pragma unroll
                    for (int u = 0; u < 3; ++u)
                        if (e0 + 32 * u < hi) store(e0 + 32 * u, acc[u]);
                }
            } else {
                for (int e = lo + tid; e < hi; e += 32) {
                    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
                    for (int k0 = 0; k0 < sg.n; k0 += 16) {  // batches of 16 independent loads
                        float4 x[16];
                        const float4* q = src + (int64_t)k0 * E4 + e;
                        const int n_ld = sg.n - k0;
#pragma unroll
                        for (int u = 0; u < 16; ++u) {
                            x[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                            if (u < n_ld) x[u] = __ldcg(q + u * E4);
                        }
#pragma unroll
                        for (int u = 0; u < 16; ++u) {
                            acc.x += x[u].x;
                            acc.y += x[u].y;
                            acc.z += x[u].z;
                            acc.w += x[u].w;
                        }
                    }
                    store(e, acc);
                }
            }
            __syncwarp();
            if (lane == 0 && unit + kRing - 1 < U) {  // the partials have been read: their places may be used again
                __threadfence();
                atomicAdd(c_p1, 1);  // (every CTA of the problem has added its one before: c_o was complete)
            }
        }
    } else {
        // =========================== softmax warpgroups ===========================
        const int sw = warp - 4;                 // 0..kSW-1
        const int wg = sw >> 2;                  // column group
        const int quarter = warp & 3;            // TMEM lane quarter this warp may touch
        const int key_l = quarter * 32 + lane;   // key within the tile (P1/P2) or d (epilogue)
        const int tid_s = threadIdx.x - 128;     // 0..128*CG-1
        const int c0 = wg * NH;                  // first column of this warpgroup
        const uint32_t t_lane = tmem_base + ((uint32_t)(quarter * 32) << 16);
        const int stat_r0 = p.a.first_stat_row * G;
        const bool ph_fast = (8 % G) == 0;  // per-head statistic: column i of a 16-column chunk is head i mod 8 mod G
        const float cs0 = p.scale_log2;
        float vsc = 1.f;  // SC: scale of this unit's V
        // F8: powers of two that travel with the operands (see the kernel's header)
        constexpr float kPExp = 16384.f;         // P~ is held times 2^14
        constexpr float kLoExp = 2048.f;         // the remainder of its fp16 rounding times 2^11
        uint32_t g_conv = 0, g_total = 0;        // F8: tiles expanded so far / of the units up to three ahead (K and V)
        const uint32_t f8_ahead = F8 ? (uint32_t)min(p.n_slots - 2, 2) : 0u;  // tiles expanded ahead of the one in use
        int q_next = 0;                          // F8: first unit whose Q is not converted yet
        uint32_t qn_s = 0;                       // F8: Q buffers seen (phase of q_full / q_ready)
        int g_unit = 0;                          // F8: first unit whose tiles are not in g_total yet
        // F8: expands the next raw tile (in the order the producer loads them) into the next operand slot.
        // A thread of the softmax warps takes 16-byte pieces of the tile's 1024: piece q of row r holds
        // d = 16 q .. 16 q + 15, i.e. the 16-byte chunks 2 (q % 4) and 2 (q % 4) + 1 of row r in the 64-wide
        // half q / 4 (rows of 128 B, chunks swizzled with the row's low three bits).
        uint32_t cv_r = 0, cv_rph = 0, cv_s = 0, cv_sph = 0;  // ring positions of the next tile to expand (no division per tile)
        // The thread's pieces, the same for every tile: source offset in the raw stage (low half) and offset of
        // the first of the two 16-byte chunks in the slot (high half; the second is its neighbour, offset ^ 16).
        // Eight consecutive threads take eight consecutive rows and eight different pieces: their loads and
        // both of their stores then fall on eight different 16-byte bank groups.
        constexpr int kIter = (1024 + 128 * CG - 1) / (128 * CG);
        uint32_t cv_off[kIter];
#pragma unroll
        for (int k = 0; k < kIter; ++k) {
            const int i = tid_s + k * 128 * CG;
            const int l = i & 7, blk = i >> 3, row = 8 * (blk >> 3) + l, q = (l + blk) & 7;
            const int c0 = (q & 3) * 2, sw = row & 7;
            cv_off[k] = (uint32_t)(row * 128 + q * 16) | ((uint32_t)((q >> 2) * 16384 + row * 128 + ((c0 ^ sw) << 4)) << 16);
        }
        auto convert_tile = [&]() -> bool {
            const uint32_t r = cv_r, rph = cv_rph, s = cv_s, sph = cv_sph;
            if (++cv_r == (uint32_t)p.n_raw) {
                cv_r = 0;
                cv_rph ^= 1;
            }
            if (++cv_s == (uint32_t)p.n_slots) {
                cv_s = 0;
                cv_sph ^= 1;
            }
            if (!bar_wait(B.raw_full + 8 * r, rph, ctl)) return false;
            if (!bar_wait(B.slot_empty + 8 * s, sph ^ 1, ctl)) return false;
            const uint8_t* raw = sgen + (s_raw - sbase) + r * 16384;
            uint8_t* slot = sgen + (s_slots - sbase) + s * kSlotBytes;
            uint4 in[kIter];
#pragma unroll
            for (int k = 0; k < kIter; ++k)  // every load of the thread is in flight before the first is used
                if (tid_s + k * 128 * CG < 1024) in[k] = *reinterpret_cast<const uint4*>(raw + (cv_off[k] & 0xffffu));
#pragma unroll
            for (int k = 0; k < kIter; ++k) {
                if (tid_s + k * 128 * CG < 1024) {
                    uint32_t o[8];
                    e4m3x4_to_f16x4(in[k].x, o[0], o[1]);
                    e4m3x4_to_f16x4(in[k].y, o[2], o[3]);
                    e4m3x4_to_f16x4(in[k].z, o[4], o[5]);
                    e4m3x4_to_f16x4(in[k].w, o[6], o[7]);
                    uint8_t* dst = slot + (cv_off[k] >> 16);
                    *reinterpret_cast<uint4*>(dst) = make_uint4(o[0], o[1], o[2], o[3]);
                    *reinterpret_cast<uint4*>(reinterpret_cast<uintptr_t>(dst) ^ 16) = make_uint4(o[4], o[5], o[6], o[7]);
                }
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(B.slot_full + 8 * s);
                mbar_arrive(B.raw_empty + 8 * r);
            }
            return true;
        };
        auto ensure_converted = [&](uint32_t g_need) -> bool {
            while (g_conv <= g_need && g_conv < g_total) {
                if (!convert_tile()) return false;
                ++g_conv;
            }
            return true;
        };
        // F8: Q of every unit up to `unit` as fp16, in place (a 16-bit element stays where it is, so the
        // swizzle does not matter); exact for magnitudes in [6.1e-5, 65504]
        auto ensure_q = [&](int unit) -> bool {
            for (; q_next <= unit && q_next < U; ++q_next) {
                const Work s2 = get_work(sc, q_next);
                if (!s2.valid()) continue;
                if (!bar_wait(B.q_full, qn_s & 1, ctl)) return false;
                ++qn_s;
                uint32_t* qw = reinterpret_cast<uint32_t*>(sgen + (s_q - sbase));
                for (int i = tid_s; i < q_bytes / 4; i += 128 * CG) {
                    const uint32_t w = qw[i];
                    const __half2 h = __floats2half2_rn(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
                    qw[i] = *reinterpret_cast<const uint32_t*>(&h);
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(B.q_ready);
            }
            return true;
        };
        constexpr float kNegBig = -1.0e30f;      // finite stand-in for -inf: keeps ex2 arguments NaN-free
        uint32_t pv_idx = 0, slot_base = 0, o_phase = 0, sync_n = 0, sfull_par = 0;
        uint32_t rbase = 0;                      // region of the unit's first tile (see the MMA warp)
        auto region_of = [&](int c) -> uint32_t {  // of tile c of the unit (c <= n_cache)
            const uint32_t r = rbase + c;
            return r >= (uint32_t)p.n_cache ? r - p.n_cache : r;
        };
        uint32_t pb = 0;                         // P buffer of the next tile
        bool ok = true;

        // O^T (d on lanes, rows on columns, hi and lo parts), rescaled from the CTA-local to the
        // global normaliser -> this CTA's partial [r][d]
        auto epilogue = [&](int unit, const Work& sg) -> bool {
            const int64_t obase = ((int64_t)(unit % kRing) * gridDim.x + blockIdx.x) * R * kD;
            if (!bar_wait(B.o_full, o_phase, ctl)) return false;
            o_phase ^= 1;
            tc_fence_after();
            uint32_t v[NH], w[NH];
            load_cols<NH>(t_lane + col_o + c0, v);
            load_cols<NH>(t_lane + col_o + N + c0, w);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(B.o_empty);
            auto value = [&](int i) -> float {
                const float fac = SC ? fac_s[c0 + i] * vsc : fac_s[c0 + i];
                return (F8 ? fmaf(__uint_as_float(w[i]), 1.f / kLoExp, __uint_as_float(v[i]))
                           : __uint_as_float(v[i]) + __uint_as_float(w[i])) * fac;
            };
            if (sg.n > 1) {
                float* dst = p.o_part + obase + c0 * kD + key_l;
#pragma unroll
                for (int i = 0; i < NH; ++i)
                    if (c0 + i < R) dst[i * kD] = value(i);
            } else if (key_l < p.D) {  // no other CTA has a part of the problem: this is the output
                const int64_t out0 =
                    ((int64_t)sg.layer * p.a.kv.batch + sg.b) * p.a.n_q * p.a.kv.n_q_heads * p.D + sg.h * G * p.D + key_l;
                const bool half = p.a.out_bf16 != 0;
                char* dst = reinterpret_cast<char*>(p.a.out) + out0 * (half ? 2 : 4);
#pragma unroll
                for (int i = 0; i < NH; ++i) {
                    if (c0 + i < R) {
                        const int off = roff_s[c0 + i];
                        if (half) *reinterpret_cast<__nv_bfloat16*>(dst + 2 * off) = __float2bfloat16_rn(value(i));
                        else *reinterpret_cast<float*>(dst + 4 * off) = value(i);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(B.pub_o);  // the publisher warp fences and bumps the counter
            return true;
        };

        for (int unit = 0; unit < U && ok; ++unit) {
            const Work sg = get_work(sc, unit);
            if (!sg.valid()) {  // keeps step with the publisher warp
                if (sw == kSW - 1 && lane == 0) mbar_arrive(B.pub_p1);
                ok = bar_wait(B.lse_ready, unit & 1, ctl);
                if (lane == 0) mbar_arrive(B.pub_o);
                continue;
            }
            const int n_t = sg.t1 - sg.t0;
            if (F8) {
                for (; g_unit <= unit + 3 && g_unit < U; ++g_unit) {
                    const Work s2 = get_work(sc, g_unit);
                    g_total += 2u * (uint32_t)(s2.t1 - s2.t0);
                }
            }
            // SC (an 8-bit cache expanded to bf16 without its scales): K's per-(layer, KV head) scale joins
            // the softmax scale, V's the output
            float cs = cs0;
            if (SC) {
                const int64_t sh = (int64_t)sg.layer * p.a.kv.n_kv_heads + sg.h;
                if (p.a.kv.k_scale) cs *= __ldg(p.a.kv.k_scale + sh);
                vsc = p.a.kv.v_scale ? __ldg(p.a.kv.v_scale + sh) : 1.f;
            }
            if (F8) {
                vsc *= 1.f / kPExp;
                ok = ensure_q(unit);
                if (!ok) break;
            }
            // ------------------------------ P1 ------------------------------
            float m[NH], l[NH];
#pragma unroll
            for (int i = 0; i < NH; ++i) {
                m[i] = kNegBig;
                l[i] = 0.f;
            }
            for (int c = 0; c < n_t && ok; ++c) {
                const int t = sg.t0 + c;
                if (F8) {
                    ok = ensure_converted(slot_base + c + f8_ahead);
                    if (!ok) break;
                }
                const uint32_t rg = region_of(c);
                ok = bar_wait(B.s_full + 8 * rg, (sfull_par >> rg) & 1, ctl);
                if (!ok) break;
                sfull_par ^= 1u << rg;
                tc_fence_after();
                uint32_t v[NH];
                load_cols<NH>(t_lane + col_s + rg * N + c0, v);
                float sc[NH];
#pragma unroll
                for (int i = 0; i < NH; ++i) sc[i] = __uint_as_float(v[i]) * cs;
                if (t * kTile + kTile > sg.T - p.a.n_q + 1) {
                    // tile holds keys some window rows may not see (or keys beyond the context)
                    const int hidden = (t * kTile + key_l - (sg.T - p.a.n_q)) * G - c0;  // columns before it do not see the key
#pragma unroll
                    for (int i = 0; i < NH; ++i)
                        if (i < hidden) sc[i] = kNegBig;
                }
                // The reference of a column is one for the whole warp, so that the sums of its lanes simply add up at the
                // end: lane 0's first score, moved up to the tile's largest when some score is 2^8 above it (one
                // warp-uniform branch per tile).  (A maximum over the lanes at the end of every unit: 267 instead
                // of 257 us at the 32B shape, 64 K, batch 4.)
                if (c == 0) {
#pragma unroll
                    for (int i = 0; i < NH; ++i) m[i] = __shfl_sync(0xffffffffu, sc[i], 0);
                }
                bool need = false;
#pragma unroll
                for (int i = 0; i < NH; ++i) need |= sc[i] > m[i] + 8.f;
                if (__any_sync(0xffffffffu, need)) {
#pragma unroll
                    for (int i = 0; i < NH; ++i) {
                        const float mn = fmaxf(m[i], warp_max_all(sc[i]));
                        l[i] *= ex2(m[i] - mn);
                        m[i] = mn;
                    }
                }
#pragma unroll
                for (int i = 0; i < NH; ++i) l[i] += ex2(sc[i] - m[i]);
            }
            if (!ok) break;
            // reduce (m, l) over the 32 key lanes of this warp, then over the 4 warps via smem
            {
                if (lane == 0) {  // (the references are the same on all lanes)
#pragma unroll
                    for (int i = 0; i < NH; i += 4)
                        *reinterpret_cast<float4*>(red_m + sw * NC + i) = make_float4(m[i], m[i + 1], m[i + 2], m[i + 3]);
                }
                int col = 0;
                sum_step<NH, NH, 16>(l, lane, col);
                constexpr uint32_t kDup = sum_dupmask(NH);
                constexpr int kLeft = sum_final_n(NH);
                if ((lane & kDup) == 0) {
#pragma unroll
                    for (int j = 0; j < kLeft; ++j) red_l[sw * NC + col + j] = l[j];
                }
            }
            ok = warps_sync(B.sm_sync, sync_n, ctl);
            if (!ok) break;
            if (sw == kSW - 1) {
                // the last softmax warp merges the four lane quarters of every column, publishes the
                // CTA's partial and leaves the CTA-local normaliser for the P V pass
                const int64_t base = ((int64_t)(unit % kRing) * gridDim.x + blockIdx.x) * R;
                for (int col = lane; col < R; col += 32) {
                    const int wgi = col / NC, ci = col - wgi * NC;
                    float M = kNegBig;
#pragma unroll
                    for (int w = 0; w < 4; ++w) M = fmaxf(M, red_m[(wgi * 4 + w) * NC + ci]);
                    float Ls = 0.f;
#pragma unroll
                    for (int w = 0; w < 4; ++w) Ls += red_l[(wgi * 4 + w) * NC + ci] * ex2(red_m[(wgi * 4 + w) * NC + ci] - M);
                    const bool has = M > 0.5f * kNegBig;              // the row saw at least one key here
                    const float loc = has ? M + log2f(Ls) : 1.0e30f;  // no key: P = exp2(s - big) = 0
                    loc_s[col] = loc;
                    if (sg.n > 1) {
                        p.ml_part[base + col] = make_float2(M, has ? Ls : 0.f);
                    } else {  // the only CTA of the problem: its normaliser is the row's
                        fac_s[col] = has ? 1.f : 0.f;
                        if (p.a.lse) {
                            const int j = col / G, g = col - j * G;
                            p.a.lse[(((int64_t)sg.layer * p.a.kv.batch + sg.b) * p.a.n_q + j) * p.a.kv.n_q_heads + sg.h * G + g] =
                                loc * 0.69314718055994530942f;
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(B.pub_p1);  // the publisher warp takes it from here
            }
            ok = warps_sync(B.sm_sync, sync_n, ctl);
            if (!ok) break;
            {
                // ------------------------------ P2a: P V with the CTA-local normaliser ------------------
                // P~ = exp2(S - lse_local) needs nothing from other CTAs, so V streams and the tensor
                // cores run while the partials of the other CTAs are still on their way; the partial
                // O is rescaled by exp2(lse_local - LSE) per row in the epilogue.
                // Column-split like P1: every warpgroup works on the same tile, NC columns each, so
                // a tile's P is ready after one short pass; the score columns of the next tile are
                // fetched from tensor memory while the current ones are being turned into P.
                {
                    const float4* loc4 = reinterpret_cast<const float4*>(loc_s + c0);
                    uint32_t v[NH];
#pragma unroll
                    for (int q = 0; q < NH; q += 8) tmem_ld8(t_lane + col_s + rbase * N + c0 + q, v + q);
                    for (int c = 0; c < n_t && ok; ++c) {
                        const int t = sg.t0 + c;
                        const uint32_t pvi = pv_idx + c;
                        const int key = t * kTile + key_l;
                        if (F8) {  // V tile c + 2 (or the next unit's first K tiles) becomes an operand meanwhile
                            ok = ensure_converted(slot_base + n_t + c + f8_ahead);
                            if (!ok) break;
                        }
                        tc_wait_ld();
                        float pr[NH];
#pragma unroll
                        for (int i = 0; i < NH; i += 4) {
                            const float4 ls = loc4[i >> 2];
                            // F8: 2^14 P~ (the fp16 parts below then stay normal numbers down to 2^-28)
                            pr[i + 0] = ex2(fmaf(__uint_as_float(v[i + 0]), cs, F8 ? 14.f - ls.x : -ls.x));
                            pr[i + 1] = ex2(fmaf(__uint_as_float(v[i + 1]), cs, F8 ? 14.f - ls.y : -ls.y));
                            pr[i + 2] = ex2(fmaf(__uint_as_float(v[i + 2]), cs, F8 ? 14.f - ls.z : -ls.z));
                            pr[i + 3] = ex2(fmaf(__uint_as_float(v[i + 3]), cs, F8 ? 14.f - ls.w : -ls.w));
                        }
                        if (c + 1 < n_t) {  // next tile's columns: in flight during the rest of this tile
#pragma unroll
                            for (int q = 0; q < NH; q += 8) tmem_ld8(t_lane + col_s + region_of(c + 1) * N + c0 + q, v + q);
                        }
                        if (t * kTile + kTile > sg.T - p.a.n_q + 1) {
                            const int hidden = (key - (sg.T - p.a.n_q)) * G - c0;
#pragma unroll
                            for (int i = 0; i < NH; ++i)
                                if (i < hidden) pr[i] = 0.f;  // select, so NaN-safe
                        }
                        // P~ replaces the tile's scores in tensor memory: the statistic pass then only
                        // weights it with exp2(lse_local - LSE) per row, no second exponential
#pragma unroll
                        for (int q = 0; q < NH; q += 8)
                            tmem_st8(t_lane + col_s + region_of(c) * N + c0 + q, reinterpret_cast<const uint32_t*>(pr) + q);
                        // the P buffer is free once the P V product p_bufs tiles back is done ("done"
                        // barriers are indexed by the tile's sequence number mod 4)
                        if (pvi >= (uint32_t)p.p_bufs) {
                            const uint32_t prev = pvi - p.p_bufs;
                            ok = bar_wait(B.p_empty + 8 * (prev & 3), (prev >> 2) & 1, ctl);
                            if (!ok) break;
                        }
                        // [P_hi | P_lo]^T as the B operand, rows contiguous (MN-major, no swizzle): the
                        // 16-byte vector of row block j (rows 8j..8j+7 of the concatenation) and key k
                        // lives at j*2048 + (k/8)*128 + (k%8)*16
                        uint8_t* p_row = sgen + (s_p - sbase) + pb * p_bytes + (key_l >> 3) * 128 + (key_l & 7) * 16;
#pragma unroll
                        for (int nb = 0; nb < NH / 8; ++nb) {
                            uint32_t hi[4], lo[4];
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                // p = hi + lo with both parts cut to bf16 by truncation (plain integer ops, no
                                // conversion instructions): hi keeps the top 16 bits, lo the top 16 bits of the
                                // exact remainder, so p - (hi + lo) < 2^-14 p
                                const uint32_t ua = __float_as_uint(pr[nb * 8 + 2 * q]), ub = __float_as_uint(pr[nb * 8 + 2 * q + 1]);
                                if (F8) {
                                    // fp16 rounding of 2^14 P~ and the fp16 rounding of 2^11 times what it left over
                                    const __half2 h = __floats2half2_rn(__uint_as_float(ua), __uint_as_float(ub));
                                    const float2 hf = __half22float2(h);
                                    const __half2 l = __floats2half2_rn((__uint_as_float(ua) - hf.x) * kLoExp,
                                                                        (__uint_as_float(ub) - hf.y) * kLoExp);
                                    hi[q] = *reinterpret_cast<const uint32_t*>(&h);
                                    lo[q] = *reinterpret_cast<const uint32_t*>(&l);
                                    continue;
                                }
                                hi[q] = __byte_perm(ua, ub, 0x7632);
                                const float ra = __uint_as_float(ua) - __uint_as_float(ua & 0xffff0000u);
                                const float rb = __uint_as_float(ub) - __uint_as_float(ub & 0xffff0000u);
                                lo[q] = __byte_perm(__float_as_uint(ra), __float_as_uint(rb), 0x7632);
                            }
                            const int jh = wg * (NH / 8) + nb, jl = jh + N / 8;
                            *reinterpret_cast<uint4*>(p_row + jh * 2048) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                            *reinterpret_cast<uint4*>(p_row + jl * 2048) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                        }
                        if (t * kTile + kTile > sg.T) {
                            // ragged last tile: V rows at or beyond T may hold anything; zero them in
                            // shared memory so that 0 * garbage never reaches the accumulator
                            const uint32_t vslot = slot_base + n_t + c;
                            const uint32_t vs = vslot % p.n_slots, vsph = (vslot / p.n_slots) & 1;
                            ok = bar_wait(B.slot_full + 8 * vs, vsph, ctl);
                            if (!ok) break;
                            if (key >= sg.T && wg < 2) {  // warpgroups 0 and 1 clear one 64-wide half each
                                uint8_t* vrow = sgen + (s_slots - sbase) + vs * kSlotBytes + wg * kHalf +
                                                (key_l >> 3) * kGroup + (key_l & 7) * 128;
#pragma unroll
                                for (int ch = 0; ch < 8; ++ch) *reinterpret_cast<uint4*>(vrow + 16 * ch) = make_uint4(0, 0, 0, 0);
                            }
                        }
                        fence_proxy_async();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(B.p_full + 8 * pb);
                        if (++pb == (uint32_t)p.p_bufs) pb = 0;
                    }
                }
                if (!ok) break;
                tc_wait_st();
                tc_fence_before();
                pv_idx += n_t;
                slot_base += 2 * n_t;
                // ---- the row LSE and the rescale factors, combined by the publisher warp meanwhile ----
                ok = bar_wait(B.lse_ready, unit & 1, ctl);
                if (!ok) break;
                if (!LP && sg.n > 1) {  // many CTAs per head: too many partials for one warp, all softmax threads fold them
                    if (lane == 0) ok = counter_wait(p.counters + sg.prob, sg.n, ctl, 33);
                    ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;  // lane 0's acquire, then warp-wide
                    if (!ok) break;
                    const float2* src = p.ml_part + ((int64_t)(unit % kRing) * gridDim.x + sg.cta0()) * R;
                    // tpr threads of one warp share a row: each folds every tpr-th partial, then shuffles
                    int tpr = 32;
                    while (tpr * R > 128 * CG) tpr >>= 1;
                    const int r = tid_s / tpr, sub = tid_s - r * tpr;
                    float M = kNegBig, Ls = 0.f;
                    if (r < R) {
                        for (int k0 = sub; k0 < sg.n; k0 += 8 * tpr) {  // batches of 8 independent loads
                            float2 x[8];
#pragma unroll
                            for (int u = 0; u < 8; ++u)
                                x[u] = (k0 + u * tpr < sg.n) ? __ldcg(src + (int64_t)(k0 + u * tpr) * R + r)
                                                              : make_float2(kNegBig, 0.f);
#pragma unroll
                            for (int u = 0; u < 8; ++u) {
                                const float Mn = fmaxf(M, x[u].x);
                                Ls = Ls * ex2(M - Mn) + x[u].y * ex2(x[u].x - Mn);
                                M = Mn;
                            }
                        }
                    }
                    for (int o = tpr >> 1; o > 0; o >>= 1) {
                        const float M2 = __shfl_xor_sync(0xffffffffu, M, o);
                        const float L2 = __shfl_xor_sync(0xffffffffu, Ls, o);
                        const float Mn = fmaxf(M, M2);
                        Ls = Ls * ex2(M - Mn) + L2 * ex2(M2 - Mn);
                        M = Mn;
                    }
                    if (sub == 0 && r < R) {
                        const float lse2 = M + log2f(Ls);
                        const float loc = loc_s[r];
                        fac_s[r] = loc < 1.0e29f ? ex2(loc - lse2) : 0.f;  // local -> global normaliser
                        if (sg.rank == 0 && p.a.lse) {
                            const int j = r / G, g = r - j * G;
                            const int64_t row = (((int64_t)sg.layer * p.a.kv.batch + sg.b) * p.a.n_q + j) * p.a.kv.n_q_heads + sg.h * G + g;
                            p.a.lse[row] = lse2 * 0.69314718055994530942f;
                        }
                    }
                }
                if (F8) {  // the next unit's Q has landed by now: its K Q^T can start as the statistic pass frees regions
                    ok = ensure_q(unit + 1);
                    if (!ok) break;
                }
                ok = warps_sync(B.sm_sync, sync_n, ctl);  // every warp is done with the P V pass
                if (!ok) break;
                tc_fence_after();  // the P~ stores of the other warps, ordered by the barrier
                // ------------------------------ P2b: the Eq. 3 statistic ------------------------------
                // second visit of the cached tiles, which hold P~ = exp2(S - lse_local) by now (masked
                // entries are 0): weighted with exp2(lse_local - LSE) per row they are the exactly
                // normalised probabilities, whose column sums are the statistic.  No exponential, no
                // shared memory, no tensor cores; the tile's TMEM region is released afterwards.
                for (int c = wg; c < n_t; c += CG) {
                    const int t = sg.t0 + c;
                    const int key = t * kTile + key_l;
                    const uint32_t rg = region_of(c);
                    float st = 0.f;
                    float sth[PH ? 8 : 1];  // PH: column i belongs to head i mod G, and G divides 8
#pragma unroll
                    for (int i = 0; i < (PH ? 8 : 1); ++i) sth[i] = 0.f;
#pragma unroll 1
                    for (int cb = 0; cb < N; cb += 16) {
                        if (cb + 16 <= stat_r0) continue;  // rows outside the statistic window
                        uint32_t v[16];
                        tmem_ld8(t_lane + col_s + rg * N + cb, v);
                        tmem_ld8(t_lane + col_s + rg * N + cb + 8, v + 8);
                        tc_wait_ld();
                        const float4* fac4 = reinterpret_cast<const float4*>(fac_s + cb);
                        float pr[16];
#pragma unroll
                        for (int i = 0; i < 16; i += 4) {
                            const float4 f = fac4[i >> 2];
                            pr[i + 0] = __uint_as_float(v[i + 0]) * f.x;
                            pr[i + 1] = __uint_as_float(v[i + 1]) * f.y;
                            pr[i + 2] = __uint_as_float(v[i + 2]) * f.z;
                            pr[i + 3] = __uint_as_float(v[i + 3]) * f.w;
                        }
                        if (PH && ph_fast) {
#pragma unroll
                            for (int i = 0; i < 16; ++i) sth[i & 7] += (cb + i >= stat_r0) ? pr[i] : 0.f;
                        } else if (PH) {
                            // any group size up to 8: accumulator g takes the columns r with r mod G == g
                            int g = cb % G;
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                const float val = (cb + i >= stat_r0) ? pr[i] : 0.f;
#pragma unroll
                                for (int t = 0; t < 8; ++t) sth[t] += (g == t) ? val : 0.f;
                                g = (g + 1 == G) ? 0 : g + 1;
                            }
                        } else if (cb >= stat_r0) {
#pragma unroll
                            for (int i = 0; i < 16; ++i) st += pr[i];
                        } else {
#pragma unroll
                            for (int i = 0; i < 16; ++i) st += (cb + i >= stat_r0) ? pr[i] : 0.f;
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(B.s_free + 8 * rg);
                    if (PH) {
                        // fast path: fold the eight residues mod 8 down to the G residues mod G
                        if (ph_fast && G <= 4) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) sth[i] += sth[i + 4];
                        }
                        if (ph_fast && G <= 2) {
                            sth[0] += sth[2];
                            sth[1] += sth[3];
                        }
                        if (ph_fast && G == 1) sth[0] += sth[1];
                        if (key < sg.T && p.a.stat_group_max) {
                            // one score per KV head: the largest of the group's per-head scores
                            float best = sth[0];
#pragma unroll
                            for (int g = 1; g < 8; ++g)
                                if (g < G) best = fmaxf(best, sth[g]);
                            float* dst = p.a.stats + (int64_t)sg.prob * p.a.stat_stride + key;
                            const float val = p.a.stat_accumulate ? *dst + best : best;
                            *dst = val;
                            if (p.a.hist) atomicAdd(p.a.hist + (int64_t)sg.prob * kScoreBins + (__float_as_uint(val) >> 21), 1u);
                        } else if (key < sg.T) {
#pragma unroll
                            for (int g = 0; g < 8; ++g) {
                                if (g < G) {
                                    float* dst = p.a.stats + ((int64_t)sg.prob * G + g) * p.a.stat_stride + key;
                                    const float val = p.a.stat_accumulate ? *dst + sth[g] : sth[g];
                                    *dst = val;
                                    if (p.a.hist) atomicAdd(p.a.hist + ((int64_t)sg.prob * G + g) * kScoreBins + (__float_as_uint(val) >> 21), 1u);
                                }
                            }
                        }
                    } else if (key < sg.T) {
                        float* dst = p.a.stats + (int64_t)sg.prob * p.a.stat_stride + key;
                        if (F8) st *= 1.f / kPExp;  // the cache holds 2^14 P~
                        const float val = p.a.stat_accumulate ? *dst + st : st;
                        *dst = val;
                        // first radix pass of the selection, fused: count the score's top 11 bits in this
                        // CTA's shared-memory histogram (two 16-bit counters per word: a CTA holds at most
                        // 4096 keys of a head)
                        if (p.a.hist) {
                            const uint32_t bin = __float_as_uint(val) >> 21;
                            atomicAdd(hist_s + (bin >> 1), 1u << ((bin & 1u) * 16));
                        }
                    }
                }
                if (!PH && p.a.hist) {
                    // the CTA's counts of this head join the global ones: one reduction per bin that is not
                    // empty (a few dozen), and the shared-memory copy is clear again for the next unit
                    ok = warps_sync(B.sm_sync, sync_n, ctl);
                    if (!ok) break;
                    uint32_t* hg = p.a.hist + (int64_t)sg.prob * kScoreBins;
                    for (int w = tid_s; w < kScoreBins / 2; w += 128 * CG) {
                        const uint32_t v = hist_s[w];
                        if (v) {
                            hist_s[w] = 0u;
                            if (v & 0xffffu) atomicAdd(hg + 2 * w, v & 0xffffu);
                            if (v >> 16) atomicAdd(hg + 2 * w + 1, v >> 16);
                        }
                    }
                }
            }
            rbase = region_of(n_t);
            // ---- this unit's accumulator: rescale and hand to the reducers ----
            ok = epilogue(unit, sg);
            if (!ok) break;
        }
    }

    // ---- teardown ----
    tc_fence_before();
    __syncthreads();
    if (*abort_flag && threadIdx.x == 0) set_status(p.status, SPEC_ERR_TIMEOUT);  // (unless the cause has been recorded)
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
    if (!*abort_flag) reset_counters_if_last(p, reinterpret_cast<int*>(const_cast<uint32_t*>(tmem_slot)));
}

template <int NC, int CG, bool LP, bool PH, bool SC, bool F8, bool WR>
int launch_cfg(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq, const FastParams& fp,
               int grid, size_t smem_bytes, cudaStream_t stream)
{
    auto kern = verify_cached_kernel<NC, CG, LP, PH, SC, F8, WR>;
    // the largest size any plan of this instance asks for, once per device: the call costs the host as much as a launch
    static std::atomic<bool> opted_in[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SPEC_ERR_CUDA;
    if (!opted_in[dev]) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess)
            return SPEC_ERR_CUDA;
        opted_in[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(128 + 128 * CG);
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = stream;
    // All CTAs must become co-resident (they wait on each other's partials).  The grid never exceeds
    // the SM count at one CTA per SM, so that follows as soon as the previous kernel's CTAs have left:
    // the launch only asks for programmatic stream serialisation, which lets each CTA take an SM the
    // moment the previous layer's CTA on it exits (a cooperative launch would wait for the whole
    // previous grid first: 1.4 us per layer).  A CTA whose peers cannot become resident (SMs held by
    // an unrelated long kernel) ends in SPEC_ERR_TIMEOUT like any other stall.  If the driver refuses
    // the attribute the launch falls back to a cooperative one.
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see griddepcontrol in the kernel
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    static std::atomic<bool> pdl_refused[64] = {};  // per device: a driver that refuses the attribute is asked only once
    const bool pdl_ok = !pdl_refused[dev];
    cudaError_t err = pdl_ok ? cudaLaunchKernelEx(&cfg, kern, tk, tv, tq, fp) : cudaErrorNotSupported;
    if (err != cudaSuccess) {
        if (pdl_ok) cudaGetLastError();
        pdl_refused[dev] = true;
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        err = cudaLaunchKernelEx(&cfg, kern, tk, tv, tq, fp);
    }
    if (err != cudaSuccess) {
        cudaGetLastError();
        return SPEC_ERR_CUDA;
    }
    count_launch(1);
    return SPEC_OK;
}

// One combination of statistic, cache format and tile layout: the instance of a call's row count.
template <bool PH, bool SC, bool F8, bool WR>
int launch_rows(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq, const FastParams& fp, int grid,
                size_t smem_bytes, cudaStream_t stream)
{
    const bool lp = fp.cph <= kLsePubMax;
#define SPEC_CASE(n, nc, cg)                                                                              \
    case n:                                                                                               \
        return lp ? launch_cfg<nc, cg, true, PH, SC, F8, WR>(tk, tv, tq, fp, grid, smem_bytes, stream)    \
                  : launch_cfg<nc, cg, false, PH, SC, F8, WR>(tk, tv, tq, fp, grid, smem_bytes, stream);
    // 17 to 24 rows pad a quarter of the MMA's 32: three warpgroups of eight columns instead of four (16 chats of
    // 0.6-6 K tokens: 57.5 -> 56.1 us per launch, five sequences of 4-30 K: 91.3 -> 88.4.  33 to 36 rows of 48 in
    // three groups of twelve gave nothing: those launches are not bound by the softmax warps.)
    if (fp.N == 32 && fp.R <= 24)
        return lp ? launch_cfg<8, 3, true, PH, SC, F8, WR>(tk, tv, tq, fp, grid, smem_bytes, stream)
                  : launch_cfg<8, 3, false, PH, SC, F8, WR>(tk, tv, tq, fp, grid, smem_bytes, stream);
    switch (fp.N) {  // (columns per warpgroup, warpgroups)
        SPEC_CASE(16, 8, 2)
        SPEC_CASE(32, 8, 4)
        SPEC_CASE(48, 16, 3)
        SPEC_CASE(64, 16, 4)
        SPEC_CASE(80, 40, 2)
        SPEC_CASE(96, 24, 4)
        SPEC_CASE(112, 56, 2)
        SPEC_CASE(128, 32, 4)
        default: return SPEC_ERR_UNSUPPORTED_SHAPE;
    }
#undef SPEC_CASE
}

}  // namespace
}  // namespace sm100
}  // namespace spec
