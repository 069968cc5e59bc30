// Recall selection of Eq. 4: sink + TopK over the middle span + recent, per (layer, sequence,
// KV head).  One CTA per problem.  The scores are sums of probabilities (finite, >= 0), so the
// fp32 bit pattern orders like the value and selection works on bit patterns: integer work only.  (Any other pattern a
// caller leaves there, a sign bit or a NaN, is ordered as the unsigned number it is.)
//
// The scores are read ONCE.  A strided sample of 4096 of them gives a floor that the K_mid-th largest lies
// above with a wide margin (6 sigma); one sweep of 16-byte loads collects what reaches the floor (a few
// percent: score and position) in shared memory; the threshold is found on that list by a histogram of
// (bits - floor) scaled to the list's own range, refined until its bin is small, whose entries are ranked
// pair by pair (larger score, then lower position).  Chosen positions become bits of a position bitmap, which is
// read off in order, window by window where the context exceeds the bitmap's 128 K.  A span that fits the list needs no
// sample (every score is a list entry); hundreds of equal scores at the threshold, or a threshold of zero, are ranked in
// the bitmap.  Where this fails (a sample that misleads, a budget above the list) one sweep per radix digit and an
// ordered compaction do it.
//
// What bounds it: HBM at many long problems, else the chain of memory latencies, block barriers and first
// instruction fetches (about 8 us; code that runs once stays rolled and shared).  256 problems (32 layers x
// 8 heads) of 131 K scores: 105 -> 47 us; of 32 K: 35 -> 20 us.  The two sweeps of
// histogram and collection that this replaced waited for every load and read the scores twice.
//
// Counts of the scores' top 11 bits may arrive from the verification kernel, which counts every score it writes.  They
// are cleared for the next round and not used: as a floor a bin of theirs (an eighth of an octave) is coarser than the
// sample's, and loading it, taking the positions outside the span out again and the longer list cost more than the
// sample saves (us with / without, the clearing included: 8 problems of 6 K 9.6 / 8.5, 256 of 6 K 18.5 / 12.1, 256 of 131 K 45.8 / 43.3).
#include <atomic>

#include "spec_common.cuh"

namespace spec {

namespace {

constexpr int kThreads = 512;      // two CTAs per SM at 64 registers: 256 problems (32 layers x 8 heads) are one wave
constexpr int kWarps = kThreads / 32;
constexpr int kBins = kScoreBins;
constexpr int kBpt = kBins / kThreads;  // bins per thread
constexpr int kItems = 16;         // consecutive candidates per thread in the compaction sweep
constexpr int kListWords = 20480;  // list: 10240 entries (score, position), or 20480 scores in order: 80 KB
constexpr int kDense = 4096;       // spans up to here are list entries as they are (eight per thread)
constexpr int kPair = 512;         // entries ranked pair by pair (they reuse the histogram's storage)
static_assert(3 * kPair <= kBins, "score, position and choice of each");
constexpr int kSample = 4096;      // eight per thread: a relative error of the floor's rank of 8 % at 3 % kept
constexpr int kV = 4;              // vectors per thread and trip of the sweep; the next trip's are in flight meanwhile
constexpr int kTrip = kV * kThreads;           // vectors per trip
constexpr int kMapWords = 4096;                // position bitmap: 128 K keys at a time
constexpr int kWindow = 32 * kMapWords;
// Bins of the sample's histogram: an exponent and five bits, 32 to the octave, for the 64 octaves below 2^16 (a
// score is a sum of at most some hundred probabilities); smaller scores share the last one.
constexpr int kSampleShift = 18;
constexpr uint32_t kSampleBase = 0x47800000u - ((uint32_t)kBins << kSampleShift);

struct Shared {
    int hist[kBins];
    uint32_t bitmap[kMapWords];  // chosen positions
    int warp_tmp[kWarps];
    int bucket, above, count, total, list_n, pair_n;
    uint32_t max;
};

// Exclusive block-wide prefix sum of one int per thread; sh.total gets the block sum (two barriers; every thread
// may read sh.total and call again).
__device__ __noinline__ int block_exclusive_scan(Shared& sh, int x)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    __syncthreads();  // warp_tmp may still be read from a previous scan
    if (lane == 31) sh.warp_tmp[warp] = inc;
    __syncthreads();
    int w = lane < kWarps ? sh.warp_tmp[lane] : 0;  // every warp scans the warps' sums for itself
#pragma unroll
    for (int o = 1; o < kWarps; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += y;
    }
    if (threadIdx.x == kWarps - 1) sh.total = w;
    const int before = __shfl_sync(0xffffffffu, w, warp > 0 ? warp - 1 : 0);
    return (warp > 0 ? before : 0) + inc - x;
}

// Walks the bins of the histogram from the largest digit down (thread t owns reversed bins 4t .. 4t + 3) and
// leaves the one in which the running count reaches `want` (bucket, above, count); false if the counts do
// not reach it.  Called with the counts complete (a barrier behind them); clears them for the next use.
__device__ __noinline__ bool find_bucket(Shared& sh, int want)
{
    static_assert(kBpt == 4, "four bins per thread");
    int4* mine = reinterpret_cast<int4*>(sh.hist + kBins - 4 - 4 * (int)threadIdx.x);
    const int4 c = *mine;
    *mine = make_int4(0, 0, 0, 0);
    int ex = block_exclusive_scan(sh, c.x + c.y + c.z + c.w);
    const int cc[4] = {c.w, c.z, c.y, c.x};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (ex < want && want <= ex + cc[k]) {
            sh.bucket = kBins - 1 - 4 * (int)threadIdx.x - k;
            sh.above = ex;
            sh.count = cc[k];
        }
        ex += cc[k];
    }
    __syncthreads();
    return sh.total >= want;
}

// 16 bytes of scores; volatile, so that a load written ahead of other work is also issued ahead of it, and behind the
// wait for the kernel before.  Not through the read-only path: that kernel may still be writing them when this one starts.
__device__ __forceinline__ uint4 load_vec(const uint4* p)
{
    uint4 v;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
// asks L2 for `bytes` (a multiple of 16) from a 16-byte aligned address; nothing waits for it
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

__device__ __forceinline__ int sample_bin(uint32_t u)
{
    return u <= kSampleBase ? 0 : min((int)((u - kSampleBase) >> kSampleShift), kBins - 1);
}

// Takes one off where u < floor, unsigned as the comparison that stores (two instructions: the borrow of u - floor; adding
// up comparisons made the sweep of 131 K scores 4 % longer).
__device__ __forceinline__ void less_below(int& count, uint32_t u, uint32_t floor)
{
    asm("{\n\t.reg .u32 t;\n\tsub.cc.u32 t, %1, %2;\n\tsubc.u32 %0, %0, 0;\n\t}" : "+r"(count) : "r"(u), "r"(floor));
}

// Where u >= floor: stores u and its position in the list slot at shared address `at` (positions `off` bytes further) and
// moves on by a slot.  Predicated, not branched: a warp has about twenty hits in the 512 scores of a trip, spread over
// most of its lanes, and a branch per score made the sweep bound by instruction issue (380 per warp and trip, 33 us
// instead of 25 at 256 x 131 K scores; with a branch per vector 480 and 49 us).
__device__ __forceinline__ void push_if(uint32_t u, uint32_t floor, uint32_t& at, uint32_t off, int pos)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .u32 q;\n\t"
        "setp.ge.u32 p, %1, %2;\n\t"
        "add.u32 q, %0, %3;\n\t"
        "@p st.shared.u32 [%0], %1;\n\t"
        "@p st.shared.u32 [q], %4;\n\t"
        "@p add.u32 %0, %0, 4;\n\t}"
        : "+r"(at) : "r"(u), "r"(floor), "r"(off), "r"(pos) : "memory");
}

// Calls f(bits, position) for every candidate of [lo, hi), eight loads per thread in flight (slow path).
template <typename F>
__device__ __forceinline__ void sweep(const uint32_t* __restrict__ st, int lo, int hi, F f)
{
    for (int base = lo + threadIdx.x; base < hi; base += 8 * kThreads) {
        uint32_t u[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) u[k] = base + k * kThreads < hi ? __ldcg(st + base + k * kThreads) : 0u;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (base + k * kThreads < hi) f(u[k], base + k * kThreads);
    }
}

// Entries [i0, i1) of the list, for the functions that stand outside the kernel: position(i) of entry i.
struct List {
    const uint32_t* u;
    const int* pos;  // null: a dense list, where entry i is position i + shift
    int i0, i1, shift;
    __device__ int position(int i) const { return pos ? pos[i] : i + shift; }
};

// Floor of a span longer than a window, to 16 bits below the octave, from a sample that grows with it (4096 of every 256 K
// scores), so that the rank wanted lies 4 sigma above the expected one and 5 below the list's end at every length
// (a budget of 4096 over 1 M scores: 1015 us for 8 problems when one in four lists overflowed, 144 so).  0: the list
// cannot hold enough.
__device__ __noinline__ uint32_t floor_of_long_span(Shared& sh, const uint4* vec, int nv, int span, int k_mid, int cap)
{
    const int rounds = (span >> 18) + 1;
    const float expect = (float)k_mid * rounds * kSample / span, room = (float)cap * rounds * kSample / span;
    const int want = (int)min(expect + 6.f * sqrtf(expect) + 8.f, room - 5.f * sqrtf(room));
    if ((float)want < expect + 4.f * sqrtf(expect)) return 0u;
    auto each_sample = [&](auto f) {
#pragma unroll 1
        for (int r = 0; r < 2 * rounds; ++r) {
            const int64_t k = (threadIdx.x >> 2) + r * (kThreads / 4);
            const uint4 v = load_vec(vec + (int)(k * (nv - 4) / (rounds * (kSample / 16) - 1)) + (threadIdx.x & 3));
            f(v.x);
            f(v.y);
            f(v.z);
            f(v.w);
        }
    };
    __syncthreads();
    each_sample([&](uint32_t u) { atomicAdd(&sh.hist[sample_bin(u)], 1); });
    __syncthreads();
    if (!find_bucket(sh, want)) return 0u;
    if (sh.bucket == 0) return 1u;  // every score but the zeros, if the list holds them
    const int bin = sh.bucket, rest = want - sh.above;
    each_sample([&](uint32_t u) {
        if (sample_bin(u) == bin) atomicAdd(&sh.hist[(u >> (kSampleShift - 11)) & 2047u], 1);
    });
    __syncthreads();
    find_bucket(sh, rest);
    return kSampleBase + ((uint32_t)bin << kSampleShift) + ((uint32_t)sh.bucket << (kSampleShift - 11));
}

// The lowest n bits of m.
__device__ __forceinline__ uint32_t lowest(uint32_t m, int n)
{
    for (int drop = n > 0 ? __popc(m) - n : 0; drop > 0; --drop) m &= ~(0x80000000u >> __clz((int)m));
    return n > 0 ? m : 0u;
}

// The index set of a context above one window, with many equal scores at the threshold, or with a threshold of zero:
// entries above [bin_lo, bin_lo + last], and the best `need` inside (last = 0: the first `need`, whose number does not
// matter; bin_lo = 0 as well: the list holds every score but the zeros, and the first `need` positions of [lo, hi) that
// it lacks are added).  The bitmap is clear and the histogram free.
__device__ __noinline__ void write_windows(Shared& sh, const List l, uint32_t bin_lo, uint32_t last, int need, int lo, int hi,
                                           int* out)
{
    const int tid = threadIdx.x;
    const bool zeros = bin_lo == 0u && last == 0u && l.pos, equal = last == 0u && !zeros;
    constexpr int kWpt = kMapWords / kThreads;  // bitmap words per thread, consecutive ones
    uint32_t* bits = sh.bitmap + kWpt * tid;
    auto count = [&]() {
        int cnt = 0;
        for (int k = 0; k < kWpt; ++k) cnt += __popc(bits[k]);
        return cnt;
    };
    uint32_t* pu = reinterpret_cast<uint32_t*>(sh.hist);
    int *pp = sh.hist + kPair, *pc = sh.hist + 2 * kPair;  // inside the bin: score, position; chosen: position, or -1
    for (int i = l.i0 + tid; i < l.i1; i += kThreads) {
        const uint32_t u = l.u[i];
        if (last && u >= bin_lo && u - bin_lo <= last) {
            const int at = atomicAdd(&sh.pair_n, 1);
            pu[at] = u;
            pp[at] = l.position(i);
        }
    }
    __syncthreads();
    const int np = sh.pair_n;
    for (int e = tid; e < np; e += kThreads) {
        int rank = 0;
        for (int j = 0; j < np; ++j) rank += (pu[j] > pu[e]) | ((pu[j] == pu[e]) & (pp[j] < pp[e]));
        pc[e] = rank < need ? pp[e] : -1;
    }
#pragma unroll 1
    for (int w0 = 0; w0 < hi; w0 += kWindow) {
        auto mark = [&](int pos) {
            const uint32_t d = (uint32_t)(pos - w0);
            if (pos >= 0 && d < (uint32_t)kWindow) atomicOr(&sh.bitmap[d >> 5], 1u << (d & 31));
        };
        __syncthreads();
        if (equal) {  // the first `need` of them, in the order of positions
            for (int i = l.i0 + tid; i < l.i1; i += kThreads)
                if (l.u[i] == bin_lo) mark(l.position(i));
            __syncthreads();
            int keep = need - block_exclusive_scan(sh, count());
            for (int k = 0; k < kWpt; ++k) {
                const int n = __popc(bits[k]);
                bits[k] = lowest(bits[k], keep);
                keep -= n;
            }
            __syncthreads();
            need -= min(need, sh.total);
        }
        for (int i = l.i0 + tid; i < l.i1; i += kThreads)
            if (l.u[i] >= bin_lo && l.u[i] - bin_lo > last) mark(l.position(i));
        for (int e = tid; e < np; e += kThreads) mark(pc[e]);
        __syncthreads();
        if (zeros) {
            auto absent = [&](int k) {  // positions of [lo, hi) without a bit in a word
                const int pos0 = w0 + 32 * (kWpt * tid + k);
                uint32_t m = ~bits[k];
                if (pos0 < lo) m &= lo - pos0 < 32 ? 0xffffffffu << (lo - pos0) : 0u;
                if (hi - pos0 < 32) m &= hi > pos0 ? (1u << (hi - pos0)) - 1u : 0u;
                return m;
            };
            int n = 0;
            for (int k = 0; k < kWpt; ++k) n += __popc(absent(k));
            int keep = need - block_exclusive_scan(sh, n);
            for (int k = 0; k < kWpt; ++k) {
                const uint32_t m = absent(k);
                bits[k] |= lowest(m, keep);
                keep -= __popc(m);
            }
            __syncthreads();
            need -= min(need, sh.total);
        }
        int at = block_exclusive_scan(sh, count());
        for (int k = 0; k < kWpt; ++k) {
            const int pos0 = w0 + 32 * (kWpt * tid + k) - 1;
            for (uint32_t m = bits[k]; m; m &= m - 1) out[at++] = pos0 + __ffs((int)m);
            bits[k] = 0u;
        }
        __syncthreads();
        out += sh.total;
        if (hi - w0 <= kWindow) break;  // (w0 + kWindow may pass 2^31)
    }
}

// Slow path: one sweep per radix digit, then an ordered compaction.  The histogram is clear.
__device__ __noinline__ void select_by_sweeps(Shared& sh, const uint32_t* __restrict__ st, int lo, int hi, int k_mid,
                                              int32_t* __restrict__ out)
{
    uint32_t prefix = 0, mask = 0;
    int need = k_mid;  // how many to take among candidates matching the decided prefix
    for (int pass = 0; pass < 3; ++pass) {
        const int shift = pass == 0 ? 21 : (pass == 1 ? 10 : 0);
        const uint32_t digits = pass == 2 ? 1023u : 2047u;
        __syncthreads();
        sweep(st, lo, hi, [&](uint32_t u, int) {
            if ((u & mask) == prefix) atomicAdd(&sh.hist[(u >> shift) & digits], 1);
        });
        __syncthreads();
        find_bucket(sh, need);
        prefix |= (uint32_t)sh.bucket << shift;
        mask |= digits << shift;
        need -= sh.above;
    }
    const uint32_t thr = prefix;  // take every candidate > thr and the first `need` equal to it
    // One block scan per trip: the counts of "above the threshold" (high half) and "equal to it" (low
    // half) travel in one word; a candidate's slot is (candidates above it so far) + (equal ones so far,
    // capped at the number still needed).
    int gt_seen = 0, eq_seen = 0;
    for (int base = lo; base < hi; base += kThreads * kItems) {
        const int i0 = base + (int)threadIdx.x * kItems;
        uint32_t u[kItems];
        int packed = 0;
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            u[k] = (i0 + k < hi) ? __ldcg(st + i0 + k) : 0u;
            if (i0 + k < hi) packed += u[k] > thr ? (1 << 16) : (u[k] == thr ? 1 : 0);
        }
        const int ex = block_exclusive_scan(sh, packed);
        int gt = gt_seen + (ex >> 16), eq = eq_seen + (ex & 0xffff);
#pragma unroll
        for (int k = 0; k < kItems; ++k) {
            if (i0 + k < hi) {
                if (u[k] > thr) {
                    out[gt + min(eq, need)] = i0 + k;
                    ++gt;
                } else if (u[k] == thr) {
                    if (eq < need) out[gt + eq] = i0 + k;
                    ++eq;
                }
            }
        }
        __syncthreads();  // sh.total is written by one thread of the scan
        gt_seen += sh.total >> 16;
        eq_seen += sh.total & 0xffff;
    }
}

__global__ void __launch_bounds__(kThreads, 2)
select_recall_kernel(const float* __restrict__ stats, int64_t stat_stride, int batch, int n_kv_heads,
                     const int32_t* __restrict__ sel_len, int k_sink, int k_recent, int k_total, int list_words,
                     int32_t* __restrict__ indices, int32_t* __restrict__ n_indices,
                     uint32_t* __restrict__ hist_g)
{
    __shared__ __align__(16) Shared sh;
    extern __shared__ __align__(16) uint32_t dyn_smem[];
    const int cap = list_words / 2;
    uint32_t* list = dyn_smem;                           // score bit patterns
    int* lpos = reinterpret_cast<int*>(dyn_smem + cap);  // [cap] their positions (a dense list needs none)

    const int64_t prob = blockIdx.x;
    const int b = (int)((prob / n_kv_heads) % batch);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // The launch may begin under the kernel before it (programmatic stream serialisation); everything that kernel
    // leaves is read after this wait, and the next kernel is let go only then.
    for (int i = tid; i < kMapWords / 4; i += kThreads) reinterpret_cast<uint4*>(sh.bitmap)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) {
        sh.list_n = 0;
        sh.pair_n = 0;
        sh.max = 0u;
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int T = __ldcg(sel_len + b);  // (not through the read-only path, which could be moved ahead of the wait)
    int32_t* out = indices + prob * k_total;
    const uint32_t* st = reinterpret_cast<const uint32_t*>(stats + prob * stat_stride);
    const int lo = k_sink, hi = T - k_recent;  // candidate span [lo, hi), holds > k_mid entries where T > k_total
    const int k_mid = k_total - k_sink - k_recent;
    const int span = hi - lo;
    // Short spans, and spans of which a large part is kept, are list entries as they are.
    const bool dense = span + 3 <= list_words && (span <= kDense || k_mid > span / 4);
    bool fast = true;
    for (int i = tid; i < kBins; i += kThreads) {
        sh.hist[i] = 0;
        if (hist_g) hist_g[prob * kBins + i] = 0u;
    }

    if (T <= k_total) {  // everything fits: keep every position
        for (int i = tid; i < k_total; i += kThreads) out[i] = i < T ? i : -1;
        if (tid == 0) n_indices[prob] = T > 0 ? T : 0;
        return;
    }
    for (int i = tid; i < k_sink; i += kThreads) out[i] = i;
    for (int i = tid; i < k_recent; i += kThreads) out[k_sink + k_mid + i] = hi + i;
    if (tid == 0) n_indices[prob] = k_total;
    if (k_mid == 0) return;

    // whole 16-byte vectors of the span start at va; at most three scores at either end are left over
    const int va = lo + (int)((16u - (uint32_t)(reinterpret_cast<uintptr_t>(st + lo) & 15)) >> 2 & 3);
    const int nv = hi > va ? (hi - va) >> 2 : 0;
    const uint4* vec = reinterpret_cast<const uint4*>(st + va);
    const int n_head = min(va, hi) - lo, n_end = max(hi - va - 4 * nv, 0);
    const int pad = (4 - (va - lo)) & 3;  // a dense list keeps position lo + i - pad at index i: va falls on 16 bytes
    const int trips = (nv + kTrip - 1) / kTrip;
    auto prefetch_trip = [&](int t) {
        const int v0 = t * kTrip;
        if (v0 < nv) prefetch_l2(vec + v0, (uint32_t)min(kTrip, nv - v0) * 16u);
    };

    // ---- the floor ----
    uint32_t floor_bits = 0;
    if (!dense && hi > kWindow) {
        floor_bits = floor_of_long_span(sh, vec, nv, span, k_mid, cap);
        fast = floor_bits != 0u;
        if (tid < 4) prefetch_trip(tid);
    } else if (!dense) {
        // 256 blocks of four vectors (64 bytes), evenly spread: eight scores per thread
        uint4 s[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int k = (tid >> 2) + r * (kThreads / 4);
            s[r] = load_vec(vec + (int)((int64_t)k * (nv - 4) / (kSample / 16 - 1)) + (tid & 3));
        }
        // rank in the sample: the expected one plus 6 sigma (neighbours may be alike), within what the list holds
        const float r = (float)k_mid * kSample / span;
        const int want = min((int)(r + 6.f * sqrtf(r) + 8.f), (int)(0.9f * cap * kSample / span));
        const uint32_t u[8] = {s[0].x, s[0].y, s[0].z, s[0].w, s[1].x, s[1].y, s[1].z, s[1].w};
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 8; ++k) atomicAdd(&sh.hist[sample_bin(u[k])], 1);
        // The span is asked into L2 four trips (128 KB) ahead of the sweep: a trip waits for L2 and not for HBM.
        if (tid < 4) prefetch_trip(tid);
        __syncthreads();
        fast = find_bucket(sh, want);
        const uint32_t bin = (uint32_t)sh.bucket;
        floor_bits = bin ? kSampleBase + (bin << kSampleShift) : 0u;
        if (bin && fast && sh.count * 4 > want) {  // flat scores, for which 2 % is a coarse step: eleven more bits
            const int rest = want - sh.above;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (sample_bin(u[k]) == (int)bin) atomicAdd(&sh.hist[(u[k] >> (kSampleShift - 11)) & 2047u], 1);
            __syncthreads();
            find_bucket(sh, rest);
            floor_bits |= (uint32_t)sh.bucket << (kSampleShift - 11);
        }
        floor_bits = max(floor_bits, 1u);  // (zero scores stay out: if they are needed the list is too short)
    }

    // ---- one sweep: the candidates at or above the floor ----
    int n_list = 0;
    if (fast) {
        __syncthreads();
        uint32_t mx = 0u;
        const bool edge = tid < n_head + n_end;  // this thread takes one of the scores outside the vectors
        const int edge_pos = tid < n_head ? lo + tid : hi - n_end + (tid - n_head);
        if (dense) {
#pragma unroll 1
            for (int i = tid; i < nv; i += kThreads) {
                const uint4 w = load_vec(vec + i);
                *reinterpret_cast<uint4*>(list + pad + (va - lo) + 4 * i) = w;
                mx = max(mx, max(max(w.x, w.y), max(w.z, w.w)));
            }
            if (edge) {
                const uint32_t u = __ldcg(st + edge_pos);
                list[pad + edge_pos - lo] = u;
                mx = max(mx, u);
            }
        } else {
            if (edge) {
                const uint32_t u = __ldcg(st + edge_pos);
                const int at = u >= floor_bits ? atomicAdd(&sh.list_n, 1) : cap;
                if (at < cap) {
                    list[at] = u;
                    lpos[at] = edge_pos;
                }
            }
            const uint32_t list_s = (uint32_t)__cvta_generic_to_shared(list);
            uint4 w[kV], x[kV];
            auto load = [&](uint4 (&d)[kV], int base) {
#pragma unroll
                for (int k = 0; k < kV; ++k)
                    d[k] = base + k * kThreads < nv ? load_vec(vec + base + k * kThreads) : make_uint4(0u, 0u, 0u, 0u);
            };
            load(w, tid);
#pragma unroll 1
            for (int t = 0; t < trips; ++t) {
                const int base = t * kTrip + tid;
                load(x, base + kTrip);
                if (tid == 0) prefetch_trip(t + 4);
                int mine = 4 * kV;  // hits
#pragma unroll
                for (int k = 0; k < kV; ++k) {  // (scores past the end read as 0 and the floor is above 0)
                    less_below(mine, w[k].x, floor_bits);
                    less_below(mine, w[k].y, floor_bits);
                    less_below(mine, w[k].z, floor_bits);
                    less_below(mine, w[k].w, floor_bits);
                }
                int inc = mine;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += y;
                }
                int at = 0;  // one shared counter update per warp
                if (lane == 31 && inc) at = atomicAdd(&sh.list_n, inc);
                at = __shfl_sync(0xffffffffu, at, 31) + inc - mine;
                if (at + mine <= cap) {  // (a list that overflows is not used)
                    uint32_t la = list_s + 4 * at;
#pragma unroll
                    for (int k = 0; k < kV; ++k) {
                        const int pos = va + 4 * (base + k * kThreads);
                        push_if(w[k].x, floor_bits, la, 4 * cap, pos);
                        push_if(w[k].y, floor_bits, la, 4 * cap, pos + 1);
                        push_if(w[k].z, floor_bits, la, 4 * cap, pos + 2);
                        push_if(w[k].w, floor_bits, la, 4 * cap, pos + 3);
                    }
                }
#pragma unroll
                for (int k = 0; k < kV; ++k) w[k] = x[k];
            }
            __syncthreads();
            const int n = min(sh.list_n, cap);
#pragma unroll 1
            for (int i = 4 * tid; i < n; i += 4 * kThreads) {
                const uint4 q = *reinterpret_cast<const uint4*>(list + i);
                mx = max(mx, max(max(q.x, i + 1 < n ? q.y : 0u), max(i + 2 < n ? q.z : 0u, i + 3 < n ? q.w : 0u)));
            }
        }
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) atomicMax(&sh.max, mx);
        __syncthreads();
        n_list = dense ? span : sh.list_n;
        if (floor_bits == 1u && n_list < k_mid && n_list <= cap && !dense) {  // everything but the zeros is in the list: the rest are zeros
            write_windows(sh, List{list, lpos, 0, n_list, 0}, 0u, 0u, k_mid - n_list, lo, hi, out + k_sink);
            return;
        }
        fast = n_list >= k_mid && (dense || n_list <= cap);
    }

    // ---- the threshold on the list: bins over its own range, refined until the threshold's bin is small ----
    const int i0 = dense ? pad : 0, i1 = i0 + n_list;  // list entries
    uint32_t bin_lo = floor_bits, last = 0xffffffffu;  // the threshold lies in [bin_lo, bin_lo + last]
    int need = k_mid;                                  // entries to take from there
    auto each_entry = [&](auto f) {  // f(bits, list index), four neighbouring entries per thread and trip
#pragma unroll 1
        for (int i = 4 * tid; i < i1; i += 4 * kThreads) {
            const uint4 q = *reinterpret_cast<const uint4*>(list + i);
            if (i >= i0) f(q.x, i);
            if (i + 1 >= i0 && i + 1 < i1) f(q.y, i + 1);
            if (i + 2 >= i0 && i + 2 < i1) f(q.z, i + 2);
            if (i + 3 >= i0 && i + 3 < i1) f(q.w, i + 3);
        }
    };
    if (fast) {
        int shift = max(0, 21 - __clz((int)(sh.max - floor_bits)));
#pragma unroll 1
        for (;;) {
            each_entry([&](uint32_t u, int) {
                const uint32_t d = u - bin_lo;
                if (d <= last) atomicAdd(&sh.hist[d >> shift], 1);
            });
            __syncthreads();
            find_bucket(sh, need);
            need -= sh.above;
            bin_lo += (uint32_t)sh.bucket << shift;
            last = (1u << shift) - 1u;
            if (sh.count <= kPair) break;
            if (shift == 0) break;  // more than kPair equal scores at the threshold
            shift = max(0, shift - 11);
            __syncthreads();  // (sh.bucket and its fellows are read before the next search writes them)
        }
        __syncthreads();
    }
    if (!fast) {
        select_by_sweeps(sh, st, lo, hi, k_mid, out + k_sink);
        return;
    }
    if (hi > kWindow || sh.count > kPair) {
        write_windows(sh, List{list, dense ? nullptr : lpos, i0, i1, lo - pad}, bin_lo, last, need, lo, hi, out + k_sink);
        return;
    }
    // above the bin: chosen; inside: set aside and ranked pair by pair
    uint32_t* pu = reinterpret_cast<uint32_t*>(sh.hist);
    int* pp = sh.hist + kPair;
    each_entry([&](uint32_t u, int i) {
        if (u < bin_lo) return;
        const int pos = dense ? lo + i - pad : lpos[i];
        if (u - bin_lo > last) {
            atomicOr(&sh.bitmap[pos >> 5], 1u << (pos & 31));
        } else {
            const int at = atomicAdd(&sh.pair_n, 1);
            pu[at] = u;
            pp[at] = pos;
        }
    });
    __syncthreads();
    const int np = sh.pair_n;
#pragma unroll 1
    for (int e = tid >> 3; e < np; e += kThreads / 8) {  // eight lanes per entry
        const uint32_t u = pu[e];
        const int pos = pp[e];
        int rank = 0;
#pragma unroll 2
        for (int j = tid & 7; j < np; j += 8) {
            const uint32_t v = pu[j];
            rank += (v > u) | ((v == u) & (pp[j] < pos));
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffu << (lane & 24), rank, o);
        if ((tid & 7) == 0 && rank < need) atomicOr(&sh.bitmap[pos >> 5], 1u << (pos & 31));
    }
    __syncthreads();
    // ---- the index set off the bitmap: consecutive words per thread, gathered in the list's storage (read for the
    // last time above) so that the store is coalesced ----
    const int wpt = (hi + 32 * kThreads - 1) / (32 * kThreads);  // at most eight
    const uint32_t* bits = sh.bitmap + wpt * tid;
    int cnt = 0;
#pragma unroll 1
    for (int k = 0; k < wpt; ++k) cnt += __popc(bits[k]);
    int at = block_exclusive_scan(sh, cnt);
#pragma unroll 1
    for (int k = 0; k < wpt; ++k) {
        const int pos0 = 32 * (wpt * tid + k) - 1;
#pragma unroll 1
        for (uint32_t m = bits[k]; m; m &= m - 1) list[at++] = (uint32_t)(pos0 + __ffs((int)m));
    }
    __syncthreads();
#pragma unroll 1
    for (int i = tid; i < k_mid; i += kThreads) out[k_sink + i] = (int)list[i];
}

// Top-11-bit counts of stats[prob][0 : len[b]) for the verification kernels that do not count while
// they write the statistic.
__global__ void __launch_bounds__(256)
score_hist_kernel(const float* __restrict__ stats, int64_t stat_stride, int batch, int heads,
                  const int32_t* __restrict__ len, int max_len, uint32_t* __restrict__ hist)
{
    const int64_t prob = blockIdx.y;
    const int b = (int)((prob / heads) % batch);
    const int T = min(max(len[b], 0), max_len);
    const uint32_t* st = reinterpret_cast<const uint32_t*>(stats + prob * stat_stride);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < T; i += gridDim.x * blockDim.x)
        atomicAdd(hist + prob * kBins + (__ldcg(st + i) >> 21), 1u);
}

}  // namespace

int select_launch(const float* stats, int64_t stat_stride, int n_layers, int batch, int n_kv_heads,
                  const int32_t* sel_len, int k_sink, int k_recent, int k_total, int32_t* indices,
                  int32_t* n_indices, uint32_t* hist, cudaStream_t stream)
{
    const long probs = (long)n_layers * batch * n_kv_heads;
    static std::atomic<bool> opted_in[64] = {};  // per device: the kernel's dynamic shared memory exceeds the default limit
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SPEC_ERR_CUDA;
    if (!opted_in[dev]) {
        if (cudaFuncSetAttribute(select_recall_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kListWords * 4) != cudaSuccess)
            return SPEC_ERR_CUDA;
        opted_in[dev] = true;
    }
    // no context is longer than a row of scores: short rows take less shared memory, and more CTAs share an SM
    const int64_t row = (stat_stride + 7) / 4 * 4;
    const int list_words = (int)(row < kListWords ? row : kListWords);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)probs);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = (size_t)list_words * 4;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, select_recall_kernel, stats, stat_stride, batch, n_kv_heads, sel_len, k_sink, k_recent, k_total,
                           list_words, indices, n_indices, hist) != cudaSuccess) {
        cudaGetLastError();
        return SPEC_ERR_CUDA;
    }
    count_launch(1);
    return SPEC_OK;
}

int score_hist_launch(const float* stats, int64_t stat_stride, long probs, int batch, int heads, const int32_t* len,
                      int max_len, uint32_t* hist, cudaStream_t stream)
{
    if (probs > 65535) return SPEC_ERR_UNSUPPORTED_SHAPE;
    const int bx = max_len > 256 * 16 ? 16 : (max_len + 255) / 256;
    score_hist_kernel<<<dim3(bx > 0 ? bx : 1, (unsigned)probs), 256, 0, stream>>>(stats, stat_stride, batch, heads, len,
                                                                                 max_len, hist);
    count_launch(1);
    return cudaGetLastError() == cudaSuccess ? SPEC_OK : SPEC_ERR_CUDA;
}

}  // namespace spec
