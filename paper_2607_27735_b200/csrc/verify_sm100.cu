// Host side of the sm_100a verification path: shape checks, the work plan (how KV heads are
// grouped into units and split over the CTAs), TMA tensor maps, and the choice between the
// score-cache kernel (K and V read once) and the two-sweep kernel (any context length).
#include <climits>
#include <cstdlib>
#include <numeric>

#include "sm100_common.cuh"
#include "verify_sm100.cuh"

namespace spec {

using namespace sm100;

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

struct Plan {
    bool cached;
    int HG, cph, n_units, N, n_slots, p_bufs, box_rows, boxes, n_cache, n_raw;
    int n_cls, cls_size[kMaxClass], cls_subs[kMaxClass], n_counters;
    size_t smem_bytes;
    size_t ctr_off, ml_off, o_off, total;
};

int box_rows_for(int page_size)
{
    if (page_size >= kTile) return (page_size % kTile == 0) ? kTile : 0;
    if (page_size >= 8 && kTile % page_size == 0) return page_size;
    return 0;
}

// Score tiles the tensor-memory cache holds next to the output accumulator.
int cache_tiles(int N)
{
    const int n = (kTmemCols - 2 * N) / N;
    return n > 32 ? 32 : n;
}

// Heads of a sequence that are worked on at once when every one gets the same share of the SMs (a divisor of the KV heads;
// 0: a head's share exceeds `tiles` key tiles however it is cut).  from_l2: K is swept a second time.
int best_head_group(const KvView& kv, int max_ctx_len, int nsm, int tiles, bool from_l2)
{
    const int nb = (max_ctx_len + kTile - 1) / kTile;
    int best_hg = 0;
    double best = -1.0;
    for (int hg = 1; hg <= kv.n_kv_heads; ++hg) {
        if (kv.n_kv_heads % hg) continue;
        const int cph = nsm / hg;
        if (cph < 1) continue;
        const int tpc = (nb + cph - 1) / cph;
        if (tpc > tiles) continue;
        double score = (double)nb * hg / ((double)nsm * tpc);  // fraction of CTA-tile slots doing work
        if (from_l2) {
            const double k_mib = (double)hg * max_ctx_len * 256.0 / (1 << 20);
            if (k_mib > 40.0) score -= 0.3;  // the unit's K must stay L2-resident
            if ((long)kv.n_layers * kv.batch * (kv.n_kv_heads / hg) < 2) score -= 0.1;  // a single unit cannot be pipelined
        }
        score += 0.001 * hg;  // ties: fewer partials per head
        if (score > best) {
            best = score;
            best_hg = hg;
        }
    }
    return best_hg;
}

// Workspace of a call whose partials come from `ctas` CTAs with R rows each.
size_t workspace_layout(const KvView& kv, int R, int ctas, size_t* ctr_off, size_t* ml_off, size_t* o_off)
{
    size_t off = kStatusBytes;
    *ctr_off = off;
    off += verify_counter_bytes(kv);
    off = (off + 255) & ~(size_t)255;
    *ml_off = off;
    off += (size_t)kRing * ctas * R * sizeof(float2);
    off = (off + 255) & ~(size_t)255;
    *o_off = off;
    off += (size_t)kRing * ctas * R * kD * sizeof(float);
    return (off + 255) & ~(size_t)255;
}

// variant: 0 = prefer the score-cache kernel, 1 = two-sweep only, 2 = score-cache only.  max_ctas > 0: on at most that
// many CTAs (a caller whose workspace holds no more partials).
bool make_plan(const KvView& kv, int n_q, int max_ctx_len, int variant, Plan* pl, int max_ctas = 0)
{
    const int G = kv.n_q_heads / kv.n_kv_heads, R = n_q * G;
    pl->n_raw = 0;
    // an 8-bit cache is read by the score-cache kernel only (its F8 instances), at head_dim 128
    if (kv.fp8 && (variant == 1 || kv.head_dim != kD)) return false;
    // head_dim 64 runs on the score-cache kernel only (one 64-wide half per tile, V padded with zero rows)
    if (!(kv.head_dim == kD || (kv.head_dim == 64 && variant != 1)) || R > 128 || G > 256 || n_q > 256) return false;
    const int box_rows = box_rows_for(kv.page_size);
    if (box_rows == 0) return false;
    const int nsm = max_ctas > 0 && max_ctas < sm_count() ? max_ctas : sm_count();
    const int N = (R + 15) / 16 * 16;
    const int nb = (max_ctx_len + kTile - 1) / kTile;
    const long lb = (long)kv.n_layers * kv.batch;
    const int n_cache = cache_tiles(N);

    int best_hg = 0;
    bool cached = false;
    int best_cph = 0;
    if (variant != 1) {
        // Score-cache kernel: HG teams of cph CTAs, each team a problem (one KV head of one (layer, sequence)) at a
        // time.  A CTA's share of the longest context must fit the TMEM cache; among the team sizes that do, the
        // one with the least time by a simple model: rounds of problems x (fixed cycles of a round + cycles of a
        // key tile's K and V at the SM's share of HBM x tiles per CTA).  A round of a team of one has no exchange
        // between CTAs.  (Shorter sequences of the batch may run on parts of a team: see Sched in the kernel.)
        const long probs = lb * kv.n_kv_heads;
        double best = 1e300;
        for (int cph = nsm < nb ? nsm : nb; cph >= 1; --cph) {
            const int tpc = (nb + cph - 1) / cph;
            if (tpc > n_cache) break;
            int teams = nsm / cph;
            if (teams > probs) teams = (int)probs;
            const long rounds = (probs + teams - 1) / teams;
            const double t = (double)rounds * ((cph > 1 ? 9000.0 : 6000.0) + 2900.0 * tpc);
            if (t < best) {
                best = t;
                best_hg = teams;
                best_cph = cph;
            }
        }
        cached = best_hg != 0;
        // CTAs that the teams leave over join them
        if (cached && best_cph < nb) best_cph = nsm / best_hg < nb ? nsm / best_hg : nb;
        // A single sequence: no more CTAs than its tiles per CTA need, so that the shares are even and fewer exchange
        // partials (8 heads of 4 K: 18 -> 16 CTAs per head, 18.2 -> 17.1 us per launch; 2 heads of 111 K: 148 -> 128,
        // 49.0 -> 45.0).
        if (cached && kv.batch == 1) {
            const int tpc = (nb + best_cph - 1) / best_cph;
            best_cph = (nb + tpc - 1) / tpc;
        }
        // Short contexts of a batch ask for teams of a few CTAs, whose parts (4, 2, 1) fit the lengths less closely
        // than those of a team of 24 (24, 12, 6, 3): 16 chats of 0.6-6 K tokens 54.0 -> 48.9 us per launch, 16
        // sequences of 3 K 54.5 -> 50.5.  (Over an 8-bit cache, whose rounds cost more, 36.9 -> 40.8: not there.)
        if (cached && best_cph < 8 && kv.batch >= 4 && nb >= 24 && nsm >= 24 && !kv.fp8) {
            best_cph = 24;
            best_hg = nsm / 24 < probs ? nsm / 24 : (int)probs;
        }
    }
    if (!cached) {
        if (variant == 2 || kv.head_dim != kD || kv.fp8) return false;
        best_hg = best_head_group(kv, max_ctx_len, nsm, INT_MAX, true);
        if (best_hg == 0) return false;
    }
    pl->cached = cached;
    pl->n_cache = n_cache;
    pl->HG = best_hg;
    pl->cph = cached ? best_cph : nsm / best_hg;
    pl->n_units = cached ? (int)((lb * kv.n_kv_heads + best_hg - 1) / best_hg) : (int)(lb * (kv.n_kv_heads / best_hg));
    pl->n_cls = 1;
    pl->cls_size[0] = pl->cph;
    pl->cls_subs[0] = 1;
    for (int f = 1; cached && f < kMaxClass && (pl->cph >> f) >= 1; ++f) {
        pl->cls_size[f] = pl->cph >> f;
        pl->cls_subs[f] = pl->cph / pl->cls_size[f];
        pl->n_cls = f + 1;
    }
    pl->n_counters = (int)(2 * lb * kv.n_kv_heads);
    pl->N = N;
    pl->box_rows = box_rows;
    pl->boxes = kTile / box_rows;
    const size_t cap = 227 * 1024;
    size_t fixed = 0;
    int slots = 0;
    if (cached) {
        // one Q buffer, two P buffers ([hi | lo] rows, 8-row blocks: 2N * 256 B each), 12.25 KB of
        // barriers and small arrays; the rest is the K/V tile ring
        pl->p_bufs = 2;
        pl->n_raw = kv.fp8 ? 3 : 0;  // 8-bit cache: three raw stages of 16 KB in front of the slots
        fixed = 1024 /*alignment slack*/ + (size_t)N * 256 + 2 * (size_t)(2 * N * 256) + 12544 + (size_t)pl->n_raw * 16384;
        slots = fixed < cap ? (int)((cap - fixed) / kSlotBytes) : 0;
        if (slots > 8) slots = 8;
        // more P buffers (up to four) where they cost no K/V slot: the P V product of a tile then has two tiles
        // of softmax work to hide behind
        while (slots >= 4 && pl->p_bufs < 4 && fixed + (size_t)(2 * N * 256) + (size_t)slots * kSlotBytes <= cap) {
            ++pl->p_bufs;
            fixed += (size_t)(2 * N * 256);
        }
        if (slots < 4) {
            pl->p_bufs = 1;
            fixed -= (size_t)(2 * N * 256);
            slots = fixed < cap ? (int)((cap - fixed) / kSlotBytes) : 0;
        }
        if (kv.fp8) {
            // 8-bit cache: the raw stages already hold whole tiles in flight, so three operand slots do;
            // P buffers first (the P V product of a tile hides behind the next tiles' softmax work)
            slots = 0;
            for (int pb = 3; pb >= 1 && slots < 3; --pb) {
                for (int nr = 3; nr >= 2 && slots < 3; --nr) {
                    fixed = 1024 + (size_t)N * 256 + (size_t)pb * (2 * N * 256) + 12544 + (size_t)nr * 16384;
                    slots = fixed < cap ? (int)((cap - fixed) / kSlotBytes) : 0;
                    if (slots > 8) slots = 8;
                    pl->p_bufs = pb;
                    pl->n_raw = nr;
                }
            }
        }
    } else {
        const size_t p_bytes = (size_t)((2 * N + 63) / 64) * 16384;
        for (int pb = 2; pb >= 1; --pb) {  // two P buffers if that still leaves a 4-deep K/V ring
            fixed = 1024 /*alignment slack*/ + 2 * (size_t)N * 256 + pb * p_bytes + 12544;
            slots = fixed < cap ? (int)((cap - fixed) / kSlotBytes) : 0;
            pl->p_bufs = pb;
            if (slots >= 4) break;
        }
    }
    if (slots > 8) slots = 8;
    if (slots < 3) return false;
    pl->n_slots = slots;
    pl->smem_bytes = fixed + (size_t)slots * kSlotBytes;
    // room for every CTA, whatever the split: what a split for a long context leaves out one for a shorter may use
    pl->total = workspace_layout(kv, R, nsm, &pl->ctr_off, &pl->ml_off, &pl->o_off);
    return true;
}

// The map's axes behind the head dimension, (slot, head, page, layer), for elements of `es` bytes.  No axis of a map may have
// stride 0: one that has (every head, page or layer the same rows) gets extent 1, and coordinates on it the factor 0.
void map_axes(const KvView& kv, int n_pages, int es, cuuint64_t dims[5], cuuint64_t strides[4], FastParams* fp)
{
    const cuuint64_t n[4] = {(cuuint64_t)kv.page_size, (cuuint64_t)kv.n_kv_heads, (cuuint64_t)n_pages, (cuuint64_t)kv.n_layers};
    const int64_t st[4] = {kv.slot_stride, kv.head_stride, kv.page_stride, kv.layer_stride};
    dims[0] = (cuuint64_t)kv.head_dim;
    for (int i = 0; i < 4; ++i) {
        dims[i + 1] = st[i] ? n[i] : 1;
        strides[i] = st[i] ? (cuuint64_t)st[i] * es : 16;
    }
    fp->row_head = st[1] ? 1 : 0;
    fp->row_page = st[2] ? 1 : 0;
    fp->row_layer = st[3] ? 1 : 0;
}

bool encode_kv_map(CUtensorMap* map, const void* base, const KvView& kv, int n_pages, int box_rows, FastParams* fp)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[5], strides[4];
    map_axes(kv, n_pages, 2, dims, strides, fp);
    const cuuint32_t box[5] = {64, (cuuint32_t)box_rows, 1, 1, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The cache as rows of two 64-wide halves: dimensions (64, 8 rows, half, groups of 8 rows in a page, (layer, page, head)).
// One box, a page, then brings whole rows, the halves of eight of them as two swizzled 1 KB blocks side by side.  The last
// dimension counts in the greatest common divisor of the three strides.
// False where a row cannot be numbered in 31 bits: the caller takes the other map.
bool encode_kv_map_rows(CUtensorMap* map, const void* base, const KvView& kv, int n_pages, FastParams* fp)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const int64_t st[3] = {kv.n_layers > 1 ? kv.layer_stride : 0, n_pages > 1 ? kv.page_stride : 0,
                           kv.n_kv_heads > 1 ? kv.head_stride : 0};
    const int64_t n[3] = {kv.n_layers, n_pages, kv.n_kv_heads};
    int64_t unit = 0, last = 0;
    for (int64_t s : st) unit = std::gcd(unit, s);
    if (unit == 0) unit = 8;
    for (int i = 0; i < 3; ++i) last += st[i] / unit * (n[i] - 1);
    if (last >= INT_MAX || kv.slot_stride >= 1ll << 35 || unit >= 1ll << 38) return false;
    fp->row_layer = (int)(st[0] / unit);
    fp->row_page = (int)(st[1] / unit);
    fp->row_head = (int)(st[2] / unit);
    const cuuint64_t dims[5] = {64, 8, 2, (cuuint64_t)kv.page_size / 8, (cuuint64_t)last + 1};
    const cuuint64_t strides[4] = {(cuuint64_t)kv.slot_stride * 2, 128, (cuuint64_t)kv.slot_stride * 16, (cuuint64_t)unit * 2};
    const cuuint32_t box[5] = {64, 8, 2, (cuuint32_t)kv.page_size / 8, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Whether tiles are copied as whole rows.  The copy unit takes 100-150 cycles over a box however small it is, and with the
// halves in boxes of their own a tile takes twice as many: where that bounds the stream, whole rows; elsewhere the halves,
// which products and softmax take slightly faster.  Time with whole rows against halves in %, 25 shapes, by tokens of a page:
//                             8           16          32          64          128
//   up to 64 score columns  -35..-3    -27..-1    -10..+0.2   -4.3..+0.5  -1.4..+0.5   (short calls gain least)
//   more: longer softmax     -5..-0.4   -2..+0.3  +0.2..+0.8  +0.2..+0.7      0..+0.9
bool copy_whole_rows(const KvView& kv, int N)
{
    return kv.head_dim == kD && !kv.fp8 && !kv.k_scale && !kv.v_scale && kv.page_size <= (N <= 64 ? 64 : 16);
}

// 8-bit cache: a box is box_rows whole rows of 128 bytes, unswizzled (the softmax warps expand it)
bool encode_kv_map_u8(CUtensorMap* map, const void* base, const KvView& kv, int n_pages, int box_rows, FastParams* fp)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[5], strides[4];
    map_axes(kv, n_pages, 1, dims, strides, fp);
    const cuuint32_t box[5] = {128, (cuuint32_t)box_rows, 1, 1, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 5, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_q_map(CUtensorMap* map, const void* q, const KvView& kv, int n_q, int G)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)kv.head_dim, (cuuint64_t)kv.n_q_heads,
                                (cuuint64_t)kv.n_layers * kv.batch * n_q};
    const cuuint64_t strides[2] = {(cuuint64_t)kv.head_dim * 2, (cuuint64_t)kv.n_q_heads * kv.head_dim * 2};
    const cuuint32_t box[3] = {64, (cuuint32_t)G, (cuuint32_t)n_q};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(q), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ---- rows in two passes ----------------------------------------------------------------------
// A single (layer, sequence) whose n_q * G rows do not fit the score cache at its context length
// (many speculated rows at a very long context) is verified as two calls of the score-cache kernel:
// rows [0, nA) against the context shortened by the nB rows that follow them, then rows [nA, n_q)
// against the whole context.  Both are ordinary causal verifications of the same cache; their
// statistics add up (the window rule is applied to each part's own rows).  K and V are read
// twice, which still beats the two-sweep kernel at these shapes.
struct SplitPlan {
    int nA, nB;
    size_t main_bytes, ctx_off, stat_off, total;
    int64_t stat_stride;
};

bool make_split_plan(const KvView& kv, int n_q, int max_ctx_len, SplitPlan* sp, int max_ctas = 0)
{
    if (kv.n_layers * kv.batch != 1 || n_q < 2) return false;
    Plan full;
    if (make_plan(kv, n_q, max_ctx_len, 2, &full, max_ctas)) return false;  // fits in one pass
    sp->nA = (n_q + 1) / 2;
    sp->nB = n_q - sp->nA;
    Plan pa, pb;
    if (!make_plan(kv, sp->nA, max_ctx_len, 2, &pa, max_ctas) || !make_plan(kv, sp->nB, max_ctx_len, 2, &pb, max_ctas))
        return false;
    sp->main_bytes = pa.total > pb.total ? pa.total : pb.total;
    sp->ctx_off = sp->main_bytes;
    sp->stat_off = sp->ctx_off + 256;
    sp->stat_stride = ((int64_t)max_ctx_len + 63) / 64 * 64;
    sp->total = sp->stat_off + (size_t)kv.n_kv_heads * sp->stat_stride * sizeof(float);
    sp->total = (sp->total + 255) & ~(size_t)255;
    return true;
}

__global__ void shorten_ctx_kernel(const int32_t* ctx_len, int by, int32_t* out) { out[0] = ctx_len[0] - by; }

// stats <- (first part's value where it wrote one) + second part's value
__global__ void add_stats_kernel(float* stats, int64_t stat_stride, const float* second, int64_t second_stride,
                                 const int32_t* ctx_len, int max_ctx_len, int nB, int n_kv_heads, int accumulate)
{
    const int T = min(max(ctx_len[0], 0), max_ctx_len);  // the two verification kernels report a length out of range
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (int64_t)n_kv_heads * T;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int h = (int)(i / T), key = (int)(i - (int64_t)h * T);
        const float first = (key < T - nB || accumulate) ? stats[h * stat_stride + key] : 0.f;  // the first part wrote keys < T - nB
        stats[h * stat_stride + key] = first + second[h * second_stride + key];
    }
}

}  // namespace

// Two counters per problem whatever the split, and one for the CTAs that have finished.
size_t verify_counter_bytes(const KvView& kv)
{
    return (2 * (size_t)kv.n_layers * kv.batch * kv.n_kv_heads + 1) * sizeof(int);
}

bool verify_sm100_supported(const KvView& kv, int n_q, int variant)
{
    Plan pl;
    if (!make_plan(kv, n_q, kTile, variant == 2 ? 0 : variant, &pl)) return false;
    return kv.slot_stride >= kv.head_dim;
}

void verify_sm100_describe(const KvView& kv, int n_q, int max_ctx_len, int32_t out[8])
{
    for (int i = 0; i < 8; ++i) out[i] = 0;
    Plan pl;
    SplitPlan sp;
    int kind = 0;
    if (make_split_plan(kv, n_q, max_ctx_len, &sp) && make_plan(kv, sp.nA, max_ctx_len, 2, &pl)) kind = 3;
    else if (make_plan(kv, n_q, max_ctx_len, 0, &pl)) kind = pl.cached ? 2 : 1;
    if (!kind || kv.slot_stride < kv.head_dim) return;
    const int v[8] = {kind, pl.HG, pl.cph, pl.n_units, pl.N, pl.n_cache, pl.n_slots, pl.p_bufs};
    for (int i = 0; i < 8; ++i) out[i] = v[i];
}

size_t verify_sm100_workspace(const KvView& kv, int n_q, int max_ctx_len, int max_ctas)
{
    // the same bytes serve either variant and every shorter context, with or without the rows in two passes
    size_t best = 0;
    for (int ctx : {max_ctx_len, max_ctas > 0 ? max_ctx_len : kTile}) {
        Plan pl;
        if (make_plan(kv, n_q, ctx, 0, &pl, max_ctas) && pl.total > best) best = pl.total;
    }
    SplitPlan sp;
    if (make_split_plan(kv, n_q, max_ctx_len, &sp, max_ctas) && sp.total > best) best = sp.total;
    return best;
}

size_t verify_sm100_even_workspace(const KvView& kv, int n_q, int max_ctx_len)
{
    const int nsm = sm_count(), G = kv.n_q_heads / kv.n_kv_heads;
    size_t best = 0, ctr, ml, o;
    auto cached = [&](int rows) -> size_t {  // rows that the score cache can hold
        const int R = rows * G;
        const int hg = best_head_group(kv, max_ctx_len, nsm, cache_tiles((R + 15) / 16 * 16), false);
        return hg ? workspace_layout(kv, R, hg * (nsm / hg), &ctr, &ml, &o) : 0;
    };
    Plan pl;
    if (make_plan(kv, n_q, max_ctx_len, 1, &pl)) best = workspace_layout(kv, n_q * G, pl.HG * pl.cph, &ctr, &ml, &o);
    if (make_plan(kv, n_q, max_ctx_len, 2, &pl)) {
        const size_t b = cached(n_q);
        return b > best ? b : best;
    }
    SplitPlan sp;
    if (make_split_plan(kv, n_q, max_ctx_len, &sp)) {
        const size_t b = cached(sp.nA) + (sp.total - sp.main_bytes);  // (nA >= nB)
        if (b > best) best = b;
    }
    return best;
}

// Whether verify_sm100_launch would accept these arguments (same decisions, nothing launched).
bool verify_sm100_can_run(const VerifyArgs& a, int variant)
{
    const bool scaled = a.kv.k_scale || a.kv.v_scale || a.kv.fp8;
    if (scaled && (a.stat_per_head || a.stat_group_max)) return false;  // no such instance of the kernel
    if (a.stat_per_head || a.stat_group_max) {
        const int G = a.kv.n_q_heads / a.kv.n_kv_heads;
        Plan pl;
        if (variant == 1 || G > 8 || !make_plan(a.kv, a.n_q, a.max_ctx_len, 2, &pl, a.max_ctas)) return false;
        variant = 2;
    }
    SplitPlan sp;
    if (variant == 0 && make_split_plan(a.kv, a.n_q, a.max_ctx_len, &sp, a.max_ctas)) return a.workspace_bytes >= sp.total;
    Plan pl;
    if (!make_plan(a.kv, a.n_q, a.max_ctx_len, variant, &pl, a.max_ctas)) return false;
    if ((a.kv.k_scale || a.kv.v_scale) && !pl.cached) return false;
    return a.workspace_bytes >= pl.total;
}

int verify_sm100_launch(const VerifyArgs& a, int variant, cudaStream_t stream, int* used_variant)
{
    if ((a.kv.k_scale || a.kv.v_scale || a.kv.fp8) && (a.stat_per_head || a.stat_group_max))
        return SPEC_ERR_UNSUPPORTED_SHAPE;
    if (a.stat_per_head || a.stat_group_max) {
        // only the score-cache kernel keeps one score per attention head, for groups of up to 8;
        // everything else goes to the generic kernels
        const int G = a.kv.n_q_heads / a.kv.n_kv_heads;
        Plan pl;
        if (variant == 1 || G > 8 || !make_plan(a.kv, a.n_q, a.max_ctx_len, 2, &pl, a.max_ctas))
            return SPEC_ERR_UNSUPPORTED_SHAPE;
        variant = 2;
    }
    SplitPlan sp;
    if (variant == 0 && make_split_plan(a.kv, a.n_q, a.max_ctx_len, &sp, a.max_ctas)) {
        if (a.workspace_bytes < sp.total) return SPEC_ERR_WORKSPACE_TOO_SMALL;
        char* ws = static_cast<char*>(a.workspace);
        int32_t* ctx_a = reinterpret_cast<int32_t*>(ws + sp.ctx_off);
        float* second = reinterpret_cast<float*>(ws + sp.stat_off);
        const int64_t row_elems = (int64_t)a.kv.n_q_heads * a.kv.head_dim;
        shorten_ctx_kernel<<<1, 1, 0, stream>>>(a.ctx_len, sp.nB, ctx_a);
        count_launch(1);
        VerifyArgs pa = a;  // rows [0, nA): the context ends where the other rows begin
        pa.n_q = sp.nA;
        pa.ctx_len = ctx_a;
        pa.first_stat_row = a.first_stat_row < sp.nA ? a.first_stat_row : sp.nA;
        pa.workspace_bytes = sp.main_bytes;
        pa.hist = nullptr;  // the histogram is of the summed statistic: counted after the closing add
        int rc = verify_sm100_launch(pa, 2, stream, nullptr);
        if (rc != SPEC_OK) return rc;
        VerifyArgs pb = a;  // rows [nA, n_q) against the whole context; their statistic goes to scratch
        pb.n_q = sp.nB;
        pb.q = a.q + sp.nA * row_elems;
        pb.out = a.out_bf16 ? reinterpret_cast<float*>(reinterpret_cast<__nv_bfloat16*>(a.out) + sp.nA * row_elems)
                            : a.out + sp.nA * row_elems;
        pb.lse = a.lse ? a.lse + (int64_t)sp.nA * a.kv.n_q_heads : nullptr;
        pb.first_stat_row = a.first_stat_row > sp.nA ? a.first_stat_row - sp.nA : 0;
        pb.stats = second;
        pb.stat_stride = sp.stat_stride;
        pb.stat_accumulate = 0;
        pb.hist = nullptr;
        pb.workspace_bytes = sp.main_bytes;
        rc = verify_sm100_launch(pb, 2, stream, nullptr);
        if (rc != SPEC_OK) return rc;
        add_stats_kernel<<<sm_count(), 256, 0, stream>>>(a.stats, a.stat_stride, second, sp.stat_stride, a.ctx_len, a.max_ctx_len, sp.nB,
                                                         a.kv.n_kv_heads, a.stat_accumulate);
        count_launch(1);
        if (cudaGetLastError() != cudaSuccess) return SPEC_ERR_CUDA;
        if (used_variant) *used_variant = 3;
        return SPEC_OK;
    }
    Plan pl;
    if (!make_plan(a.kv, a.n_q, a.max_ctx_len, variant, &pl, a.max_ctas)) return SPEC_ERR_UNSUPPORTED_SHAPE;
    // per-(layer, KV head) scales (an 8-bit cache expanded to bf16): only the score-cache kernel applies them
    if ((a.kv.k_scale || a.kv.v_scale) && !pl.cached) return SPEC_ERR_UNSUPPORTED_SHAPE;
    if (a.workspace_bytes < pl.total) return SPEC_ERR_WORKSPACE_TOO_SMALL;
    const int G = a.kv.n_q_heads / a.kv.n_kv_heads;
    const int n_pages = a.kv.n_pages;
    CUtensorMap tk, tv, tq;
    FastParams fp;
    fp.whole_rows = 0;
    if (a.kv.fp8) {
        if (!encode_kv_map_u8(&tk, a.kv.k8, a.kv, n_pages, pl.box_rows, &fp) ||
            !encode_kv_map_u8(&tv, a.kv.v8, a.kv, n_pages, pl.box_rows, &fp))
            return SPEC_ERR_CUDA;
    } else if (pl.cached && copy_whole_rows(a.kv, pl.N) && encode_kv_map_rows(&tk, a.kv.k, a.kv, n_pages, &fp) &&
               encode_kv_map_rows(&tv, a.kv.v, a.kv, n_pages, &fp)) {
        fp.whole_rows = 1;
    } else if (!encode_kv_map(&tk, a.kv.k, a.kv, n_pages, pl.box_rows, &fp) ||
               !encode_kv_map(&tv, a.kv.v, a.kv, n_pages, pl.box_rows, &fp)) {
        return SPEC_ERR_CUDA;
    }
    if (!encode_q_map(&tq, a.q, a.kv, a.n_q, G)) return SPEC_ERR_CUDA;
    char* ws = static_cast<char*>(a.workspace);
    fp.a = a;
    fp.HG = pl.HG;
    fp.NHG = pl.cached ? 1 : a.kv.n_kv_heads / pl.HG;
    fp.cph = pl.cph;
    // two-sweep: units per layer and head groups per sequence; score cache: problems per sequence and KV heads
    set_divisor(&fp, 0, pl.cached ? a.kv.n_layers * a.kv.n_kv_heads : a.kv.batch * fp.NHG);
    set_divisor(&fp, 1, pl.cached ? a.kv.n_kv_heads : fp.NHG);
    set_divisor(&fp, 2, fp.cph);
    fp.n_cls = pl.n_cls;
    for (int f = 0; f < pl.n_cls; ++f) {
        fp.cls_size[f] = pl.cls_size[f];
        fp.cls_subs[f] = pl.cls_subs[f];
        set_divisor(&fp.cls_mul[f], &fp.cls_sh[f], pl.cls_size[f]);
    }
    fp.one_round = pl.cached && a.kv.batch == 1 && a.kv.n_layers * a.kv.n_kv_heads <= pl.HG;
    fp.n_counters = pl.n_counters;
    set_divisor(&fp, 3, a.kv.n_q_heads / a.kv.n_kv_heads);
    fp.n_units = pl.n_units;
    fp.N = pl.N;
    fp.R = a.n_q * G;
    fp.G = G;
    fp.D = a.kv.head_dim;
    fp.n_slots = pl.n_slots;
    fp.n_raw = pl.n_raw;
    fp.p_bufs = pl.p_bufs;
    fp.box_rows = pl.box_rows;
    fp.boxes = pl.boxes;
    fp.scale_log2 = a.kv.scale * 1.4426950408889634f;
    fp.counters = reinterpret_cast<int*>(ws + pl.ctr_off);
    fp.ml_part = reinterpret_cast<float2*>(ws + pl.ml_off);
    fp.o_part = reinterpret_cast<float*>(ws + pl.o_off);
    fp.status = reinterpret_cast<int*>(ws);
    fp.n_pages = n_pages;
    fp.n_cache = pl.n_cache;
    fp.wait_limit = wait_limit();
    // no memset: the workspace arrives zeroed and the kernel's last CTA re-zeroes the counters
    if (used_variant) *used_variant = pl.cached ? 2 : 1;
    const int grid = pl.cph * pl.HG;
    return pl.cached ? launch_cached(tk, tv, tq, fp, grid, pl.smem_bytes, stream)
                     : launch_twosweep(tk, tv, tq, fp, grid, pl.smem_bytes, stream);
}

}  // namespace spec
