// Interface of the sm_100a (tcgen05 / TMA) verification path (verify_sm100.cu).
#pragma once
#include "spec_common.cuh"

namespace spec {
// variant: 0 = automatic (score-cache kernel when a CTA's share of keys fits tensor memory,
// else the two-sweep kernel), 1 = two-sweep only, 2 = score-cache only
bool verify_sm100_supported(const KvView& kv, int n_q, int variant);
// max_ctas > 0: for a call on at most that many CTAs
size_t verify_sm100_workspace(const KvView& kv, int n_q, int max_ctx_len, int max_ctas = 0);
// What a call would need whose CTAs are dealt out evenly to a divisor of the KV heads: the measure by which the calls without
// a workspace are taken or refused, whatever split they then run with.
size_t verify_sm100_even_workspace(const KvView& kv, int n_q, int max_ctx_len);
// Bytes behind the status block that the cross-CTA counters of a call may take: the same for every split of the same
// number of problems, so that calls with different row counts may share a workspace.
size_t verify_counter_bytes(const KvView& kv);
// spec_verify_attn_hist on at most max_ctas CTAs (0: no bound).
int verify_call(const spec_kv_t* kv, const void* q, int32_t n_q, const int32_t* ctx_len, int32_t max_ctx_len,
                int32_t stat_window, float* out, float* lse, float* stats, int64_t stat_stride, void* workspace,
                size_t workspace_bytes, uint32_t flags, uint32_t* score_hist, int max_ctas, void* cuda_stream);
// CTAs a call without a workspace may use in a scratch of `bytes`, or an error where the shape is refused
// (see verify_sm100_even_workspace).
int verify_ctas_within(const spec_kv_t* kv, int32_t n_q, int32_t max_ctx_len, size_t bytes);
// Clears the status word itself; *used_variant gets 1 (two-sweep) or 2 (score-cache).
int verify_sm100_launch(const VerifyArgs& a, int variant, cudaStream_t stream, int* used_variant);
// whether that call would accept the arguments (nothing is launched)
bool verify_sm100_can_run(const VerifyArgs& a, int variant);
// What AUTO would launch for this shape: out = {kernel (0 none, 1 two-sweep, 2 score-cache, 3 score-cache on two
// halves of the rows), KV heads per unit, CTAs per head, units, score columns, cached tiles, K/V slots, P buffers}.
void verify_sm100_describe(const KvView& kv, int n_q, int max_ctx_len, int32_t out[8]);

}  // namespace spec
