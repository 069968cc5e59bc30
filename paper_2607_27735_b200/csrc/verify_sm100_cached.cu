// Instances of the score-cache kernel over a bf16 cache, and the choice among all of them.  (The instances are spread
// over several files so that they compile side by side.)
#include "verify_sm100_cached.cuh"

namespace spec {
namespace sm100 {

int launch_cached_per_head(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq, const FastParams& fp, int grid,
                           size_t smem_bytes, cudaStream_t stream);
int launch_cached_rows(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq, const FastParams& fp, int grid,
                       size_t smem_bytes, cudaStream_t stream);
int launch_cached_per_head_rows(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq, const FastParams& fp, int grid,
                                size_t smem_bytes, cudaStream_t stream);
int launch_cached_scaled(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq, const FastParams& fp, int grid,
                         size_t smem_bytes, cudaStream_t stream);
int launch_cached_8bit(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq, const FastParams& fp, int grid,
                       size_t smem_bytes, cudaStream_t stream);

int launch_cached(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq, const FastParams& fp, int grid,
                  size_t smem_bytes, cudaStream_t stream)
{
    const bool ph = fp.a.stat_per_head != 0 || fp.a.stat_group_max != 0;
    // per-(layer, KV head) scales: instances of their own (the bf16 instances carry no code for them),
    // built for the per-KV-head statistic only
    const bool sc = fp.a.kv.k_scale != nullptr || fp.a.kv.v_scale != nullptr;
    const bool f8 = fp.a.kv.fp8 != 0;  // 8-bit cache read directly (always an SC instance)
    if ((sc || f8) && (ph || fp.whole_rows)) return SPEC_ERR_UNSUPPORTED_SHAPE;
    if (f8) return launch_cached_8bit(tk, tv, tq, fp, grid, smem_bytes, stream);
    if (sc) return launch_cached_scaled(tk, tv, tq, fp, grid, smem_bytes, stream);
    if (ph && fp.whole_rows) return launch_cached_per_head_rows(tk, tv, tq, fp, grid, smem_bytes, stream);
    if (ph) return launch_cached_per_head(tk, tv, tq, fp, grid, smem_bytes, stream);
    if (fp.whole_rows) return launch_cached_rows(tk, tv, tq, fp, grid, smem_bytes, stream);
    return launch_rows<false, false, false, false>(tk, tv, tq, fp, grid, smem_bytes, stream);
}

}  // namespace sm100
}  // namespace spec
