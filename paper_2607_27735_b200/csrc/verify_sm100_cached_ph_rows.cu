// Instances of the score-cache kernel with one score per attention head, tiles copied as whole rows.
#include "verify_sm100_cached.cuh"

namespace spec {
namespace sm100 {

int launch_cached_per_head_rows(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq, const FastParams& fp, int grid,
                                size_t smem_bytes, cudaStream_t stream)
{
    return launch_rows<true, false, false, true>(tk, tv, tq, fp, grid, smem_bytes, stream);
}

}  // namespace sm100
}  // namespace spec
