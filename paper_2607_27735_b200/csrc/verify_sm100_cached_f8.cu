// Instances of the score-cache kernel over an 8-bit cache.
#include "verify_sm100_cached.cuh"

namespace spec {
namespace sm100 {

int launch_cached_8bit(const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tq, const FastParams& fp, int grid,
                       size_t smem_bytes, cudaStream_t stream)
{
    return launch_rows<false, true, true, false>(tk, tv, tq, fp, grid, smem_bytes, stream);
}

}  // namespace sm100
}  // namespace spec
