// Instantiates the search kernel for one distance mode (see search_team.cuh).
#include "search_team.cuh"

namespace bang {
cudaError_t launch_search_q8(const SearchArgs &a, int dtype, size_t smem, cudaStream_t st)
{
    return launch_team<kModeQ8>(a, dtype, smem, st);
}
}  // namespace bang
