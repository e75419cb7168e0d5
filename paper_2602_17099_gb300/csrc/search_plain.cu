// K1, single-job launches: FP32 rows only.
#include "search_impl.cuh"

namespace rnsm {

cudaError_t launch_search_plain(const SearchArgs &a, int var, cudaStream_t st) {
    return launch_plain<false>(a, var, st);
}

}  // namespace rnsm
