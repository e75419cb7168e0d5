// K1, single-job launches: code rows first, FP32 rows for what they leave open.
#include "search_impl.cuh"

namespace rnsm {

cudaError_t launch_search_filter(const SearchArgs &a, int var, cudaStream_t st) {
    return launch_filter<false>(a, var, st);
}

}  // namespace rnsm
