// K1, multi-job launches: code rows first, FP32 rows for what they leave open.
#include "search_impl.cuh"

namespace rnsm {

cudaError_t launch_search_jobs_filter(const SearchArgs &a, int var, cudaStream_t st) {
    return launch_filter<true>(a, var, st);
}

}  // namespace rnsm
