// K1, multi-job launches: code rows that are the rows (integers).
#include "search_impl.cuh"

namespace rnsm {

cudaError_t launch_search_jobs_exact(const SearchArgs &a, int var, cudaStream_t st) {
    return launch_exact<true>(a, var, st);
}

}  // namespace rnsm
