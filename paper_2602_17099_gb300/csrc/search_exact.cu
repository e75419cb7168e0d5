// K1, single-job launches: code rows that are the rows (integers).
#include "search_impl.cuh"

namespace rnsm {

cudaError_t launch_search_exact(const SearchArgs &a, int var, cudaStream_t st) {
    return launch_exact<false>(a, var, st);
}

}  // namespace rnsm
