// Cooperative search kernel instances (one query per block): LP, 4 k steps
// (see search_impl.cuh).
#include "search_impl.cuh"

namespace fg {
cudaError_t launch_coop_lp_k4(const DevIndex& ix, const SearchArgs& a, const SearchPlan& p,
                           cudaStream_t s) {
    return launch_occ<MODE_LP_K4, COOP_OCC>(ix, a, p, s);
}
cudaError_t occupancy_coop_lp_k4(const SearchPlan& p, int* blocks) {
    return occupancy_occ<MODE_LP_K4, COOP_OCC>(p, blocks);
}
}  // namespace fg
