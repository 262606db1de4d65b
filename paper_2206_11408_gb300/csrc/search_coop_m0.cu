// Cooperative search kernel instances (one query per block): plain search
// (see search_impl.cuh).
#include "search_impl.cuh"

namespace fg {
cudaError_t launch_coop_m0(const DevIndex& ix, const SearchArgs& a, const SearchPlan& p,
                           cudaStream_t s) {
    return launch_occ<FINGER_MODE_PLAIN, COOP_OCC>(ix, a, p, s);
}
cudaError_t occupancy_coop_m0(const SearchPlan& p, int* blocks) {
    return occupancy_occ<FINGER_MODE_PLAIN, COOP_OCC>(p, blocks);
}
}  // namespace fg
