// search_mma_pf.cu — the AWSRC-P_F instances of search_mma.cuh.
#include "search_mma.cuh"

namespace awsrc {

cudaError_t launch_search_mma_pf(const Prm& pr, const LaunchDesc& ld, const uint64_t* masks, int64_t n_items,
                                 awsrc_candidate* cands, cudaStream_t st) {
  return pr.P == 2 ? launch_mma_p<2, AWSRC_VARIANT_PF>(pr, ld, masks, nullptr, n_items, cands, st)
                   : launch_mma_p<4, AWSRC_VARIANT_PF>(pr, ld, masks, nullptr, n_items, cands, st);
}

}  // namespace awsrc
