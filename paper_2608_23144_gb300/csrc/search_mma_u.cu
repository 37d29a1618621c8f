// search_mma_u.cu — the AWSRC-U instances of search_mma.cuh.
#include "search_mma.cuh"

namespace awsrc {

int search_mma_tiles() { return kMmaTiles; }
int search_mma_slots(const Prm& pr) { return 152 * mma_per_sm(pr.variant, pr.C / 16); }

cudaError_t launch_search_mma_u(const Prm& pr, const LaunchDesc& ld, const uint64_t* masks, const float2* pairs,
                                int64_t n_items, awsrc_candidate* cands, cudaStream_t st) {
  return pr.P == 2 ? launch_mma_p<2, AWSRC_VARIANT_U>(pr, ld, masks, pairs, n_items, cands, st)
                   : launch_mma_p<4, AWSRC_VARIANT_U>(pr, ld, masks, pairs, n_items, cands, st);
}

}  // namespace awsrc
