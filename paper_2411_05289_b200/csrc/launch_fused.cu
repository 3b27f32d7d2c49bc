// The three methods side by side.
#include "spechub_fused.cuh"
#include "spechub_launch.h"
#include "spechub_shapes.h"

namespace spechub {

int launch_fused_draft(const FusedArgs &f, int32_t *hub, float *draft_prob, unsigned rows, cudaStream_t s) {
    fused_draft_kernel<kLeanDraftThreads><<<rows, kLeanDraftThreads, 0, s>>>(f, hub, draft_prob);
    return launch_status();
}

int launch_fused_verify(const FusedArgs &f, unsigned rows, cudaStream_t s) {
    if (!f.r.draft_stats_in) fused_verify_kernel<kLeanThreads><<<rows, kLeanThreads, 0, s>>>(f);
    else if (f.r.vocab <= kLeanSmallVocab) fused_verify_kernel<kLeanSmallThreads, true><<<rows, kLeanSmallThreads, 0, s>>>(f);
    else fused_verify_kernel<kLeanThreads, true><<<rows, kLeanThreads, 0, s>>>(f);
    return launch_status();
}

}  // namespace spechub
