// The three methods side by side.
#include "spechub_fused.cuh"
#include "spechub_launch.h"
#include "spechub_shapes.h"

namespace spechub {

int launch_fused_draft(const FusedArgs &f, int32_t *hub, float *draft_prob, unsigned rows, cudaStream_t s) {
    const int th = draft_threads(f.r.vocab, rows);
    if (th == 512) fused_draft_kernel<512><<<rows, 512, 0, s>>>(f, hub, draft_prob);
    else if (th == 256) fused_draft_kernel<256><<<rows, 256, 0, s>>>(f, hub, draft_prob);
    else fused_draft_kernel<128><<<rows, 128, 0, s>>>(f, hub, draft_prob);
    return launch_status();
}

int launch_fused_verify(const FusedArgs &f, unsigned rows, cudaStream_t s) {
    const int th = verify_threads(f.r.vocab, rows);
    if (!f.r.draft_stats_in) fused_verify_kernel<kLeanThreads><<<rows, kLeanThreads, 0, s>>>(f);
    else if (th == 512) fused_verify_kernel<512, true><<<rows, 512, 0, s>>>(f);
    else if (th == 256) fused_verify_kernel<256, true><<<rows, 256, 0, s>>>(f);
    else fused_verify_kernel<128, true><<<rows, 128, 0, s>>>(f);
    return launch_status();
}

}  // namespace spechub
