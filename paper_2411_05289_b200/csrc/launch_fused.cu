// The three methods side by side.
#include "spechub_fused.cuh"
#include "spechub_launch.h"
#include "spechub_shapes.h"

namespace spechub {

int launch_fused_draft(const FusedArgs &f, int32_t *hub, float *draft_prob, unsigned rows, cudaStream_t s) {
    constexpr RowPass kFew = kFewRows<__nv_bfloat16, false>, kMany = kManyDrafts<__nv_bfloat16, false>;
    const int th = draft_threads(f.r.vocab, rows, true);
    const bool many = many_rows(th, rows) && f.r.vocab >= kRowRingVocab;
    if (th == 512) return launch_grid(fused_draft_kernel<512, kFew>, rows, 512, 0, 1, s, f, hub, draft_prob);
    if (th == 256) return launch_grid(fused_draft_kernel<256, kFew>, rows, 256, 0, 1, s, f, hub, draft_prob);
    if (th == 128 && many) return launch_grid(fused_draft_kernel<128, kMany>, rows, 128, kRowRingBytes<128, kMany>, 1, s, f, hub, draft_prob);
    if (th == 128) return launch_grid(fused_draft_kernel<128, kFew>, rows, 128, 0, 1, s, f, hub, draft_prob);
    if (th == 64) return launch_grid(fused_draft_kernel<64, kFew>, rows, 64, 0, 1, s, f, hub, draft_prob);
    return launch_grid(fused_draft_kernel<32, kFew>, rows, 32, 0, 1, s, f, hub, draft_prob);
}

int launch_fused_verify(const FusedArgs &f, unsigned rows, cudaStream_t s) {
    const int th = verify_threads(f.r.vocab, rows, 1024);
    if (!f.r.draft_stats_in) {
        if (th == 512) return launch_grid(fused_verify_kernel<512>, rows, 512, 0, 1, s, f);
        if (th == 256) return launch_grid(fused_verify_kernel<256>, rows, 256, 0, 1, s, f);
        return launch_grid(fused_verify_kernel<128>, rows, 128, 0, 1, s, f);
    }
    if (th == 512) return launch_grid(fused_verify_kernel<512, true>, rows, 512, 0, 1, s, f);
    if (th == 256) return launch_grid(fused_verify_kernel<256, true>, rows, 256, 0, 1, s, f);
    return launch_grid(fused_verify_kernel<128, true>, rows, 128, 0, 1, s, f);
}

}  // namespace spechub
