// More than two drafts per node; tree walk.
#include "spechub_launch.h"
#include "spechub_lean_kary.cuh"
#include "spechub_shapes.h"
#include "spechub_walk.cuh"

namespace spechub {

template <typename LT, bool SHIFT>
static int kary_draft(const KaryArgs &a, unsigned rows, cudaStream_t s) {
    constexpr bool kWords = sizeof(LT) == 2 && !SHIFT;
    constexpr RowPass kFew = kFewRows<LT, SHIFT>, kMany = kManyRows<LT, SHIFT>;
    const int th = draft_threads(a.r.vocab, rows, kWords);
    if constexpr (kWords)
        if (th == 32) return launch_grid(lean_kary_draft_kernel<LT, SHIFT, 32, kFew>, rows, 32, 0, 1, s, a);
    if (th == 512) return launch_grid(lean_kary_draft_kernel<LT, SHIFT, 512, kFew>, rows, 512, 0, 1, s, a);
    if (th == 256) return launch_grid(lean_kary_draft_kernel<LT, SHIFT, 256, kFew>, rows, 256, 0, 1, s, a);
    if (th == 128 && many_rows(th, rows)) return launch_grid(lean_kary_draft_kernel<LT, SHIFT, 128, kMany>, rows, 128, 0, 1, s, a);
    if (th == 128) return launch_grid(lean_kary_draft_kernel<LT, SHIFT, 128, kFew>, rows, 128, 0, 1, s, a);
    if (many_rows(th, rows)) return launch_grid(lean_kary_draft_kernel<LT, SHIFT, 64, kMany>, rows, 64, 0, 1, s, a);
    return launch_grid(lean_kary_draft_kernel<LT, SHIFT, 64, kFew>, rows, 64, 0, 1, s, a);
}
template <typename LT, bool SHIFT>
static int kary_verify(const KaryArgs &a, unsigned rows, cudaStream_t s) {
    const int th = verify_threads(a.r.vocab, rows, SHIFT ? 768 : 1024);
    if (th == 512) return launch_grid(lean_kary_verify_kernel<LT, SHIFT, 512>, rows, 512, 0, 1, s, a);
    if (th == 256) return launch_grid(lean_kary_verify_kernel<LT, SHIFT, 256>, rows, 256, 0, 1, s, a);
    return launch_grid(lean_kary_verify_kernel<LT, SHIFT, 128>, rows, 128, 0, 1, s, a);
}

int launch_kary_draft(int format, const KaryArgs &a, unsigned rows, cudaStream_t s) {
    if (format == kBf16) return kary_draft<__nv_bfloat16, false>(a, rows, s);
    if (format == kBf16Shift) return kary_draft<__nv_bfloat16, true>(a, rows, s);
    if (format == kF32) return kary_draft<float, false>(a, rows, s);
    return kary_draft<float, true>(a, rows, s);
}

int launch_kary_verify(int format, const KaryArgs &a, unsigned rows, cudaStream_t s) {
    if (a.r.node_kind) {
        const NodeOutPtrs o = {a.r.accept_idx, a.r.token, a.r.hub, a.r.beta, a.r.rate, a.r.status};
        const int rc = launch_lean_leaf(format, a.r, a.k, &o, 1, rows, s);
        if (rc != SPECHUB_OK) return rc;
    }
    if (format == kBf16) return kary_verify<__nv_bfloat16, false>(a, rows, s);
    if (format == kBf16Shift) return kary_verify<__nv_bfloat16, true>(a, rows, s);
    if (format == kF32) return kary_verify<float, false>(a, rows, s);
    return kary_verify<float, true>(a, rows, s);
}

int launch_walk(const WalkKArgs &wk, int n, cudaStream_t s) {
    const int warp_per_seq = wk.w[0].nodes <= kWalkNodes, per = warp_per_seq ? kWalkThreads / 32 : kWalkThreads;
    const unsigned blocks = (wk.w[0].batch + per - 1) / per;
    return launch_grid(walk_kernel, n * blocks, kWalkThreads, 0, 1, s, wk, warp_per_seq, blocks);
}

}  // namespace spechub
