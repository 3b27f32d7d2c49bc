// More than two drafts per node; tree walk.
#include "spechub_launch.h"
#include "spechub_lean_kary.cuh"
#include "spechub_shapes.h"
#include "spechub_walk.cuh"

namespace spechub {

template <typename LT, bool SHIFT>
static int kary_draft(const KaryArgs &a, unsigned rows, cudaStream_t s) {
    const int th = draft_threads(a.r.vocab, rows);
    if (th == 512) lean_kary_draft_kernel<LT, SHIFT, 512><<<rows, 512, 0, s>>>(a);
    else if (th == 256) lean_kary_draft_kernel<LT, SHIFT, 256><<<rows, 256, 0, s>>>(a);
    else if (th == 128) lean_kary_draft_kernel<LT, SHIFT, 128><<<rows, 128, 0, s>>>(a);
    else lean_kary_draft_kernel<LT, SHIFT, 64><<<rows, 64, 0, s>>>(a);
    return launch_status();
}
template <typename LT, bool SHIFT>
static int kary_verify(const KaryArgs &a, unsigned rows, cudaStream_t s) {
    const int th = verify_threads(a.r.vocab, rows);
    if (th == 512) lean_kary_verify_kernel<LT, SHIFT, 512><<<rows, 512, 0, s>>>(a);
    else if (th == 256) lean_kary_verify_kernel<LT, SHIFT, 256><<<rows, 256, 0, s>>>(a);
    else lean_kary_verify_kernel<LT, SHIFT, 128><<<rows, 128, 0, s>>>(a);
    return launch_status();
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

int launch_walk(const WalkKArgs &wk, cudaStream_t s) {
    const int blocks = (wk.w.batch + 127) / 128;
    if (wk.k > 2) walk_k_kernel<<<blocks, 128, 0, s>>>(wk);
    else walk_kernel<<<blocks, 128, 0, s>>>(wk.w);
    return launch_status();
}

}  // namespace spechub
