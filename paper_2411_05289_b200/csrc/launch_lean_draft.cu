// Streaming draft step and leaf rows.
#include "spechub_launch.h"
#include "spechub_lean.cuh"
#include "spechub_shapes.h"

namespace spechub {

template <int CS>
static int draft_group(const RowArgs &a, int method, unsigned rows, cudaStream_t s) {
    return launch_grid(lean_draft_kernel<kLeanThreads, CS>, rows * CS, kLeanThreads, 0, CS, s, a, method);
}

template <typename LT, bool SHIFT>
static int draft_rows(const RowArgs &a, int method, bool keep_stats, unsigned rows, cudaStream_t s) {
    constexpr bool kWords = sizeof(LT) == 2 && !SHIFT;
    constexpr RowPass kFew = kFewRows<LT, SHIFT>, kMany = kManyDrafts<LT, SHIFT>;
    const int th = draft_threads(a.vocab, rows, kWords);
    const bool many = many_rows(th, rows) && (kMany != kRing || a.vocab >= kRowRingVocab);
    constexpr RowPass kMany64 = kManyRows<LT, SHIFT>;   // (rings: rows of 128 threads)
    if constexpr (kWords)
        if (th == 32) return launch_grid(lean_draft_ck_kernel<LT, SHIFT, 32, kFew>, rows, 32, 0, 1, s, a, method, keep_stats);
    if (th == 512) return launch_grid(lean_draft_ck_kernel<LT, SHIFT, 512, kFew>, rows, 512, 0, 1, s, a, method, keep_stats);
    if (th == 256) return launch_grid(lean_draft_ck_kernel<LT, SHIFT, 256, kFew>, rows, 256, 0, 1, s, a, method, keep_stats);
    if (th == 128 && many) return launch_grid(lean_draft_ck_kernel<LT, SHIFT, 128, kMany>, rows, 128, kRowRingBytes<128, kMany>, 1, s, a, method, keep_stats);
    if (th == 128) return launch_grid(lean_draft_ck_kernel<LT, SHIFT, 128, kFew>, rows, 128, 0, 1, s, a, method, keep_stats);
    if (many) return launch_grid(lean_draft_ck_kernel<LT, SHIFT, 64, kMany64>, rows, 64, 0, 1, s, a, method, keep_stats);
    return launch_grid(lean_draft_ck_kernel<LT, SHIFT, 64, kFew>, rows, 64, 0, 1, s, a, method, keep_stats);
}

int launch_lean_draft(int format, int method, int cs, const RowArgs &a, bool keep_stats, unsigned rows, cudaStream_t s) {
    if (cs == 4) return draft_group<4>(a, method, rows, s);
    if (cs == 2) return draft_group<2>(a, method, rows, s);
    if (format == kBf16) return draft_rows<__nv_bfloat16, false>(a, method, keep_stats, rows, s);
    if (format == kBf16Shift) return draft_rows<__nv_bfloat16, true>(a, method, keep_stats, rows, s);
    if (format == kF32) return draft_rows<float, false>(a, method, keep_stats, rows, s);
    return draft_rows<float, true>(a, method, keep_stats, rows, s);
}

template <typename LT, bool SHIFT>
static int leaf_rows(const LeafArgs &la, unsigned rows, cudaStream_t s) {
    constexpr RowPass kFew = kFewRows<LT, SHIFT>, kMany = kManyRows<LT, SHIFT>;
    const int th = draft_threads(la.r.vocab, rows, false);
    if (th == 512) return launch_grid(lean_leaf_kernel<LT, SHIFT, 512, kFew>, rows, 512, 0, 1, s, la);
    if (th == 256) return launch_grid(lean_leaf_kernel<LT, SHIFT, 256, kFew>, rows, 256, 0, 1, s, la);
    if (th == 128 && many_rows(th, rows)) return launch_grid(lean_leaf_kernel<LT, SHIFT, 128, kMany>, rows, 128, 0, 1, s, la);
    if (th == 128) return launch_grid(lean_leaf_kernel<LT, SHIFT, 128, kFew>, rows, 128, 0, 1, s, la);
    if (many_rows(th, rows)) return launch_grid(lean_leaf_kernel<LT, SHIFT, 64, kMany>, rows, 64, 0, 1, s, la);
    return launch_grid(lean_leaf_kernel<LT, SHIFT, 64, kFew>, rows, 64, 0, 1, s, la);
}

// The leaf rows of an unsplit call (same CTA shape as the draft step).
int launch_lean_leaf(int format, const RowArgs &a, int k, const NodeOutPtrs *outs, int n_out, unsigned rows, cudaStream_t s) {
    LeafArgs la = {};
    la.r = a;
    la.n_out = n_out;
    la.k = k;
    for (int m = 0; m < n_out; ++m) la.out[m] = outs[m];
    if (format == kBf16) return leaf_rows<__nv_bfloat16, false>(la, rows, s);
    if (format == kBf16Shift) return leaf_rows<__nv_bfloat16, true>(la, rows, s);
    if (format == kF32) return leaf_rows<float, false>(la, rows, s);
    return leaf_rows<float, true>(la, rows, s);
}

}  // namespace spechub
