// Streaming verification of one method: its kernels and which of them a call takes.
#pragma once

#include "spechub_launch.h"
#include "spechub_lean.cuh"
#include "spechub_shapes.h"

namespace spechub {

template <int METHOD, int CS>
int verify_split(const RowArgs &a, unsigned rows, cudaStream_t s) {
    return launch_grid(lean_verify_kernel<__nv_bfloat16, false, METHOD, kLeanThreads, CS>, rows * CS, kLeanThreads, 0, CS, s, a);
}

constexpr int kRingVocab = 65536;

// One CTA per row, the passes fed by per-warp rings of bulk copies (spechub_ring.cuh).
template <int METHOD>
int verify_ring(const RowArgs &a, unsigned rows, cudaStream_t s) {
    auto kern = lean_verify_kernel<__nv_bfloat16, false, METHOD, kLeanThreads, 1, true>;
    constexpr int smem = kLeanThreads / 32 * kRingWarpBytes;
    static bool configured[kMaxDevices] = {};
    const int rc = allow_smem(reinterpret_cast<const void *>(kern), smem, configured);
    if (rc != SPECHUB_OK) return rc;
    return launch_grid(kern, rows, kLeanThreads, smem, 1, s, a);
}

// One CTA per row.  STATS: the draft row's statistics come from the draft step.
template <typename LT, bool SHIFT, int METHOD, bool STATS>
int verify_rows(const RowArgs &a, unsigned rows, cudaStream_t s) {
    const int th = verify_threads(a.vocab, rows, SHIFT ? 768 : 1024);
    if (th == 512) return launch_grid(lean_verify_kernel<LT, SHIFT, METHOD, 512, 1, false, STATS>, rows, 512, 0, 1, s, a);
    if (th == 256) return launch_grid(lean_verify_kernel<LT, SHIFT, METHOD, 256, 1, false, STATS>, rows, 256, 0, 1, s, a);
    return launch_grid(lean_verify_kernel<LT, SHIFT, METHOD, 128, 1, false, STATS>, rows, 128, 0, 1, s, a);
}

template <int METHOD>
int launch_lean_verify_method(int format, int cs, const RowArgs &a, unsigned rows, cudaStream_t s) {
    if (cs == 4) return verify_split<METHOD, 4>(a, rows, s);
    if (cs == 2) return verify_split<METHOD, 2>(a, rows, s);
    if (a.node_kind) {
        const NodeOutPtrs o = {a.accept_idx, a.token, a.hub, a.beta, a.rate, a.status};
        const int lrc = launch_lean_leaf(format, a, 2, &o, 1, rows, s);
        if (lrc != SPECHUB_OK) return lrc;
    }
    const bool stats = cs == 0 && a.draft_stats_in;
    if (format == kBf16Shift)
        return stats ? verify_rows<__nv_bfloat16, true, METHOD, true>(a, rows, s) : verify_rows<__nv_bfloat16, true, METHOD, false>(a, rows, s);
    if (format == kF32Shift)
        return stats ? verify_rows<float, true, METHOD, true>(a, rows, s) : verify_rows<float, true, METHOD, false>(a, rows, s);
    if (format == kF32)
        return stats ? verify_rows<float, false, METHOD, true>(a, rows, s) : verify_rows<float, false, METHOD, false>(a, rows, s);
    if (stats) return verify_rows<__nv_bfloat16, false, METHOD, true>(a, rows, s);
    if (cs == 1) return verify_split<METHOD, 1>(a, rows, s);
    // Rings of bulk copies: rows that L2 does not hold from pass to pass, enough of them for CTAs of 256 threads (1984
    // rows, V = 128256: RRS 468 us, without rings 537, RRSw 489, 530; V = 32000: 478, 459, 499, 455; 112 rows, V =
    // 128256: RRS 68 us, CTAs of 512 threads without rings 39).
    if constexpr (METHOD != kSpecHub)
        if (a.vocab >= kRingVocab && verify_threads(a.vocab, rows, 1024) == kLeanThreads) return verify_ring<METHOD>(a, rows, s);
    return verify_rows<__nv_bfloat16, false, METHOD, false>(a, rows, s);
}

}  // namespace spechub
