// Verification of the large-vocabulary shapes, rows streamed from HBM / L2.
#include "spechub_launch.h"
#include "spechub_lean.cuh"
#include "spechub_shapes.h"

namespace spechub {

template <int METHOD, int CS>
static int verify_cs(const RowArgs &a, unsigned rows, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = CS > 1 ? 1 : 0;
    cfg.gridDim = dim3(rows * CS); cfg.blockDim = dim3(kLeanThreads); cfg.stream = s;
    return cudaLaunchKernelEx(&cfg, lean_verify_kernel<METHOD, kLeanThreads, CS>, a) == cudaSuccess ? SPECHUB_OK : SPECHUB_ERR_LAUNCH;
}

// One CTA per row, the passes fed by per-warp rings of bulk copies (spechub_ring.cuh).
template <int METHOD>
static int verify_ring(const RowArgs &a, unsigned rows, cudaStream_t s) {
    auto kern = lean_verify_kernel<METHOD, kLeanThreads, 1, true>;
    constexpr int smem = kLeanThreads / 32 * kRingWarpBytes;
    static bool configured[kMaxDevices] = {};
    const int rc = allow_smem(reinterpret_cast<const void *>(kern), smem, configured);
    if (rc != SPECHUB_OK) return rc;
    kern<<<rows, kLeanThreads, smem, s>>>(a);
    return launch_status();
}

// The draft row's statistics come from the draft step.
template <int METHOD>
static int verify_stats(const RowArgs &a, unsigned rows, cudaStream_t s) {
    if (a.vocab <= kLeanSmallVocab)
        lean_verify_kernel<METHOD, kLeanSmallThreads, 1, false, true><<<rows, kLeanSmallThreads, 0, s>>>(a);
    else
        lean_verify_kernel<METHOD, kLeanThreads, 1, false, true><<<rows, kLeanThreads, 0, s>>>(a);
    return launch_status();
}

template <int METHOD>
static int verify_method(int cs, const RowArgs &a, unsigned rows, cudaStream_t s) {
    if (cs == 4) return verify_cs<METHOD, 4>(a, rows, s);
    if (cs == 2) return verify_cs<METHOD, 2>(a, rows, s);
    if (a.node_kind) {
        const NodeOutPtrs o = {a.accept_idx, a.token, a.hub, a.beta, a.rate, a.status};
        const int lrc = launch_lean_leaf(a, &o, 1, rows, s);
        if (lrc != SPECHUB_OK) return lrc;
    }
    if (cs == 0 && a.draft_stats_in) return verify_stats<METHOD>(a, rows, s);
    if constexpr (METHOD != kSpecHub)
        if (cs == 0) return verify_ring<METHOD>(a, rows, s);
    return verify_cs<METHOD, 1>(a, rows, s);
}

int launch_lean_verify(int method, int cs, const RowArgs &a, unsigned rows, cudaStream_t s) {
    if (method == kSpecHub) return verify_method<kSpecHub>(cs, a, rows, s);
    if (method == kRRS) return verify_method<kRRS>(cs, a, rows, s);
    return verify_method<kRRSw>(cs, a, rows, s);
}

}  // namespace spechub
