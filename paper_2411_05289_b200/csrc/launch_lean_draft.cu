// Draft step and leaf rows of the large-vocabulary shapes.
#include "spechub_launch.h"
#include "spechub_lean.cuh"
#include "spechub_shapes.h"

namespace spechub {

template <int CS>
static int draft_group(const RowArgs &a, int method, unsigned rows, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    cfg.gridDim = dim3(rows * CS); cfg.blockDim = dim3(kLeanThreads); cfg.stream = s;
    return cudaLaunchKernelEx(&cfg, lean_draft_kernel<kLeanThreads, CS>, a, method) == cudaSuccess ? SPECHUB_OK : SPECHUB_ERR_LAUNCH;
}

int launch_lean_draft(int method, int cs, const RowArgs &a, unsigned rows, cudaStream_t s) {
    if (cs == 4) return draft_group<4>(a, method, rows, s);
    if (cs == 2) return draft_group<2>(a, method, rows, s);
    lean_draft_ck_kernel<kLeanDraftThreads><<<rows, kLeanDraftThreads, 0, s>>>(a, method);
    return launch_status();
}

// The leaf rows of an unsplit call (same CTA shape as the draft step).
int launch_lean_leaf(const RowArgs &a, const NodeOutPtrs *outs, int n_out, unsigned rows, cudaStream_t s) {
    LeafArgs la = {};
    la.r = a;
    la.n_out = n_out;
    for (int m = 0; m < n_out; ++m) la.out[m] = outs[m];
    lean_leaf_kernel<kLeanDraftThreads><<<rows, kLeanDraftThreads, 0, s>>>(la);
    return launch_status();
}

}  // namespace spechub
