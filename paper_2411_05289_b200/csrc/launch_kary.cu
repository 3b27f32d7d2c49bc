// More than two drafts per node (any shape), tree walk.
#include "spechub_kary.cuh"
#include "spechub_launch.h"
#include "spechub_walk.cuh"

namespace spechub {

int launch_kary_draft(int dtype, bool aligned, int th, const KaryArgs &a, unsigned rows, cudaStream_t s) {
    if (dtype == SPECHUB_BF16) {
        if (aligned) kary_draft_kernel<__nv_bfloat16, true><<<rows, th, 0, s>>>(a);
        else kary_draft_kernel<__nv_bfloat16, false><<<rows, th, 0, s>>>(a);
    } else {
        if (aligned) kary_draft_kernel<float, true><<<rows, th, 0, s>>>(a);
        else kary_draft_kernel<float, false><<<rows, th, 0, s>>>(a);
    }
    return launch_status();
}

int launch_kary_verify(int dtype, bool aligned, int th, const KaryArgs &a, unsigned rows, cudaStream_t s) {
    if (dtype == SPECHUB_BF16) {
        if (aligned) kary_verify_kernel<__nv_bfloat16, true><<<rows, th, 0, s>>>(a);
        else kary_verify_kernel<__nv_bfloat16, false><<<rows, th, 0, s>>>(a);
    } else {
        if (aligned) kary_verify_kernel<float, true><<<rows, th, 0, s>>>(a);
        else kary_verify_kernel<float, false><<<rows, th, 0, s>>>(a);
    }
    return launch_status();
}

int launch_walk(const WalkKArgs &wk, cudaStream_t s) {
    const int blocks = (wk.w.batch + 127) / 128;
    if (wk.k > 2) walk_k_kernel<<<blocks, 128, 0, s>>>(wk);
    else walk_kernel<<<blocks, 128, 0, s>>>(wk.w);
    return launch_status();
}

}  // namespace spechub
