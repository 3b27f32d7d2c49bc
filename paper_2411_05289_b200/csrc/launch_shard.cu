// Vocabulary-sharded phases.
#include "spechub_launch.h"
#include "spechub_shard.cuh"
#include "spechub_shard_rrs.cuh"

namespace spechub {

template <typename LT, bool AL>
static void shard_phase(int phase, const ShardArgs &a, unsigned rows, int th, cudaStream_t s) {
    if (phase == kPhaseStats) shard_stats_kernel<LT, AL><<<rows, th, 0, s>>>(a);
    else if (phase == kPhaseSums) shard_sums_kernel<LT, AL><<<rows, th, 0, s>>>(a);
    else if (phase == kPhaseDecide) shard_decide_kernel<LT, AL><<<rows, th, 0, s>>>(a);
    else if (phase == kPhaseDraft) shard_draft_kernel<LT, AL><<<rows, th, 0, s>>>(a);
    else if (phase == kPhaseRrsSums) rrs_shard_sums_kernel<LT, AL><<<rows, th, 0, s>>>(a);
    else if (phase == kPhaseRrsDecide) rrs_shard_decide_kernel<LT, AL><<<rows, th, 0, s>>>(a);
    else rrs_shard_draft_kernel<LT, AL><<<rows, th, 0, s>>>(a);
}

int launch_shard_phase(int phase, int dtype, bool aligned, int th, const ShardArgs &a, unsigned rows, cudaStream_t s) {
    if (dtype == SPECHUB_BF16) {
        if (aligned) shard_phase<__nv_bfloat16, true>(phase, a, rows, th, s);
        else shard_phase<__nv_bfloat16, false>(phase, a, rows, th, s);
    } else {
        if (aligned) shard_phase<float, true>(phase, a, rows, th, s);
        else shard_phase<float, false>(phase, a, rows, th, s);
    }
    return launch_status();
}

int launch_shard_draft_finish(bool rrs, const ShardArgs &a, cudaStream_t s) {
    const unsigned blocks = (unsigned)((a.rows + 127) / 128);
    if (rrs) rrs_shard_draft_finish_kernel<<<blocks, 128, 0, s>>>(a);
    else shard_draft_finish_kernel<<<blocks, 128, 0, s>>>(a);
    return launch_status();
}

}  // namespace spechub
