// Tree walk over per-node results (Figure 2 of arXiv 2411.05289).
#pragma once

#include "spechub.h"
#include "spechub_args.cuh"
#include "spechub_common.cuh"

namespace spechub {

constexpr int kWalkThreads = 128;
constexpr int kWalkNodes = 128;   // trees of up to so many nodes: one warp per sequence

// One warp per sequence: the lanes fetch all nodes' results at once (one round trip to memory instead of two or three
// per level), and the path is followed in shared memory.  Larger trees: one thread per sequence.
// `blocks`: those of one walk; the three methods side by side walk in one launch.
__global__ void __launch_bounds__(kWalkThreads) walk_kernel(WalkKArgs A, int warp_per_seq, unsigned blocks) {
    __shared__ int sh_tok[kWalkThreads / 32][kWalkNodes], sh_acc[kWalkThreads / 32][kWalkNodes];
    pdl_begin();
    const unsigned which = blockIdx.x / blocks, block = blockIdx.x - which * blocks;
    const WalkArgs &a = A.w[which];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = warp_per_seq ? block * (kWalkThreads / 32) + warp : block * kWalkThreads + threadIdx.x;
    if (b >= a.batch) return;
    const long long r0 = static_cast<long long>(b) * a.nodes;
    if (warp_per_seq) {
        for (int n = lane; n < a.nodes; n += 32) {
            sh_tok[warp][n] = a.token[r0 + n];
            const bool leaf = a.node_kind && a.node_kind[n] == SPECHUB_NODE_LEAF;
            const int idx = a.accept_idx[r0 + n];
            // (a caller-supplied index that is no child ends the walk)
            sh_acc[warp][n] = leaf || idx < 0 || idx >= A.k ? -1 : a.child ? a.child[A.k * n + idx] : A.k * n + 1 + idx;
            if (!leaf && idx >= 0 && idx < A.k && sh_acc[warp][n] < 0) sh_acc[warp][n] = a.nodes;   // accepted, no node below
        }
        __syncwarp();
        if (lane != 0) return;
    }
    int n = 0, acc = 0, emitted = 0, step = 0;
    for (; step < a.levels && n >= 0 && n < a.nodes; ++step) {
        int tok, next;
        if (warp_per_seq) {
            tok = sh_tok[warp][n];
            next = sh_acc[warp][n];
        } else {
            tok = a.token[r0 + n];
            const bool leaf = a.node_kind && a.node_kind[n] == SPECHUB_NODE_LEAF;
            const int idx = a.accept_idx[r0 + n];
            next = leaf || idx < 0 || idx >= A.k ? -1 : a.child ? a.child[A.k * n + idx] : A.k * n + 1 + idx;
            if (!leaf && idx >= 0 && idx < A.k && next < 0) next = a.nodes;
        }
        if (a.path_nodes) a.path_nodes[static_cast<long long>(b) * a.levels + step] = n;
        if (a.path_tokens) a.path_tokens[static_cast<long long>(b) * a.levels + step] = tok;
        if (tok < 0) { ++step; break; }
        ++emitted;
        if (next < 0) { ++step; break; }   // rejected, or a leaf
        ++acc;
        n = next;
    }
    for (; step < a.levels; ++step) {
        if (a.path_nodes) a.path_nodes[static_cast<long long>(b) * a.levels + step] = -1;
        if (a.path_tokens) a.path_tokens[static_cast<long long>(b) * a.levels + step] = -1;
    }
    if (a.n_accepted) a.n_accepted[b] = acc;
    if (a.n_emitted) a.n_emitted[b] = emitted;
}

}  // namespace spechub
