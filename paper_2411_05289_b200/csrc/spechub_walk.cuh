// Tree walk over per-node results (Figure 2 of arXiv 2411.05289).
#pragma once

#include "spechub.h"
#include "spechub_args.cuh"

namespace spechub {

// ------------------------------------------------------------------------------------------------
// Tree walk (Figure 2): one thread per sequence.
// ------------------------------------------------------------------------------------------------
__global__ void walk_kernel(WalkArgs a) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= a.batch) return;
    int n = 0, acc = 0, emitted = 0, step = 0;
    for (; step < a.levels && n >= 0 && n < a.nodes; ++step) {
        const long long r = static_cast<long long>(b) * a.nodes + n;
        const int tok = a.token[r];
        if (a.path_nodes) a.path_nodes[static_cast<long long>(b) * a.levels + step] = n;
        if (a.path_tokens) a.path_tokens[static_cast<long long>(b) * a.levels + step] = tok;
        if (tok < 0) { ++step; break; }
        ++emitted;
        if (a.node_kind && a.node_kind[n] == SPECHUB_NODE_LEAF) { ++step; break; }
        const int idx = a.accept_idx[r];
        if (idx < 0 || idx > 1) { ++step; break; }   // (a caller-supplied index outside {0, 1} ends the walk)
        ++acc;
        n = a.child ? a.child[2 * n + idx] : 2 * n + 1 + idx;
    }
    for (; step < a.levels; ++step) {
        if (a.path_nodes) a.path_nodes[static_cast<long long>(b) * a.levels + step] = -1;
        if (a.path_tokens) a.path_tokens[static_cast<long long>(b) * a.levels + step] = -1;
    }
    if (a.n_accepted) a.n_accepted[b] = acc;
    if (a.n_emitted) a.n_emitted[b] = emitted;
}

// ---- tree walk with k children per node -------------------------------------------------------------
__global__ void walk_k_kernel(WalkKArgs A) {
    const WalkArgs &a = A.w;
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= a.batch) return;
    int n = 0, acc = 0, emitted = 0, step = 0;
    for (; step < a.levels && n >= 0 && n < a.nodes; ++step) {
        const long long r = static_cast<long long>(b) * a.nodes + n;
        const int tok = a.token[r];
        if (a.path_nodes) a.path_nodes[static_cast<long long>(b) * a.levels + step] = n;
        if (a.path_tokens) a.path_tokens[static_cast<long long>(b) * a.levels + step] = tok;
        if (tok < 0) { ++step; break; }
        ++emitted;
        if (a.node_kind && a.node_kind[n] == SPECHUB_NODE_LEAF) { ++step; break; }
        const int idx = a.accept_idx[r];
        if (idx < 0 || idx >= A.k) { ++step; break; }
        ++acc;
        n = a.child ? a.child[A.k * n + idx] : A.k * n + 1 + idx;
    }
    for (; step < a.levels; ++step) {
        if (a.path_nodes) a.path_nodes[static_cast<long long>(b) * a.levels + step] = -1;
        if (a.path_tokens) a.path_tokens[static_cast<long long>(b) * a.levels + step] = -1;
    }
    if (a.n_accepted) a.n_accepted[b] = acc;
    if (a.n_emitted) a.n_emitted[b] = emitted;
}

}  // namespace spechub
