// Pieces that the kernels share: pass A of the vocabulary-sharded phases (any row, fp32 or bf16), probabilities with
// pinned rounding, the acceptance test, a row's outputs.
#pragma once

#include "spechub.h"
#include "spechub_common.cuh"
#include "spechub_args.cuh"

namespace spechub {

// a draft kernel that keeps no statistics leaves a record that no verification accepts
__device__ __forceinline__ void void_draft_stat(const RowArgs &a, long long r) {
    if (a.draft_stats_out) static_cast<uint4 *>(a.draft_stats_out)[r] = make_uint4(0u, 0u, 0u, 0u);
}

// What a record's tag says about the row beside its temperature.  Verification of rows that are not read in whole words
// did not always look at records, so a buffer that an earlier iteration filled may still come with them, and the one
// logit that is compared with the recorded maximum is the same now and then: those records also carry a mark of 32 more
// logits, spread over the row.  (The 32 lanes of a warp; vocab >= 64.)
template <typename LT>
__device__ __forceinline__ unsigned row_mark(const LT *row, int vocab) {
    const unsigned i = 2 * (threadIdx.x & 31) + 1;
    const unsigned h = __float_as_uint(load_one<LT>(row, static_cast<int>(i) * (vocab >> 6))) * (0x9e3779b0u + i);
    return __reduce_xor_sync(kFull, h ^ (h >> 15));
}
__device__ __forceinline__ unsigned stat_tag(float k, unsigned mark = 0) { return kDraftStatTag ^ __float_as_uint(k) ^ mark; }

struct WarpPart {  // per-warp (max, argmax, sum without the argmax) of one row
    float ml[kMaxWarps], sx[kMaxWarps];
    int idx[kMaxWarps];
};
struct Partials {  // per-warp partials kept for the samplers, in shared memory
    WarpPart p, q;
    float acc[4][kMaxWarps];
    float mass[kMaxWarps];
    float bc[16];
    int bi[8];
    int tok;
};

__device__ __forceinline__ float temperature_of(const RowArgs &a, int b) {
    return a.temperature_per_seq ? a.temperature_per_seq[b] : a.temperature;
}

// Pass A over one row: per-warp (max, argmax, sum without the argmax) to shared memory; the
// block-wide result is returned to every thread.  Target and draft rows go through the same
// arithmetic, so identical rows give bit-identical probabilities (p = q then cancels exactly).
template <typename LT, bool AL>
__device__ ArgMaxSum pass_a(const Geo &g, const LT *row, float k, WarpPart &wp) {
    constexpr int VW = VecOf<LT>::W;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    ArgMaxSum st;
    st.init();
    for (int vi = g.seg_lo(warp) + lane; vi < g.seg_hi(warp); vi += 32) {
        float v[VW];
        load_vec<LT, AL>(row, vi, g.V, v);
        argmaxsum_push<VW>(st, v, vi * VW, k);
    }
    st = argmaxsum_warp(st, k);
    if (lane == 0) { wp.ml[warp] = st.ml; wp.sx[warp] = st.sx; wp.idx[warp] = st.idx; }
    __syncthreads();
    ArgMaxSum tot;
    tot.init();
    for (int w = 0; w < g.nwarps; ++w) {
        ArgMaxSum o;
        o.ml = wp.ml[w]; o.c = shift_of(o.ml, k); o.sx = wp.sx[w]; o.idx = wp.idx[w];
        tot = argmaxsum_merge(tot, o, k);
    }
    return tot;
}

// Probability of one logit.  The product is rounded on its own (no contraction into a later
// subtraction), so that identical target and draft rows give p(y) - q(y) = 0 exactly.
__device__ __forceinline__ float prob_of(float logit, float k, float c, float invZ) {
    return __fmul_rn(ex2(__fmaf_rn(logit, k, -c)), invZ);
}
// d = p - q and t = max(p - q, 0) - s*q, with pinned rounding so that the sums of pass B and
// the weights the sampler recomputes are the same numbers.
__device__ __forceinline__ void transport_terms(float pp, float qq, float s, float &d, float &t) {
    d = __fsub_rn(pp, qq);
    t = __fmaf_rn(-s, qq, fmaxf(d, 0.f));
}

__device__ __forceinline__ bool finite_pos(float x) { return x > 0.f && x < __int_as_float(0x7f800000); }

// ------------------------------------------------------------------------------------------------
// Verification of one row.
// ------------------------------------------------------------------------------------------------
struct NodeResult {
    int accept_idx, token, hub;
    float beta[2], rate[3];
    uint32_t status;
};

__device__ __forceinline__ void write_node(const RowArgs &a, long long r, const NodeResult &o) {
    a.accept_idx[r] = o.accept_idx;
    a.token[r] = o.token;
    if (a.hub) a.hub[r] = o.hub;
    if (a.beta) { a.beta[2 * r] = o.beta[0]; a.beta[2 * r + 1] = o.beta[1]; }
    if (a.rate) { a.rate[3 * r] = o.rate[0]; a.rate[3 * r + 1] = o.rate[1]; a.rate[3 * r + 2] = o.rate[2]; }
    if (a.status) a.status[r] = o.status;
}

// strict multiplicative acceptance test; fills beta = min(N/D, 1)
__device__ __forceinline__ bool accept_test(float r, float N, float D, float &beta, bool performed,
                                            uint32_t &status) {
    beta = (D > 0.f) ? fminf(N / D, 1.f) : 0.f;
    if (!performed) return false;
    if (!(D > 0.f)) { status |= SPECHUB_ST_ZERO_MASS_DRAFT; return false; }
    return r * D < N;
}

// Block-wide sum of up to 4 per-thread accumulators; per-warp values stay in sh.acc[i][w].
template <int NACC>
__device__ __forceinline__ void block_sums(const Geo &g, float (&x)[NACC], Partials &sh) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < NACC; ++i) {
        const float s = warp_sum(x[i]);
        if (lane == 0) sh.acc[i][warp] = s;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NACC; ++i) {
        float t = 0.f;
        for (int w = 0; w < g.nwarps; ++w) t += sh.acc[i][w];
        x[i] = t;
    }
}

}  // namespace spechub
