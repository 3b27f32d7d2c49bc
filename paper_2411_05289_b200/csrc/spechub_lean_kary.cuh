// Streaming kernels for Algorithm 1 (arXiv 2411.05289) with k > 2 drafts per node: one CTA per row, the passes and
// the samplers of spechub_lean.cuh.
//
// With P_0 = p, m_0 = 1, stage j (1 <= j <= k):
//   test j:  accept x_j  iff  r_j m_{j-1} q_j(x_j) < P_{j-1}(x_j);   P_j = max(P_{j-1} - m_{j-1} q_j, 0), m_j = sum P_j
// where q_j = q (RRS) or q with x_1..x_{j-1} taken out and renormalised (RRSw).  An id that no stage takes out of q
// sees the same subtractions one after another, so P_j(y) = max(p(y) - C_j q(y), 0) with C_j the sum of the stages'
// coefficients m g: a stage is one pass over the rows as they are, 2 exponentials per id, and nothing is kept per id.
// Without replacement a draft loses its q once drawn, and its C stops growing: the drafts that can be taken out,
// x_1..x_{k-1}, stay out of all passes and are added to every sum as single terms (all terms are positive: nothing
// cancels).  Without probability outputs a row ends with the test that accepts.
//
// Against the stages run over exponentials kept on chip (one CTA of 8 warps, two per SM, one row at a time each:
// latency-bound) this re-reads the rows from L2 but keeps 8 CTAs per SM in flight and does no work for stages that
// decide nothing.
#pragma once

#include "spechub_lean.cuh"

namespace spechub {

struct LeanKaryShared : LeanCkShared {
    int x[kMaxK];                     // the drafts
    float lp[kMaxK], lq[kMaxK];       // their logits
    float u[kMaxK + 1];               // r_1..r_k, u_res
    float cx[kMaxK];                  // C after stage j + 1
};

// Is id y one of x[0..n)?
__device__ __forceinline__ bool one_of(const int *x, int n, int y) {
    bool f = false;
    for (int i = 0; i < n; ++i) f |= x[i] == y;
    return f;
}

// ---- draft step -----------------------------------------------------------------------------------
template <typename LT, bool SHIFT, int THREADS, RowPass PASS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) lean_kary_draft_kernel(KaryArgs A) {
    __shared__ LeanKaryShared sh;
    pdl_begin();
    const RowArgs &a = A.r;
    const int K = A.k;
    const long long r = blockIdx.x;
    const int b = static_cast<int>(r / a.nodes), n = static_cast<int>(r % a.nodes);
    const StreamRow<LT, SHIFT> vq(static_cast<const LT *>(a.draft) + b * a.stride_seq + n * a.stride_node, a.vocab);
    const Geo g = make_geo(a.vocab, 8);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int lo = g.seg_lo(warp), hi = g.seg_hi(warp);
    const float k = kLog2e / temperature_of(a, b);
    const float *un = a.uniforms + r * (2 * K + 1);
    const int CK = lean_ck_interval(g), CS = lean_ck_slots(g, CK);

    LeanAcc<LT> tq, unused;
    unused.init();
    lean_pass_a_ck<SHIFT, THREADS, PASS>(vq, lo, hi, lane, k, CK, tq, sh.cks + warp * CS, sh.ckc + warp * CS, CS, sh.any[warp]);
    ArgMaxSum Q, unusedq;
    lean_reduce2<false>(tq, unused, vq, vq, lo, hi, k, sh, Q, unusedq);
    const float Zq = Q.sx + Q.own(k);
    uint32_t st = 0;
    if (warp != 0) return;
    const bool bad = !(Q.ml > neg_inf()) || !finite_pos(Zq) || !(Q.ml < -neg_inf());
    if (bad) st = SPECHUB_ST_NONFINITE;
    for (int i = 0; i < K; ++i) {
        int t = -1;
        if (!bad) {
            const int out = A.without_replacement ? i : 0;   // x[0..out) are left out
            t = lean_ck_draw(g, vq, k, Q.c, CK, ListOut{sh.x, out}, un[i], sh);
            if (t < 0 && out == 0) t = Q.idx;   // (as in lean_draft_ck_kernel)
            if (t < 0) {   // nothing left to draw from: lowest id not drawn yet
                st |= SPECHUB_ST_DEGENERATE_Q;
                for (t = 0; t < a.vocab && one_of(sh.x, i, t); ++t) {}
                if (t >= a.vocab) t = 0;
            }
        }
        if (lane == 0) {
            sh.x[i] = t;
            a.draft_tokens_out[K * r + i] = t;
        }
        __syncwarp();
        if (!bad && A.without_replacement && i + 1 < K)
            lean_ck_drop(g, vq, k, Q.c, CK, ListOut{sh.x, i + 1}, t, sh);
    }
    if (lane == 0) {
        void_draft_stat(a, r);
        if (a.status) a.status[r] = st;
    }
}

// ---- verification ---------------------------------------------------------------------------------
template <typename LT, bool SHIFT, int THREADS>
__global__ void __launch_bounds__(THREADS, lean_ctas<SHIFT>(THREADS)) lean_kary_verify_kernel(KaryArgs A) {
    __shared__ LeanKaryShared sh;
    pdl_begin();
    using V = Vec8<LT>;
    const RowArgs &a = A.r;
    const int K = A.k;
    const bool wo = A.without_replacement != 0;
    const long long r = blockIdx.x;
    const int b = static_cast<int>(r / a.nodes), n = static_cast<int>(r % a.nodes);
    if (a.node_kind && a.node_kind[n] == SPECHUB_NODE_LEAF) return;   // leaf rows belong to lean_leaf_kernel
    const StreamRow<LT, SHIFT> vp(static_cast<const LT *>(a.target) + b * a.stride_seq + n * a.stride_node, a.vocab);
    const StreamRow<LT, SHIFT> vq(static_cast<const LT *>(a.draft) + b * a.stride_seq + n * a.stride_node, a.vocab);
    const Geo g = make_geo(a.vocab, 8);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int lo = g.seg_lo(warp), hi = g.seg_hi(warp);
    const float k = kLog2e / temperature_of(a, b);
    const float pinf = -neg_inf();

    if (threadIdx.x < kMaxK + 1) {
        const int i = threadIdx.x;
        const int y = i < K ? a.draft_tokens_in[K * r + i] : -1;
        const bool in = y >= 0 && y < a.vocab;
        if (i < kMaxK) {
            sh.x[i] = y;
            sh.lp[i] = in ? vp.one(y) : neg_inf();
            sh.lq[i] = in ? vq.one(y) : neg_inf();
        }
        if (i <= K) sh.u[i] = a.uniforms[r * (2 * K + 1) + K + i];
    }
    __syncthreads();
    bool in_range = true;
    unsigned singles = 0, mine = 0;   // bit i: x[i] is a single term; those in this thread's vectors
    for (int i = 0; i < K; ++i) {
        const int y = sh.x[i];
        const bool in = y >= 0 && y < a.vocab;
        in_range &= in;
        if (wo && in && i + 1 < K && !one_of(sh.x, i, y)) {
            singles |= 1u << i;
            const int v = y >> 3;
            if (v >= lo && v < hi && ((v - lo) & 31) == lane) mine |= 1u << i;
        }
    }
    auto drop_singles = [&](int vi, V &x, V &y) {
        for (unsigned m = mine; m; m &= m - 1) {
            const int id = sh.x[__ffs(m) - 1];
            if ((id >> 3) == vi) { x.drop(id & 7); y.drop(id & 7); }
        }
    };

    // pass A: maximum and sum of both rows without the single terms
    LeanAcc<LT> tp, tq;
    tp.init();
    tq.init();
    tp.c = lean_reference(vp, lo + lane, hi, k);
    tq.c = lean_reference(vq, lo + lane, hi, k);
    stream_pairs<1>(vp, vq, lo, hi, lane, [&](int vi, V x, V y) {
        if (mine) drop_singles(vi, x, y);
        lean_push(tp, x, k);
        lean_push(tq, y, k);
    });
    const int nwarps = THREADS / 32;
    {
        const float wp = lanes_max(tp.max()), wq = lanes_max(tq.max());
        if (lane == 0) { sh.wml[0][warp] = wp; sh.wml[1][warp] = wq; }
    }
    __syncthreads();
    float mp = lane < nwarps ? sh.wml[0][lane] : neg_inf(), mq = lane < nwarps ? sh.wml[1][lane] : neg_inf();
    if (lane < K && (singles >> lane & 1)) { mp = fmaxf(mp, sh.lp[lane]); mq = fmaxf(mq, sh.lq[lane]); }
    mp = lanes_max(mp);
    mq = lanes_max(mq);
    const float Cp = shift_of(mp, k), Cq = shift_of(mq, k);
    {
        const float wp = warp_sum(tp.max() > neg_inf() ? __fmul_rn(tp.s, ex2(tp.c - Cp)) : 0.f);
        const float wq = warp_sum(tq.max() > neg_inf() ? __fmul_rn(tq.s, ex2(tq.c - Cq)) : 0.f);
        if (lane == 0) { sh.wmass[0][warp] = wp; sh.wmass[1][warp] = wq; }
    }
    __syncthreads();
    float Zp = warp_sum(lane < nwarps ? sh.wmass[0][lane] : 0.f);
    const float q_rest = warp_sum(lane < nwarps ? sh.wmass[1][lane] : 0.f);   // outside the single terms
    float Zq = q_rest;
    auto ep = [&](int i) { return lean_exp(sh.lp[i], k, Cp); };   // of draft i
    auto eq = [&](int i) { return lean_exp(sh.lq[i], k, Cq); };
    for (unsigned m = singles; m; m &= m - 1) {
        const int i = __ffs(m) - 1;
        Zp = __fadd_rn(Zp, ep(i));
        Zq = __fadd_rn(Zq, eq(i));
    }

    int accept_idx = -1, token = -1;
    uint32_t status = 0;
    const bool t0 = threadIdx.x == 0;
    auto finish = [&]() {
        if (!t0) return;
        a.accept_idx[r] = accept_idx;
        a.token[r] = token;
        if (a.hub) a.hub[r] = -1;
        if (a.status) a.status[r] = status;
    };
    auto flagged = [&](uint32_t st) {
        status = st;
        for (int i = 0; i <= K && t0; ++i) {
            if (a.beta && i < K) a.beta[K * r + i] = 0.f;
            if (a.rate) a.rate[(K + 1) * r + i] = 0.f;
        }
        finish();
    };
    if (!(mp > neg_inf()) || !(mp < pinf) || !finite_pos(Zp) || !(mq > neg_inf()) || !(mq < pinf) || !finite_pos(Zq)) {
        flagged(SPECHUB_ST_NONFINITE);
        return;
    }
    if (!in_range) { flagged(SPECHUB_ST_TOKEN_RANGE); return; }
    const float invZp = 1.f / Zp, invZq = 1.f / Zq, rho = __fdiv_rn(Zp, Zq);
    const bool lite = !a.beta && !a.rate;
    const F2 k2 = f2_make(k, k), ncp2 = f2_make(-Cp, -Cp), ncq2 = f2_make(-Cq, -Cq);

    float m = 1.f, C = 0.f;   // m_{j-1}, C_{j-1}
    bool accepted = false;
    for (int j = 0; j < K; ++j) {
        float den = 1.f;   // mass of q outside the drafts before this stage: positive terms only
        if (wo && j > 0) {
            den = q_rest;
            for (unsigned s = singles >> j << j; s; s &= s - 1) den += eq(__ffs(s) - 1);
            den *= invZq;
        }
        const bool alive = m > 0.f;
        const float coef = m * (wo ? (den > 0.f ? 1.f / den : 0.f) : 1.f);
        const float px = ep(j) * invZp, qx = eq(j) * invZq;
        bool gone = false;
        float Cj = C;
        for (int l = 0; wo && l < j; ++l)
            if (sh.x[l] == sh.x[j] && !gone) { gone = true; Cj = sh.cx[l]; }
        const float N = fmaxf(__fmaf_rn(-Cj, qx, px), 0.f), D = gone ? 0.f : coef * qx;
        if (t0 && a.beta) a.beta[K * r + j] = alive && D > 0.f ? fminf(N / D, 1.f) : 0.f;
        if (alive && !accepted) {
            if (wo && j > 0 && !(den > 0.f)) status |= SPECHUB_ST_DEGENERATE_Q;
            if (!(D > 0.f)) status |= SPECHUB_ST_ZERO_MASS_DRAFT;
            else if (sh.u[j] * D < N) { accepted = true; accept_idx = j; token = sh.x[j]; }
        }
        if (accepted && lite) { finish(); return; }   // no probability asked for: later stages decide nothing
        C += coef;
        if (t0) sh.cx[j] = C;   // (read after the barrier below)
        const F2 nc = f2_make(-C * rho, -C * rho);
        F2 s = f2_make(0.f, 0.f);
        auto term = [&](int vi, V x, V y) {
            if (mine) drop_singles(vi, x, y);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                s = f2_add(s, f2_max0(f2_fma(nc, f2_exp(y.pair(i), k2, ncq2), f2_exp(x.pair(i), k2, ncp2))));
        };
        // (to and fro: what the last pass read last is read first)
        if (j & 1) stream_pairs<1>(vp, vq, lo, hi, lane, term);
        else stream_pairs<-1>(vp, vq, lo, hi, lane, term);
        const float ws = warp_sum(f2_sum(s));
        if (lane == 0) sh.acc[j][warp] = ws;
        __syncthreads();
        float m_next = warp_sum(lane < nwarps ? sh.acc[j][lane] : 0.f);
        for (unsigned sg = singles; sg; sg &= sg - 1) {
            const int i = __ffs(sg) - 1;   // (a draft that is still in q has the C of all ids)
            m_next += fmaxf(__fmaf_rn(-(i <= j ? sh.cx[i] : C) * rho, eq(i), ep(i)), 0.f);
        }
        m_next *= invZp;
        if (t0 && a.rate) a.rate[(K + 1) * r + j] = alive ? fmaxf(m - m_next, 0.f) : 0.f;
        m = m_next;
    }
    if (t0 && a.rate) a.rate[(K + 1) * r + K] = m;
    if (!accepted) {
        // residual: every warp picks the warp whose range holds the target, single terms counted where they lie
        const bool zero = !(m > 0.f);
        if (zero) status |= SPECHUB_ST_ZERO_RESIDUAL;   // a draw from p: C = 0 for every id
        float wm = lane < nwarps ? (zero ? (gives_id(sh.wml[0][lane], k, Cp) ? sh.wmass[0][lane] : 0.f) : sh.acc[K - 1][lane]) : 0.f;
        for (unsigned sg = singles; sg; sg &= sg - 1) {
            const int i = __ffs(sg) - 1;
            if (g.warp_of_vec(sh.x[i] >> 3) == lane) wm += zero ? ep(i) : fmaxf(__fmaf_rn(-sh.cx[i] * rho, eq(i), ep(i)), 0.f);
        }
        float t;
        const int w = pair_pick(wm, sh.u[K], t);
        if (w >= 0)
            token = range_sample3(g.seg_lo(w), g.seg_hi(w), [&](int vi, float(&out)[8]) {
                const V x = vp[vi], y = vq[vi];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    float Cy = zero ? 0.f : C;
                    if (!zero)
                        for (unsigned sg = singles; sg; sg &= sg - 1)
                            if (sh.x[__ffs(sg) - 1] == vi * 8 + i) Cy = sh.cx[__ffs(sg) - 1];
                    const float e = lean_exp(x.get(i), k, Cp);
                    out[i] = zero ? e : fmaxf(__fmaf_rn(-Cy * rho, lean_exp(y.get(i), k, Cq), e), 0.f);
                }
            }, sh, t);
    }
    finish();
}

}  // namespace spechub
