// Streaming kernels: bf16 or fp32 rows of any alignment, read as logical vectors of 8 ids (spechub_vec.cuh); two or
// three passes, the later ones from L2 as far as it holds the rows.
// One CTA per row; long bf16 rows in whole words can also be split over a cluster of 2 or 4 CTAs, which meet at two or
// three cluster barriers and read each other's partial results through distributed shared memory.  Several CTAs of
// different rows share an SM, so that one row's reductions overlap another row's streaming.
//
//   pass A  per 16-byte vector: a packed bf16 max tree (4 ops), 8 x (unpack, FMA,
//           ex2, add).  The exponent reference c of a thread is the maximum of the
//           first vector it reads, not a running maximum: 2^(k l - c) is exact in
//           floating point for any c within 2^+-100 of the true one, so c only
//           moves if a partial sum leaves that range (checked once per vector).
//   argmax  only threads whose maximum equals the row maximum rescan their own
//           elements (L2 hits) for the first index; the one owner also re-sums its
//           elements without the maximum, so 1 - q(a) is a direct sum.
//   pass B  re-reads the row (L2), recomputes the probabilities and the transport
//           sums; the hub's pair is removed in the one iteration that holds it.
//
// The special-function pipe (16 ex2/clk/SM) bounds both passes: 4 ex2 per
// vocabulary pair per row.
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "spechub.h"
#include "spechub_common.cuh"
#include "spechub_stream.cuh"
#include "spechub_ring.cuh"
#include "spechub_vec.cuh"

namespace spechub {
namespace cg = cooperative_groups;

constexpr int kLeanMaxWarps = 16;
constexpr int kLeanCk = 16;       // checkpoints per warp in the draft step's pass A, at most
constexpr float kNoIds = 6.2e-33f;  // 2^-107
constexpr float kHuge = 1.0e30f;  // ~2^100: partial sums beyond this move the reference

struct LeanShared {
    float wml[2][kLeanMaxWarps];     // per-warp max logit (0 target, 1 draft)
    float wmass[2][kLeanMaxWarps];   // per-warp sum of exponentials on the row's scale
    float wmassx[2][kLeanMaxWarps];  // the same without the lowest id in that warp that attains the row maximum
    int widx[2][kLeanMaxWarps];      // that id
    float acc[16][kLeanMaxWarps];
    int any[kLeanMaxWarps];
    float mass[kLeanMaxWarps];
    float part[kLeanMaxWarps];  // sampler: per-warp sums of the range drawn from
    int tok;
    // what this CTA tells the other CTAs of its row (read through distributed shared memory)
    float x_ml[2], x_sx[2];  // slice (max logit, sum without the slice argmax), 0 target / 1 draft
    int x_idx[2];            // slice argmax
    float x_sum[8];          // pass-B / pass-C sums of the slice
    float x_mass;            // slice mass for a draw from q without a given token
    int x_tok;               // a token drawn by this CTA
    // verification: what the tests need of single ids, fetched by one warp before its pass A
    int tk[2];               // the drafts
    float lg[8];             // target logits of the drafts, draft logits of the drafts, -, r1, r2, u_res
    int stat_ok;             // from draft statistics: the row's record was accepted
};
// draft step and leaf rows: also the checkpoint sums of pass A (per warp, every CK lane-iterations) and their
// exponent references
struct LeanCkShared : LeanShared {
    float cks[kLeanMaxWarps * kLeanCk], ckc[kLeanMaxWarps * kLeanCk];
};

__device__ __forceinline__ float lanes_max(float x) {
    float m;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(x));
    return m;
}
__device__ __forceinline__ float lanes_prefix(float x) {   // inclusive, over ascending lanes
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float up = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += up;
    }
    return x;
}
// Inverse-CDF pick over one mass per lane: the lowest lane with mass whose inclusive prefix exceeds t, the last lane
// with mass if none does; -1: no mass.  t becomes the target within the lane.  The same in every lane.
__device__ __forceinline__ int lanes_pick(float m, float &t) {
    const float incl = lanes_prefix(m);
    const unsigned pos = __ballot_sync(kFull, m > 0.f), hit = __ballot_sync(kFull, m > 0.f && incl > t);
    if (!pos) return -1;
    const int L = hit ? __ffs(hit) - 1 : 31 - __clz(pos);
    t = __shfl_sync(kFull, t - (incl - m), L);
    return L;
}

// The CTAs of one row.  CS = 1 compiles to no cluster instruction at all.
template <int CS>
struct RowGroup {
    __device__ __forceinline__ static int rank() {
        if (CS == 1) return 0;
        return static_cast<int>(cg::this_cluster().block_rank());
    }
    __device__ __forceinline__ static void sync() {
        if (CS == 1) __syncthreads();
        else cg::this_cluster().sync();
    }
    template <class T>
    __device__ __forceinline__ static const T *peer(const T *local, int r) {
        if (CS == 1) return local;
        return cg::this_cluster().map_shared_rank(local, r);
    }
};

// CTAs of THREADS threads per SM.  64 registers per thread (1024 threads per SM) measured best on rows in whole words
// and for the draft step; verification of shifted rows holds two or three words per vector and row: 80 registers
// (V = 50257, 896 rows, fp32: 87 -> 78 us, RRSw in bf16 69 -> 63 us; the draft step there 23.5 us with 80, 22 us with 64).
template <bool SHIFT>
constexpr int lean_ctas(int threads) { return (SHIFT ? 768 : 1024) / threads; }

template <typename LT>
struct LeanAcc {  // one thread's pass-A state for one row
    typename Vec8<LT>::Max m2;  // running maximum (packed)
    float c;                    // exponent reference (k * some logit of this thread, or 0)
    float s;                    // sum of 2^(k l - c)
    __device__ __forceinline__ void init() { m2 = Vec8<LT>::max_none(); s = 0.f; c = 0.f; }
    __device__ __forceinline__ float max() const { return Vec8<LT>::max_value(m2); }
};

// a vector's sum of exponentials, two lanes at a time: (e0 + e2) + (e4 + e6) and (e1 + e3) + (e5 + e7)
template <typename LT>
__device__ __forceinline__ float vec_sum(const Vec8<LT> &v, F2 k2, F2 nc2) {
    return f2_sum(f2_add(f2_add(f2_exp(v.pair(0), k2, nc2), f2_exp(v.pair(1), k2, nc2)),
                         f2_add(f2_exp(v.pair(2), k2, nc2), f2_exp(v.pair(3), k2, nc2))));
}

template <typename LT>
__device__ __forceinline__ void lean_push(LeanAcc<LT> &st, const Vec8<LT> &v, float k) {
    const auto vm = v.packed_max();
    st.m2 = Vec8<LT>::max_of(st.m2, vm);
    const F2 k2 = f2_make(k, k);
    float a = vec_sum(v, k2, f2_make(-st.c, -st.c));
    if (!(a < kHuge)) {  // out of range (or NaN / +inf input): move the reference to this vector's max
        const float cn = shift_of(Vec8<LT>::max_value(vm), k);
        st.s *= ex2(st.c - cn);
        st.c = cn;
        a = vec_sum(v, k2, f2_make(-st.c, -st.c));
    }
    st.s += a;
}

// ... of a batch of vectors: the same sums in the same order, with one look at their size.  (Where that fails the vectors,
// vi, vi + 32, ..., are read again: kept for it, they would not fit the registers.)
template <typename LT>
struct LeanBatch {
    LeanAcc<LT> &st;
    F2 k2, nc2;
    float s;
    typename Vec8<LT>::Max m2;
    __device__ __forceinline__ LeanBatch(LeanAcc<LT> &a) : st(a) {}
    __device__ __forceinline__ void begin(float k) { k2 = f2_make(k, k); again(); }
    __device__ __forceinline__ void again() { nc2 = f2_make(-st.c, -st.c); s = st.s; m2 = st.m2; }
    __device__ __forceinline__ void push(const Vec8<LT> &v) {
        m2 = Vec8<LT>::max_of(m2, v.packed_max());
        s += vec_sum(v, k2, nc2);
    }
    template <int D, class IN>
    __device__ __forceinline__ void commit(const IN &in, float k, int vi, int hi) {
        if (s < kHuge) {
            st.m2 = m2;
            st.s = s;
        } else {
#pragma unroll 1
            for (int d = 0; d < D; ++d) lean_push(st, in.fix(in.checked(vi + 32 * d, hi)), k);
            again();
        }
    }
};

// the exponent reference of a thread: the maximum of its first vector that holds a finite logit
template <class ROW>
__device__ __forceinline__ float lean_reference(const ROW &row, int vi, int hi, float k) {
    for (; vi < hi; vi += 32) {
        const float m0 = row[vi].max();
        if (m0 > neg_inf()) return shift_of(m0, k);
    }
    return 0.f;
}

// ... whose first vector is at hand
template <typename LT, class ROW>
__device__ __forceinline__ float lean_reference(const Vec8<LT> &first, const ROW &row, int v0, int hi, float k) {
    const float m0 = first.max();
    return m0 > neg_inf() ? shift_of(m0, k) : lean_reference(row, v0 + 32, hi, k);
}

// This warp's range of two rows: f(vector index, target vector, draft vector), as in pair_turns
template <int STEP, typename LT, bool SHIFT, class F>
__device__ __forceinline__ void stream_pairs(const StreamRow<LT, SHIFT> &p, const StreamRow<LT, SHIFT> &q, int lo, int hi, int lane, F f) {
    if constexpr (SHIFT) {
        any_pairs<STEP>(p, q, lo, hi, lane, f);
    } else {
        const int n = (hi - lo - lane + 31) >> 5;   // this lane's vectors
        pair_turns<STEP>(WholeIn<LT>{p}, WholeIn<LT>{q}, lo + lane, STEP > 0 ? 0 : n - 1, n, f);
    }
}
// ... for the last time: L2 may let these lines go first
template <int STEP, typename LT, bool SHIFT, class F>
__device__ __forceinline__ void stream_pairs_last(const StreamRow<LT, SHIFT> &p, const StreamRow<LT, SHIFT> &q, int lo, int hi, int lane, F f) {
    if constexpr (SHIFT) {
        any_pairs<STEP>(p, q, lo, hi, lane, f);
    } else {
        uint64_t pol;
        asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
        const int n = (hi - lo - lane + 31) >> 5;
        pair_turns<STEP>(HintedIn<LT>{p, pol}, HintedIn<LT>{q, pol}, lo + lane, STEP > 0 ? 0 : n - 1, n, f);
    }
}

// Pass A over this warp's range of two rows.
// AHEAD: the next vector pair is requested before the current one is consumed (measured per
// method: it pays for RRS, 1.92 -> 1.82 ms on V = 128256, and RRSw, 468 -> 455 us on 7936 rows of 32000 ids; SpecHub
// gains 3 % on those and on few rows, and loses 5 % on 7936 rows of 128256: there it is for CTAs of 512 threads, few rows).
template <bool AHEAD, typename LT, bool SHIFT>
__device__ __forceinline__ void lean_pass_a2(const StreamRow<LT, SHIFT> &rp, const StreamRow<LT, SHIFT> &rq, int lo, int hi, int lane, float k,
                                             LeanAcc<LT> &P, LeanAcc<LT> &Q) {
    P.init();
    Q.init();
    int vi = lo + lane;
    P.c = lean_reference(rp, vi, hi, k);
    Q.c = lean_reference(rq, vi, hi, k);
    auto push = [&](int, const Vec8<LT> &a, const Vec8<LT> &b) {
        lean_push(P, a, k);
        lean_push(Q, b, k);
    };
    if constexpr (AHEAD || SHIFT) {
        stream_pairs<1>(rp, rq, lo, hi, lane, push);
    } else {
#pragma unroll 2
        for (; vi < hi; vi += 32) push(vi, rp[vi], rq[vi]);
    }
}

// Pass A over one row.  KEEP: the row is read again by pass B, and L2 is asked to keep it.  TURNS: through one set of
// registers (row_turns): in the three-method kernel two sets cost the later passes spills (7936 rows of 32000 ids 518 -> 511
// us, 3968 of 128256 907 -> 896), in RRSw's the copies cost more than those (7936 of 32000 402 -> 424).
template <bool KEEP, bool TURNS, typename LT>
__device__ __forceinline__ void lean_pass_a1(const StreamRow<LT, false> &rp, int lo, int hi, int lane, float k, LeanAcc<LT> &P) {
    P.init();
    LeanBatch<LT> B(P);
    auto run = [&](const auto &in) {
        constexpr int D = std::decay_t<decltype(in)>::kDepth;
        auto begin = [&](const Vec8<LT> &first) { P.c = lean_reference(first, rp, lo + lane, hi, k); B.begin(k); };
        auto one = [&](const Vec8<LT> &v) { B.push(v); };
        auto batch = [&](int vi) { B.template commit<D>(in, k, vi, hi); };
        if constexpr (TURNS) row_turns<D>(in, lo + lane, hi, whole_iters(lo, hi), begin, one, batch);
        else row_batches<D, true>(in, lo + lane, hi, whole_iters(lo, hi), begin, one, batch);
    };
    if constexpr (KEEP) {
        uint64_t pol;
        asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
        run(HintedIn<LT>{rp, pol});
    } else {
        run(WholeIn<LT>{rp});
    }
}

// ... of a row of any alignment (neither applies)
template <bool KEEP, bool TURNS, typename LT>
__device__ __forceinline__ void lean_pass_a1(const StreamRow<LT, true> &rp, int lo, int hi, int lane, float k, LeanAcc<LT> &P) {
    P.init();
    LeanBatch<LT> B(P);
    const Iters t = inside_iters(rp.src, rp.src, lo, hi);
    auto run = [&](const auto &in) {
        constexpr int D = std::decay_t<decltype(in)>::kDepth;
        row_batches<D, false>(in, lo + lane, hi, t,
                              [&](const Vec8<LT> &first) { P.c = lean_reference(first, rp, lo + lane, hi, k); B.begin(k); },
                              [&](const Vec8<LT> &v) { B.push(v); }, [&](int vi) { B.template commit<D>(in, k, vi, hi); });
    };
    if (rp.src.sh == 0) run(AlignedIn<LT>{rp.src});
    else run(ShiftedIn<LT>{rp.src});
}

// Pass A over both rows with the vectors coming from the warp's ring (the first pass of its stream, forwards).
template <class ROW>
__device__ __forceinline__ void lean_pass_a_ring(WarpRing &R, const ROW &vp, const ROW &vq, int lane, float k,
                                                 LeanAcc<__nv_bfloat16> &P, LeanAcc<__nv_bfloat16> &Q) {
    P.init();
    Q.init();
    const int vi0 = R.lo + lane;
    if (R.nc > 0) {
        // the reference comes from the thread's first vector that holds a finite logit: nearly always the
        // very first one, which the first chunk holds; otherwise look further in global memory
        ring_wait(R);
        if (vi0 < R.hi) {
            Vec8<__nv_bfloat16> a, b;
            ring_load(R, 0, lane, a, b);
            const float ma = a.max(), mb = b.max();
            P.c = ma > neg_inf() ? shift_of(ma, k) : lean_reference(vp, vi0 + 32, R.hi, k);
            Q.c = mb > neg_inf() ? shift_of(mb, k) : lean_reference(vq, vi0 + 32, R.hi, k);
        }
    }
#pragma unroll 1
    for (int c = 0; c < R.nc; ++c) {
        ring_wait(R);
        const int v0 = vi0 + c * kRingChunkVecs;
#pragma unroll
        for (int j = 0; j < kRingCh; ++j) {
            Vec8<__nv_bfloat16> x, y;
            ring_load(R, j, lane, x, y);
            if (j == kRingCh - 1) ring_release(R, lane);
            if (v0 + j * 32 < R.hi) {
                lean_push(P, x, k);
                lean_push(Q, y, k);
            }
        }
    }
}

// The lanes of a warp rescan, together, the elements of its lane `src` (whose maximum equals the
// row maximum `val`): lane j takes the j-th vector of that thread, so the rescan costs one load
// round trip instead of one per vector.  Returns (to every lane) the first index of val among
// those elements and the sum of 2^(k l - c) over them without that index.
template <class ROW>
__device__ __forceinline__ void lean_rescan_warp(const ROW &row, int lo, int hi, int lane, int src,
                                                 float val, float k, float c, int &first_idx,
                                                 float &s_excl) {
    int fi = 0x7fffffff;
    const int v0 = lo + src + 32 * lane;
    // the first round's vector stays in registers for the sum (ranges of up to 1024 vectors: all of them)
    auto first = Vec8<typename ROW::Elem>::none();
    if (v0 < hi) first = row[v0];
    auto find = [&](const auto &v, int vj) {
#pragma unroll
        for (int i = 7; i >= 0; --i)
            if (v.get(i) == val) fi = min(fi, vj * 8 + i);
    };
    if (v0 < hi) find(first, v0);
#pragma unroll 1
    for (int vj = v0 + 32 * 32; vj < hi; vj += 32 * 32) find(row[vj], vj);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) fi = min(fi, __shfl_xor_sync(kFull, fi, o));
    // the sum without it
    float s = 0.f;
    auto add = [&](const auto &v, int vj) {
        float e[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) e[i] = (vj * 8 + i == fi) ? 0.f : ex2(__fmaf_rn(v.get(i), k, -c));
        s += ((e[0] + e[1]) + (e[2] + e[3])) + ((e[4] + e[5]) + (e[6] + e[7]));
    };
    if (v0 < hi) add(first, v0);
#pragma unroll 1
    for (int vj = v0 + 32 * 32; vj < hi; vj += 32 * 32) add(row[vj], vj);
    s_excl = warp_sum(s);
    first_idx = fi;
}

// Row-level (max, argmax, sum without the argmax) of the target (r = 0) and, if BOTH, the draft
// (r = 1) from the per-thread pass-A states.  Leaves the per-warp masses in sh.wmass[r] / wmassx[r] for the
// samplers.  All threads call it; two barriers, and every warp merges the warps' values by itself.
template <int R, typename LT, class ROW>
__device__ __forceinline__ void lean_publish(const LeanAcc<LT> &t, const ROW &row, int lo, int hi, float k, float rm,
                                             LeanShared &sh) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float ml = t.max();
    int best = 0x7fffffff, best_lane = -1;
    float best_sx = 0.f;
    unsigned cm = __ballot_sync(kFull, ml == rm && rm > neg_inf() && rm < -neg_inf());
    while (cm) {   // (one lane of the CTA, or a few on ties)
        const int src = __ffs(cm) - 1;
        cm &= cm - 1;
        int fi; float sx;
        lean_rescan_warp(row, lo, hi, lane, src, rm, k, __shfl_sync(kFull, t.c, src), fi, sx);
        if (fi < best) { best = fi; best_lane = src; best_sx = sx; }
    }
    const float f = ml > neg_inf() ? ex2(t.c - shift_of(rm, k)) : 0.f;
    const float all = warp_sum(__fmul_rn(t.s, f));
    const float without = best_lane < 0 ? all : warp_sum(__fmul_rn(lane == best_lane ? best_sx : t.s, f));
    if (lane == 0) { sh.wmass[R][warp] = all; sh.wmassx[R][warp] = without; sh.widx[R][warp] = best; }
}
template <int R>
__device__ __forceinline__ void lean_merge_warps(const LeanShared &sh, float rm, float k, ArgMaxSum &o) {
    const int lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    const int mine = lane < nwarps ? sh.widx[R][lane] : 0x7fffffff;
    o.ml = rm;
    o.c = shift_of(rm, k);
    o.idx = __reduce_min_sync(kFull, mine);
    const float m = lane < nwarps ? (mine == o.idx ? sh.wmassx[R][lane] : sh.wmass[R][lane]) : 0.f;
    o.sx = warp_sum(m);
}
template <bool BOTH, typename LT, class ROW>
__device__ void lean_reduce2(const LeanAcc<LT> &tp, const LeanAcc<LT> &tq, const ROW &vp, const ROW &vq, int lo,
                             int hi, float k, LeanShared &sh, ArgMaxSum &P, ArgMaxSum &Q) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    const float wp = lanes_max(tp.max()), wq = BOTH ? lanes_max(tq.max()) : neg_inf();
    if (lane == 0) { sh.wml[0][warp] = wp; if (BOTH) sh.wml[1][warp] = wq; }
    __syncthreads();
    const float rmp = lanes_max(lane < nwarps ? sh.wml[0][lane] : neg_inf());
    const float rmq = BOTH ? lanes_max(lane < nwarps ? sh.wml[1][lane] : neg_inf()) : neg_inf();
    lean_publish<0>(tp, vp, lo, hi, k, rmp, sh);
    if (BOTH) lean_publish<1>(tq, vq, lo, hi, k, rmq, sh);
    __syncthreads();
    lean_merge_warps<0>(sh, rmp, k, P);
    if (BOTH) lean_merge_warps<1>(sh, rmq, k, Q);
    else { Q.ml = neg_inf(); Q.c = 0.f; Q.idx = 0x7fffffff; Q.sx = 0.f; }
}

// CTA-wide inverse-CDF draw over the vectors [lo, hi): weights(vi, w[8]) the weights of vector vi, tt = target prefix
// within the range.  One block of consecutive vectors per thread is summed, every warp picks the warp that holds the
// target from the warps' sums, and that warp spreads the picked thread's vectors over its lanes: two load round
// trips, two barriers.  Called by all threads of the CTA; returns to every thread the lowest id whose inclusive prefix
// exceeds tt; when rounding leaves none, the last id with positive weight of the picked block; -1: no mass.
template <class WF>
__device__ int range_sample3(int lo, int hi, WF weights, LeanShared &sh, float tt) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nth = blockDim.x;
    const int Bv = (hi - lo + nth - 1) / nth;  // vectors per thread
    float tot = 0.f;
    {
        const int b0 = lo + threadIdx.x * Bv, b1 = min(hi, b0 + Bv);
#pragma unroll 4
        for (int vi = b0; vi < b1; ++vi) {
            float w[8];
            weights(vi, w);
            tot += ((w[0] + w[1]) + (w[2] + w[3])) + ((w[4] + w[5]) + (w[6] + w[7]));
        }
    }
    const float wt = warp_sum(tot);
    if (lane == 0) sh.part[warp] = wt;
    __syncthreads();
    const int W = lanes_pick(lane < (nth >> 5) ? sh.part[lane] : 0.f, tt);
    if (W < 0) { __syncthreads(); return -1; }
    if (warp == W) {
        const int L = lanes_pick(tot, tt);
        int found = -1;
        const int c0 = lo + (W * 32 + max(L, 0)) * Bv, c1 = min(hi, c0 + Bv);
        float prefix = 0.f;
        int lastpos = -1;
        for (int v0 = c0; v0 < c1 && found < 0; v0 += 32) {
            const int vi = v0 + lane;
            float w[8];
            if (vi < c1) {
                weights(vi, w);
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) w[i] = 0.f;
            }
            float lsum = 0.f;
            int lp = -1;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                lsum += w[i];
                if (w[i] > 0.f) lp = vi * 8 + i;
            }
            const float in2 = lanes_prefix(lsum);
            const unsigned hit2 = __ballot_sync(kFull, lsum > 0.f && prefix + in2 > tt);
            if (hit2) {
                float acc = prefix + (in2 - lsum);
                int cand = -1, lastin = -1;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    acc += w[i];
                    if (w[i] > 0.f) {
                        lastin = vi * 8 + i;
                        if (cand < 0 && acc > tt) cand = lastin;
                    }
                }
                found = __shfl_sync(kFull, cand < 0 ? lastin : cand, __ffs(hit2) - 1);
            } else {
                lastpos = max(lastpos, __reduce_max_sync(kFull, lp));
                prefix += __shfl_sync(kFull, in2, 31);
            }
        }
        if (found < 0) found = lastpos;
        if (lane == 0) sh.tok = found;
    }
    __syncthreads();
    return sh.tok;   // (written again only after the first barrier of a later draw)
}

// (a call instead of inlined code: where a kernel draws several times, that takes registers from its passes)
struct LanePick { int lane; float t; };
static __device__ __noinline__ LanePick pair_pick_call(float m, float u) {
    LanePick o;
    o.lane = pair_pick(m, u, o.t);
    return o;
}
// ... over this CTA's part of a row: mass[w] = total weight of warp w's range (the coarse CDF).  WHOLE: the part is the
// row and u the uniform; else u is the target prefix within the part.  CALL: pick by pair_pick_call.
template <bool WHOLE, bool CALL = false, class WF>
__device__ int block_sample3(const Geo &g, WF weights, const float *mass, LeanShared &sh, float u) {
    const int lane = threadIdx.x & 31;
    const float m = lane < g.nwarps ? mass[lane] : 0.f;
    float t = u;
    int w;
    if (WHOLE && CALL) {
        const LanePick x = pair_pick_call(m, u);
        w = x.lane;
        t = x.t;
    } else {
        w = WHOLE ? pair_pick(m, u, t) : lanes_pick(m, t);
    }
    if (w < 0) return -1;
    return range_sample3(g.seg_lo(w), g.seg_hi(w), weights, sh, t);
}

// Pick the CTA of a row whose part holds the target t of an inverse-CDF draw over per-CTA masses
// m[0..n) (ascending token ranges).  Returns the rank (-1 if no mass) and the mass before it.
__device__ __forceinline__ int pick_part(const float *m, int n, double t, double &base) {
    int sel = -1, last = -1;
    double lastbase = 0., run = 0.;
    base = 0.;
    for (int r = 0; r < n; ++r) {
        if (m[r] > 0.f) {
            last = r;
            lastbase = run;
            if (sel < 0 && run + m[r] > t) { sel = r; base = run; }
        }
        run += m[r];
    }
    if (sel < 0) { sel = last; base = lastbase; }
    return sel;
}

// What every CTA of a row knows about one of its rows after the slices were merged.
struct RowStat {
    float ml, C, sx;  // row max logit, its shift, sum without the row argmax
    float own;        // the row argmax's own term 2^(k ml - C) (1 up to the rounding of C)
    int idx;          // row argmax
    __device__ __forceinline__ void set(const ArgMaxSum &o, float k) { ml = o.ml; C = o.c; sx = o.sx; idx = o.idx; own = o.own(k); }
};

// Merge the slices' (max, argmax, sum without argmax) in rank order (Section 4: a = argmax q).
template <int CS>
__device__ __forceinline__ void merge_slices(const LeanShared &sh, int r, float k, RowStat &st) {
    ArgMaxSum tot;
    tot.init();
#pragma unroll
    for (int c = 0; c < CS; ++c) {
        const LeanShared *ps = RowGroup<CS>::peer(&sh, c);
        ArgMaxSum o;
        o.ml = ps->x_ml[r]; o.c = shift_of(o.ml, k); o.sx = ps->x_sx[r]; o.idx = ps->x_idx[r];
        tot = argmaxsum_merge(tot, o, k);
    }
    st.ml = tot.ml; st.C = tot.c; st.sx = tot.sx; st.idx = tot.idx; st.own = tot.own(k);
}

// Does a part of a row with the maximum logit ml have an exponential above 0 on the row's scale?  (Its sum, made on its
// own scale, may be above 0 there although all of its exponentials are below the smallest normal number.)
__device__ __forceinline__ bool gives_id(float ml, float k, float C) { return ml > neg_inf() && ex2(__fmaf_rn(ml, k, -C)) > 0.f; }

// Mass of slice c of a row (row scale) for a draw from softmax(row) without token `excl`
// (excl < 0: none; only a slice's own argmax can be left out here).  The slices' published
// partials stay valid until the kernel ends.
template <int CS>
__device__ __forceinline__ float slice_mass(const LeanShared &sh, int r, const RowStat &st, int c, int excl,
                                            float k) {
    const LeanShared *ps = RowGroup<CS>::peer(&sh, c);
    const float ml = ps->x_ml[r];
    if (!gives_id(ml, k, st.C)) return 0.f;
    const float own = (ps->x_idx[r] != excl) ? own_term(ml, k) : 0.f;
    return (ps->x_sx[r] + own) * rescale(ml, shift_of(ml, k), st.C);
}

// Draw inside this CTA's slice from softmax(row) without token `excl`.  u: target (row scale, relative to the start of
// the slice); CS = 1: the uniform.  sh.wmass[r] holds the per-warp sums of the slice on the
// slice's own scale.
template <int CS, class ROW>
__device__ int lean_sample_slice(const Geo &g, const ROW &row, float k, const RowStat &st,
                                 int excl, float u, int r, LeanShared &sh) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int locarg = sh.x_idx[r];
    const float lml = sh.x_ml[r];
    const float f = rescale(lml, shift_of(lml, k), st.C);
    const float C = st.C;
    if (threadIdx.x < g.nwarps) {
        const int w = threadIdx.x;
        const float m = (excl >= 0 && excl == locarg && sh.widx[r][w] == locarg ? sh.wmassx[r][w] : sh.wmass[r][w]) * f;
        sh.mass[w] = gives_id(sh.wml[r][w], k, C) ? m : 0.f;
    }
    __syncthreads();
    if (excl >= 0 && excl != locarg && g.holds_vec(excl >> 3)) {
        // an arbitrary token of this slice is removed: its warp re-sums its range
        const int wex = g.warp_of_vec(excl >> 3);
        if (warp == wex) {
            float s = 0.f;
            for (int vi = g.seg_lo(warp) + lane; vi < g.seg_hi(warp); vi += 32) {
                const auto v = row[vi];
#pragma unroll
                for (int i = 0; i < 8; ++i) s += (vi * 8 + i == excl) ? 0.f : ex2(__fmaf_rn(v.get(i), k, -C));
            }
            s = warp_sum(s);
            if (lane == 0) sh.mass[warp] = s;
        }
        __syncthreads();
    }
    auto wf = [&](int vi, float(&w)[8]) {
        const auto v = row[vi];
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = (vi * 8 + i == excl) ? 0.f : ex2(__fmaf_rn(v.get(i), k, -C));
    };
    return block_sample3<CS == 1>(g, wf, sh.mass, sh, u);
}

// Draw from softmax(row) without `excl` (the row argmax, a slice argmax, or nothing) over the
// whole row: every CTA of the row calls it; the CTA whose slice holds the target draws and
// returns the token, the others return -2.  -1: no mass.
template <int CS, class ROW>
__device__ int lean_sample_row(const Geo &g, const ROW &row, float k, const RowStat &st, int me,
                               int excl, float u, int r, LeanShared &sh) {
    float m[CS];
    double total = 0.;
#pragma unroll
    for (int c = 0; c < CS; ++c) { m[c] = slice_mass<CS>(sh, r, st, c, excl, k); total += m[c]; }
    if (!(total > 0.)) return -1;
    if (CS == 1) return lean_sample_slice<1>(g, row, k, st, excl, u, r, sh);
    double base;
    const int sel = pick_part(m, CS, u * total, base);
    if (sel != me) return -2;
    return lean_sample_slice<CS>(g, row, k, st, excl, static_cast<float>(u * total - base), r, sh);
}

// CTA sums of NACC per-thread accumulators; the per-warp sums stay in sh.acc[OFF + i][w].  ANY: also whether `any` is
// set in some thread.  One barrier; a second call in the same kernel takes other rows of sh.acc.
template <int NACC, int OFF, bool ANY = false>
__device__ __forceinline__ void lean_block_sums(float (&x)[NACC], LeanShared &sh, unsigned *any = nullptr) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
#pragma unroll
    for (int i = 0; i < NACC; ++i) {
        const float s = warp_sum(x[i]);
        if (lane == 0) sh.acc[OFF + i][warp] = s;
    }
    if (ANY) {
        const int a = __any_sync(kFull, *any != 0);
        if (lane == 0) sh.any[warp] = a;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NACC; ++i) x[i] = warp_sum(lane < nwarps ? sh.acc[OFF + i][lane] : 0.f);
    if (ANY) *any = __any_sync(kFull, lane < nwarps && sh.any[lane]);
}

// Sum NACC per-thread accumulators over the whole row: CTA sums, then the slices in rank order.
// part[i][c] receives slice c's sum of accumulator i; sh.acc[OFF + i][w] keeps this CTA's per-warp sums.
// Contains one row-group barrier.  OFF: first exchange slot used (a second call in the same
// kernel takes other slots, so no CTA overwrites what a slower one has not read yet).
template <int CS, int NACC, int OFF, bool ANY = false>
__device__ __forceinline__ void lean_row_sums(float (&x)[NACC], float (&part)[NACC][CS], LeanShared &sh,
                                              unsigned *any = nullptr) {
    lean_block_sums<NACC, OFF, ANY>(x, sh, any);
    if (CS == 1) {
#pragma unroll
        for (int i = 0; i < NACC; ++i) part[i][0] = x[i];
        return;
    }
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 0; i < NACC; ++i) sh.x_sum[OFF + i] = x[i];
    }
    RowGroup<CS>::sync();
#pragma unroll
    for (int i = 0; i < NACC; ++i) {
        float t = 0.f;
#pragma unroll
        for (int c = 0; c < CS; ++c) {
            part[i][c] = RowGroup<CS>::peer(&sh, c)->x_sum[OFF + i];
            t += part[i][c];
        }
        x[i] = t;
    }
}

// ------------------------------------------------------------------------------------------------
// Draft step, one CTA per row, with a finer coarse CDF.  Pass A records, every CK lane-iterations,
// the warp's sum since its previous checkpoint: sub-blocks of 32 * CK consecutive vectors, at most
// kLeanCk per warp.  A draw then picks a sub-block from those sums and rescans only that (a few KB
// instead of a warp's whole range), which is what the two-pass sampler costs most.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ int lean_ck_interval(const Geo &g) {
    const int iters = (g.seg + 31) >> 5;
    return 4 * max(1, (iters + 4 * kLeanCk - 1) / (4 * kLeanCk));   // a multiple of the unroll of pass A
}
__device__ __forceinline__ int lean_ck_slots(const Geo &g, int CK) {   // sub-blocks per warp
    return (((g.seg + 31) >> 5) + CK - 1) / CK;
}

// How the draft step's and the leaf rows' passes take their rows (us of the draft step unless it says otherwise).
//   kTurns    from registers, one set (row_turns): rows in whole words, and bf16 shifted rows of more than one wave of these
//             CTAs (many_rows; 3840 of 64001 ids 147, by two sets 159; 4900 of 8201 52.2, 56.8), whose sums are looked at
//             after every vector then: a batch's own sum and maximum are registers that these kernels would spill (7680 of
//             50257 ids 203, by batches 214; 3968 of 128257 236, 251)
//   kBatches  from registers, two sets that take turns (row_batches): other shifted rows, longer to make into vectors (448
//             bf16 rows of 16393 ids 14.0, by one set 14.3, 224 of 64001 17.7, 18.5; 1400 fp32 rows of 64001 91.5, 104)
//   kRing     from rings of bulk copies (spechub_ring.cuh): the draft step of two drafts on bf16 rows in whole words of 40960 ids
//             and more, in more than one wave of CTAs of 128 threads (7936 of 128256 ids 322, by one set 333; 3584 of 48000
//             70.4, 72.7).  In less than a wave an SM's rings hold too few bytes in flight, and no row is behind others that
//             hide its end (651 of 101056 57.7, 45.6; 896 of 64000 37.1, 33.3).  Shorter rows gain 1 to 3 % by themselves, but
//             verification behind them starts later (RRSw step on 3840 rows of 32000 with leaves 165, without rings 158:
//             kernels of other needs of shared memory do not meet on an SM).  More drafts wait for their draws longer than
//             for the bytes (three drafts, 3250 rows of 32000: 75.2, 70.1), as do leaf rows behind a draft step
//             (verification, 7680 rows of 32000, half of them leaves: 212, 206).  Not fp32 rows (480 of 128256, a step
//             173, 170: a vector is 32 bytes, its reads from shared memory meet in the banks).
enum RowPass { kTurns, kBatches, kRing };
template <typename LT, bool SHIFT> constexpr RowPass kFewRows = SHIFT ? kBatches : kTurns;
template <typename LT, bool SHIFT> constexpr RowPass kManyRows = SHIFT && sizeof(LT) == 2 ? kTurns : kFewRows<LT, SHIFT>;
template <typename LT, bool SHIFT> constexpr RowPass kManyDrafts = !SHIFT && sizeof(LT) == 2 ? kRing : kManyRows<LT, SHIFT>;
constexpr int kRowRingVocab = 40960;   // (draft_threads: 128 threads in more than a wave of rows)
template <int THREADS, RowPass PASS> constexpr int kRowRingBytes = PASS == kRing ? THREADS / 32 * kRowWarpBytes : 0;

// late (kRing): whether a bulk copy did not arrive within its bounded wait (the results are of the part in front of it).
template <bool SHIFT, int THREADS, RowPass PASS, typename LT, class ROW>
__device__ __forceinline__ void lean_pass_a_ck(const ROW &rq, int lo, int hi, int lane, float k, int CK,
                                               LeanAcc<LT> &Q, float *cks, float *ckc, int slots, int &late) {
    LeanAcc<LT> st;
    st.init();
    float cref = 0.f;               // the reference every lane is expected to hold
    float tot = 0.f, ctot = 0.f;    // this thread's sum over all checkpoints, on the scale ctot
    int j = 0;
    // One exponent reference for the whole warp: the maximum of its first 32 vectors that hold a finite logit (nearly
    // always the very first ones; a warp whose range begins with masked ids looks further).  Behind the pass's first
    // loads (a step on 448 rows of 32000 ids: 44.9 us, 46.0 where they wait for the search).
    auto reference = [&](const Vec8<LT> &first) {
        float m0 = lanes_max(first.max());
#pragma unroll 1
        for (int vb = lo + 32; !(m0 > neg_inf()) && vb < hi; vb += 32)
            m0 = lanes_max(vb + lane < hi ? rq[vb + lane].max() : neg_inf());
        st.c = cref = ctot = shift_of(m0, k);
    };
    // checkpoint: the warp's sum since the last one.  A lane that had to move its reference (sums
    // beyond 2^100, rare) is brought to the warp's largest reference first.
    auto checkpoint = [&]() {
        float contrib = st.s, cnow = cref;
        if (__any_sync(kFull, st.c != cref)) {
            float cm = st.c;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) cm = fmaxf(cm, __shfl_xor_sync(kFull, cm, o));
            contrib = st.s > 0.f ? st.s * ex2(st.c - cm) : 0.f;
            cnow = cm;
        }
        const float cs = warp_sum(contrib);
        if (lane == 0) { cks[j] = cs; ckc[j] = cnow; }
        ++j;
        if (st.c != ctot) { tot = tot > 0.f ? tot * ex2(ctot - st.c) : 0.f; ctot = st.c; }
        tot += st.s;
        st.s = 0.f;
    };
    int since = 0;
    bool missing = false;
    LeanBatch<LT> B(st);
    auto begin = [&](const Vec8<LT> &first) { reference(first); B.begin(k); };
    constexpr bool kByVector = SHIFT && PASS == kTurns;   // (the same sums)
    auto one = [&](const Vec8<LT> &v) {
        if constexpr (kByVector) lean_push(st, v, k);
        else B.push(v);
    };
    auto batch = [&](const auto &in, int vi) {
        constexpr int D = std::decay_t<decltype(in)>::kDepth;
        if constexpr (!kByVector) B.template commit<D>(in, k, vi, hi);
        since += D;
        if (since >= CK) { checkpoint(); since = 0; B.again(); }
    };
    auto run = [&](const auto &in, const Iters &t) {   // (the loads of the next vectors also overlap the checkpoint's shuffle chain)
        constexpr int D = std::decay_t<decltype(in)>::kDepth;
        if constexpr (PASS == kBatches) row_batches<D, false>(in, lo + lane, hi, t, begin, one, [&](int vi) { batch(in, vi); });
        else row_turns<D>(in, lo + lane, hi, t, begin, one, [&](int vi) { batch(in, vi); });
    };
    if constexpr (SHIFT) {
        const Iters t = inside_iters(rq.src, rq.src, lo, hi);
        if (rq.src.sh == 0) run(AlignedIn<LT>{rq.src}, t);
        else run(ShiftedIn<LT>{rq.src}, t);
    } else if constexpr (PASS == kRing) {
        extern __shared__ __align__(128) unsigned char row_ring_mem[];
        __shared__ __align__(8) uint64_t row_ring_bars[THREADS / 32][kRowStages];
        const int warp = warp_index();
        const WholeIn<LT> in = {rq};
        RowRing R;
        row_ring_begin(R, row_ring_mem + warp * kRowWarpBytes, row_ring_bars[warp], rq.vec(lo),
                       (hi - lo) * static_cast<int>(sizeof(Vec8<LT>)), lane);
        missing = !ring_batches(R, lo, hi, lane, begin, one, [&](int vi) { batch(in, vi); });
    } else {
        run(WholeIn<LT>{rq}, whole_iters(lo, hi));
    }
    if (PASS == kRing && lane == 0) late = missing;
    if (since > 0) checkpoint();
    if (lane == 0)
        for (; j < slots; ++j) { cks[j] = 0.f; ckc[j] = 0.f; }
    Q.m2 = st.m2; Q.c = st.c; Q.s = tot;
}

// Did a copy of some warp's not arrive?  (Behind lean_reduce2; the whole warp.)
__device__ __forceinline__ bool lean_late(const LeanCkShared &sh, const Geo &g) {
    const int lane = threadIdx.x & 31;
    return __any_sync(kFull, lane < g.nwarps && sh.any[lane] != 0);
}

// The draws are made by one warp, the others are done: a sub-block is a few vectors per lane, and a CTA-wide draw costs
// every warp its barriers and its share of the picking (V = 32000: 5800 of the 12000 warp instructions of a row).
struct NoneOut {   // ids that a draw leaves out: none, one, the first n of a list
    template <class V> __device__ __forceinline__ void apply(int, V &) const {}
};
struct OneOut {
    int y;
    template <class V> __device__ __forceinline__ void apply(int vi, V &v) const { if (vi == (y >> 3)) v.drop(y & 7); }
};
struct ListOut {
    const int *x;
    int n;
    template <class V> __device__ __forceinline__ void apply(int vi, V &v) const {
        for (int i = 0; i < n; ++i)
            if (vi == (x[i] >> 3)) v.drop(x[i] & 7);
    }
};
// this lane's share of a sub-block: its consecutive vectors [b0 + lane * Bv, ...), summed without the ids left out
template <class ROW, class OUT>
__device__ __forceinline__ float ck_lane_sum(const ROW &row, float k, float C, int v0, int v1, OUT out) {
    float s = 0.f;
#pragma unroll 4
    for (int vi = v0; vi < v1; ++vi) {
        auto v = row[vi];
        out.apply(vi, v);
        s += vec_sum(v, f2_make(k, k), f2_make(-C, -C));
    }
    return s;
}
struct CkBlock { int b0, b1, Bv; };
__device__ __forceinline__ CkBlock ck_block(const Geo &g, int CK, int slot) {
    const int slots = lean_ck_slots(g, CK), w = slot / slots, j = slot - w * slots;
    CkBlock o;
    o.b0 = g.seg_lo(w) + 32 * CK * j;
    o.b1 = min(g.seg_hi(w), o.b0 + 32 * CK);
    o.Bv = (o.b1 - o.b0 + 31) >> 5;
    return o;
}

// The sub-block that holds id y is summed again without the ids left out: subtracting their own terms would cancel
// when they carry most of the sub-block's mass.  C = the row's exponent shift.
template <class ROW, class OUT>
__device__ __forceinline__ void lean_ck_drop(const Geo &g, const ROW &row, float k, float C, int CK, OUT out, int y, LeanCkShared &sh) {
    const int lane = threadIdx.x & 31, w = g.warp_of_vec(y >> 3);
    const int slot = w * lean_ck_slots(g, CK) + ((y >> 3) - g.seg_lo(w)) / (32 * CK);
    const CkBlock b = ck_block(g, CK, slot);
    const int v0 = b.b0 + lane * b.Bv;
    const float s = warp_sum(ck_lane_sum(row, k, C, v0, min(b.b1, v0 + b.Bv), out));
    if (lane == 0) { sh.cks[slot] = s; sh.ckc[slot] = C; }
    __syncwarp();
}

// Inverse-CDF draw from softmax(row) over the checkpoint sub-blocks, the ids left out having no weight (their
// sub-blocks' sums say so already).  C = the row's exponent shift.  Returns the token, -1 if nothing has mass.  Called
// by one warp, after the checkpoints are visible.
// A sub-block's sum is of its own scale: brought to the row's it may be above 0 where all its exponentials are below the
// smallest normal number, 0, and it has no id to give.  All of those together stay below kNoIds (2^19 ids), which targets
// are kept above where the draw's mass is not itself that small.
template <class ROW, class OUT>
__device__ __forceinline__ int lean_ck_draw(const Geo &g, const ROW &row, float k, float C, int CK, OUT out, float u, const LeanCkShared &sh) {
    const int lane = threadIdx.x & 31;
    const int nslot = g.nwarps * lean_ck_slots(g, CK), per = (nslot + 31) >> 5;   // (consecutive sub-blocks per lane)
    auto slot_mass = [&](int s) {
        const float cs = s < nslot ? sh.cks[s] : 0.f;
        return cs > 0.f ? cs * ex2(sh.ckc[s] - C) : 0.f;
    };
    float ls = 0.f;
    for (int i = 0; i < per; ++i) ls += slot_mass(lane * per + i);
    float t;
    int slot = pair_pick(ls, u, t, kNoIds);
    if (slot < 0) return -1;
    if (per > 1) {   // the sub-block within the lane's
        const int first = slot * per;
        int last = -1;
        slot = -1;
        float acc = 0.f, tt = 0.f, lastacc = 0.f;
        for (int i = 0; i < per; ++i) {
            const float m = slot_mass(first + i);
            if (m > 0.f) {
                last = first + i;
                lastacc = acc;
                if (slot < 0 && acc + m > t) { slot = first + i; tt = t - acc; }
            }
            acc += m;
        }
        if (slot < 0) { slot = last; tt = t - lastacc; }
        t = tt;
    }
    const CkBlock b = ck_block(g, CK, slot);
    const int v0 = b.b0 + lane * b.Bv;
    const int L = lanes_pick(ck_lane_sum(row, k, C, v0, min(b.b1, v0 + b.Bv), out), t);
    if (L < 0) return -1;
    // the picked lane's vectors over the lanes
    const int c0 = b.b0 + L * b.Bv, c1 = min(b.b1, c0 + b.Bv);
    float prefix = 0.f;
    int lastpos = -1;
    for (int vb = c0; vb < c1; vb += 32) {
        const int vi = vb + lane;
        float w[8], lsum = 0.f;
        auto v = row[min(vi, c1 - 1)];
        out.apply(vi, v);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            w[i] = vi < c1 ? ex2(__fmaf_rn(v.get(i), k, -C)) : 0.f;
            lsum += w[i];
        }
        const float incl = lanes_prefix(lsum);
        const unsigned pos = __ballot_sync(kFull, lsum > 0.f), hit = __ballot_sync(kFull, lsum > 0.f && prefix + incl > t);
        if (!pos) continue;
        const int M = hit ? __ffs(hit) - 1 : 31 - __clz(pos);
        float acc = prefix + (incl - lsum);
        int cand = -1, lastin = -1;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            acc += w[i];
            if (w[i] > 0.f) {
                lastin = vi * 8 + i;
                if (cand < 0 && acc > t) cand = lastin;
            }
        }
        lastpos = __shfl_sync(kFull, cand < 0 ? lastin : cand, M);
        if (hit) return lastpos;
        prefix += __shfl_sync(kFull, incl, 31);
    }
    return lastpos;
}

// Leaf rows (Figure 2: after the last accepted draft the bonus token is a draw from p) of a call
// whose rows are not split over clusters get a kernel of their own, shaped like the draft step:
// pass A over p with checkpoints, then the sub-block sampler.  CTAs of verifying rows leave at
// once; the verification kernels skip the leaf rows.  Up to three output sets receive the result
// (the three-method call: the methods share u_res, hence the bonus token).
template <typename LT, bool SHIFT, int THREADS, RowPass PASS>
__global__ void __launch_bounds__(THREADS, lean_ctas<SHIFT>(THREADS)) lean_leaf_kernel(LeafArgs A) {
    __shared__ LeanCkShared sh;
    pdl_begin();
    const RowArgs &a = A.r;
    const long long r = blockIdx.x;
    const int b = static_cast<int>(r / a.nodes), n = static_cast<int>(r % a.nodes);
    if (!(a.node_kind && a.node_kind[n] == SPECHUB_NODE_LEAF)) return;
    const StreamRow<LT, SHIFT> vp(static_cast<const LT *>(a.target) + b * a.stride_seq + n * a.stride_node, a.vocab);
    const Geo g = make_geo(a.vocab, 8);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int lo = g.seg_lo(warp), hi = g.seg_hi(warp);
    const float k = kLog2e / temperature_of(a, b);
    const int K = A.k;
    const float ures = a.uniforms[r * (2 * K + 1) + 2 * K];
    const int CK = lean_ck_interval(g), CS = lean_ck_slots(g, CK);
    LeanAcc<LT> tp, unused;
    unused.init();
    lean_pass_a_ck<SHIFT, THREADS, PASS>(vp, lo, hi, lane, k, CK, tp, sh.cks + warp * CS, sh.ckc + warp * CS, CS, sh.any[warp]);
    ArgMaxSum Ps, unusedq;
    lean_reduce2<false>(tp, unused, vp, vp, lo, hi, k, sh, Ps, unusedq);
    const float Zp = Ps.sx + Ps.own(k);
    if (warp != 0) return;
    uint32_t status = 0;
    int tok = -1;
    if (!(Ps.ml > neg_inf()) || !(Ps.ml < -neg_inf()) || !finite_pos(Zp)) status = SPECHUB_ST_NONFINITE;
    else if ((tok = lean_ck_draw(g, vp, k, Ps.c, CK, NoneOut{}, ures, sh)) < 0) tok = Ps.idx;   // (as in the draft step)
    if (threadIdx.x == 0) {
        for (int m = 0; m < A.n_out; ++m) {
            const NodeOutPtrs &o = A.out[m];
            o.accept_idx[r] = -1;
            o.token[r] = tok;
            if (o.hub) o.hub[r] = -1;
            for (int i = 0; i < K; ++i) {
                if (o.beta) o.beta[K * r + i] = 0.f;
                if (o.rate) o.rate[(K + 1) * r + i] = 0.f;
            }
            if (o.rate) o.rate[(K + 1) * r + K] = status ? 0.f : 1.f;
            if (o.status) o.status[r] = status;
        }
    }
}

// Passes B and C work on the exponentials themselves, in units of 1 / Z_p: with rho = Z_p / Z_q,
//   d = e_p - rho e_q = Z_p (p - q),   t = max(d, 0) - s rho e_q = Z_p (max(p - q, 0) - s q),
// two FMAs per vocabulary pair instead of two multiplications by 1/Z, a subtraction and an FMA.
// Identical target and draft rows give rho = 1 and e_p = e_q bit for bit, so d = 0 exactly.
__device__ __forceinline__ float lean_exp(float logit, float k, float c) { return ex2(__fmaf_rn(logit, k, -c)); }
__device__ __forceinline__ void lean_terms(float ep, float eq, float rho, float srho, float &d, float &t) {
    d = __fmaf_rn(-rho, eq, ep);
    t = __fmaf_rn(-srho, eq, fmaxf(d, 0.f));
}

// Sum of a row's exponentials outside id x, from the row's (maximum, argmax, sum without the argmax): RRSw's
// renormaliser 1 - q(x1) times Z_q without a pass over the row.  The argmax is left out of st.sx already; any
// other id holds at most half of the mass, so subtracting its own term costs at most one bit.
template <class ROW>
__device__ __forceinline__ float sum_without(const RowStat &st, const ROW &row, int x, float k) {
    if (x == st.idx) return st.sx;
    return __fsub_rn(__fadd_rn(st.sx, st.own), lean_exp(row.one(x), k, st.C));
}

// ------------------------------------------------------------------------------------------------
// Verification (SpecHub: Algorithm 3; RRS / RRSw: Algorithm 1) and leaf draws.
// ------------------------------------------------------------------------------------------------
// RING (RRS and RRSw, one CTA per row): the passes over both rows take their vectors from per-warp rings of
// bulk copies (spechub_ring.cuh; THREADS / 32 * kRingWarpBytes of dynamic shared memory) instead of loading
// them from global memory into registers.  Measured on V = 128256, 7936 rows: RRS 1.89 -> 1.72 ms, RRSw
// 1.99 -> 1.86 ms; SpecHub's two passes gain nothing from it (1.38 -> 1.38 .. 1.44 ms: the bookkeeping of
// the ring costs the issue slots that its pass B is short of), so SpecHub keeps the register-fed loops.
// STATS (one CTA per row): the maximum, argmax and sum of the draft row come from the record the draft
// step left (RowArgs::draft_stats_in), so pass A reads the target row only; a record that does not belong
// to the row (tag, argmax out of range, or another logit there than the recorded maximum) flags the row
// SPECHUB_ST_STATS; a shifted row (whose tag also marks it, row_mark) is then verified as without a record, its draft row
// read in a pass of its own.  The passes are register-fed, those over rows in whole words with L2 eviction hints on the
// loads (keep the target row after pass A, let the rows go at their last use): with a single row to keep in L2 between
// passes that beats the rings (RRS 1.53 -> 1.46 ms, RRSw 1.62 -> 1.60 ms on V = 128256, 7936 rows).
template <typename LT, bool SHIFT, int METHOD, int THREADS, int CS, bool RING = false, bool STATS = false>
__global__ void __launch_bounds__(THREADS, lean_ctas<SHIFT>(THREADS)) lean_verify_kernel(RowArgs a) {
    static_assert(!RING || (sizeof(LT) == 2 && !SHIFT), "the ring-fed form: bf16 rows in whole words");
    static_assert(!RING || (CS == 1 && METHOD != kSpecHub), "the ring-fed form: whole rows, RRS and RRSw");
    static_assert(!STATS || (CS == 1 && !RING), "draft statistics: whole rows, register-fed passes");
    __shared__ LeanShared sh;
    extern __shared__ __align__(128) unsigned char ring_mem[];
    __shared__ __align__(8) uint64_t ring_bars[RING ? THREADS / 32 : 1][kRingStages];
    // (Behind the leaf kernel of the same call, too: its rows are others, but what the kernels before it wrote is promised
    // only to a grid that waits itself.  Without
    // the wait a step with leaf rows took 163 us instead of 173 on 3840 rows of 32000 ids, 119 instead of 130 on 960 of 50257.)
    pdl_begin();
    const int me = RowGroup<CS>::rank();
    const long long r = blockIdx.x / CS;
    const int b = static_cast<int>(r / a.nodes), n = static_cast<int>(r % a.nodes);
    using V = Vec8<LT>;
    const StreamRow<LT, SHIFT> vp(static_cast<const LT *>(a.target) + b * a.stride_seq + n * a.stride_node, a.vocab);
    const StreamRow<LT, SHIFT> vq(static_cast<const LT *>(a.draft) + b * a.stride_seq + n * a.stride_node, a.vocab);
    const Geo g = make_geo(a.vocab, 8, CS, me);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int lo = g.seg_lo(warp), hi = g.seg_hi(warp);
    // (Pass B walks this lane's vectors backwards: what pass A read last is read again first, so
    // the tail of the row is still in L2 even when the rows in flight exceed its capacity.)
    const float k = kLog2e / temperature_of(a, b);
    const float pinf = -neg_inf();
    // leaf rows of an unsplit call belong to lean_leaf_kernel
    if (CS == 1 && a.node_kind && a.node_kind[n] == SPECHUB_NODE_LEAF) return;
    const bool leaf = CS > 1 && a.node_kind && a.node_kind[n] == SPECHUB_NODE_LEAF;
    const bool writer = (me == 0 && threadIdx.x == 0);

    NodeResult o;
    o.accept_idx = -1; o.token = -1; o.hub = -1; o.status = 0;
    o.beta[0] = o.beta[1] = 0.f; o.rate[0] = o.rate[1] = o.rate[2] = 0.f;
    // The token is written by the CTA that knows it: the row's first CTA for an accepted draft or
    // a flagged row, the CTA that draws for a residual / leaf token.
    bool token_elsewhere = false;

    // What the tests need of single ids -- the drafts, their logits, the uniforms, the draft row's record -- is fetched
    // by the last warp before it starts on pass A: two dependent look-ups that are off the path between the passes.
    // (Nothing else writes these fields; they are read after barriers.)
    if (warp == THREADS / 32 - 1) {
        const int t1 = a.draft_tokens_in[2 * r], t2 = a.draft_tokens_in[2 * r + 1];
        DraftStat ds = {};
        if (STATS) ds = static_cast<const DraftStat *>(a.draft_stats_in)[r];
        unsigned mark = 0;
        if constexpr (STATS && SHIFT) mark = row_mark(vq.src.row, a.vocab);
        int y = lane > 4 ? -1 : lane == 4 ? (STATS ? ds.idx : -1) : (lane & 1) ? t2 : t1;
        if (leaf) y = -1;
        float l = neg_inf();
        if (y >= 0 && y < a.vocab) l = lane < 2 ? vp.one(y) : vq.one(y);
        if (lane > 4 && lane < 8) l = a.uniforms[r * 5 + lane - 3];
        if (lane < 8) sh.lg[lane] = l;
        if (lane == 0) { sh.tk[0] = t1; sh.tk[1] = t2; }
        if (STATS && lane == 4) {
            bool ok = ds.tag == stat_tag(k, mark);
            // (a record of a row without a finite maximum or sum needs no look-up: the row is flagged
            // SPECHUB_ST_NONFINITE below, as it is without the record; a shifted row is read)
            const bool finite = ds.ml > neg_inf() && ds.ml < pinf && finite_pos(ds.sx + 1.f);
            if (SHIFT) ok = ok && finite;
            if (ok && finite)
                ok = ds.idx >= 0 && ds.idx < a.vocab && l == ds.ml;
            sh.stat_ok = ok;
            sh.x_ml[1] = ds.ml; sh.x_sx[1] = ds.sx; sh.x_idx[1] = ok ? ds.idx : 0;
        }
    }
    // the row's stream: pass A forwards, pass B backwards, (RRS, RRSw) pass C forwards
    WarpRing R;
    LeanAcc<LT> tp, tq;
    if constexpr (RING) {
        ring_begin(R, ring_mem + warp * kRingWarpBytes, ring_bars[warp], reinterpret_cast<const uint4 *>(vp.row),
                   reinterpret_cast<const uint4 *>(vq.row), lo, hi, 3, 2u, lane);
        lean_pass_a_ring(R, vp, vq, lane, k, tp, tq);
    } else if constexpr (STATS) {
        lean_pass_a1<true, false>(vp, lo, hi, lane, k, tp);
    } else if constexpr (CS > 1) {
        if (leaf) { tq.init(); lean_pass_a1<false, false>(vp, lo, hi, lane, k, tp); }
        else lean_pass_a2<METHOD != kSpecHub>(vp, vq, lo, hi, lane, k, tp, tq);
    } else {
        lean_pass_a2<METHOD != kSpecHub || THREADS == 512>(vp, vq, lo, hi, lane, k, tp, tq);
    }
    RowStat P, Q;
    {
        ArgMaxSum Ps, Qs;
        if (leaf || STATS) lean_reduce2<false>(tp, tq, vp, vq, lo, hi, k, sh, Ps, Qs);
        else lean_reduce2<true>(tp, tq, vp, vq, lo, hi, k, sh, Ps, Qs);
        if (threadIdx.x == 0) {
            sh.x_ml[0] = Ps.ml; sh.x_sx[0] = Ps.sx; sh.x_idx[0] = Ps.idx;
            if (!STATS) { sh.x_ml[1] = Qs.ml; sh.x_sx[1] = Qs.sx; sh.x_idx[1] = Qs.idx; }
        }
        bool from_record = STATS;
        if constexpr (STATS && SHIFT) {
            // A record that is not the row's: as if there were none (rows that were once read without looking at records
            // still come with whatever their caller has).  Same vectors, same order, so the plain call's bits but for
            // RRSw's 1 - q(x1), which is sum_without's here.
            if (!sh.stat_ok) {
                lean_pass_a1<false, false>(vq, lo, hi, lane, k, tq);
                lean_reduce2<true>(tp, tq, vp, vq, lo, hi, k, sh, Ps, Qs);
                from_record = false;
            }
        }
        if (CS == 1) {   // (the published values are read by a draw from p only, after further barriers)
            if (from_record) { Qs.ml = sh.x_ml[1]; Qs.c = shift_of(Qs.ml, k); Qs.sx = sh.x_sx[1]; Qs.idx = sh.x_idx[1]; }
            P.set(Ps, k);
            Q.set(Qs, k);
        }
    }
    if (CS > 1) {
        RowGroup<CS>::sync();  // [1] slices published
        merge_slices<CS>(sh, 0, k, P);
        merge_slices<CS>(sh, 1, k, Q);
    }
    const float r1 = sh.lg[5], r2 = sh.lg[6], ures = sh.lg[7];
    // (Z_p, its shift and rho change only in verification from draft statistics, when the two rows turn
    // out to be the same row: see below)
    float Zp = P.sx + P.own;
    const float Zq = Q.sx + Q.own;
    float cP = P.C, invZp = 1.f / Zp;
    const float cQ = Q.C, invZq = 1.f / Zq;
    float rho = __fdiv_rn(Zp, Zq);
    // With draft statistics Z_q was summed by another kernel, in another order than Z_p here.  That is
    // rounding, except when the target row is the draft row bit for bit: then Z_p = Z_q, every p - q is 0 and
    // the sums S1, R, A1 are exactly 0, which a rho of 1 +- 1e-7 would turn into noise that the tests then
    // divide by.  Pass B sees both rows and notices; the row is then redone with p's normaliser set to q's.
    unsigned diff = 0;
    auto take_q_normaliser = [&]() { Zp = Zq; invZp = invZq; cP = cQ; rho = 1.f; };
    const int x1 = sh.tk[0], x2 = sh.tk[1];
    auto prob_p = [&](int i) { return prob_of(sh.lg[i], k, cP, invZp); };       // of draft i
    auto prob_q = [&](int i) { return prob_of(sh.lg[2 + i], k, cQ, invZq); };
    auto draw_from_p = [&]() {  // every CTA of the row calls it
        const int tok = lean_sample_row<CS>(g, vp, k, P, me, -1, ures, 0, sh);
        if (tok != -2 && threadIdx.x == 0) a.token[r] = tok;
        token_elsewhere = true;
    };

    do {
        if (STATS && !SHIFT && !sh.stat_ok) { o.status = SPECHUB_ST_STATS; break; }
        if (!(P.ml > neg_inf()) || !(P.ml < pinf) || !finite_pos(Zp)) { o.status = SPECHUB_ST_NONFINITE; break; }
        if (leaf) {
            // bonus token after the last accepted draft (Figure 2): a draw from p
            draw_from_p();
            o.rate[2] = 1.f;
            break;
        }
        if (!(Q.ml > neg_inf()) || !(Q.ml < pinf) || !finite_pos(Zq)) { o.status = SPECHUB_ST_NONFINITE; break; }
        if (METHOD == kSpecHub) {
            const int hubtok = Q.idx;
            o.hub = hubtok;
            const bool pair_xa = (x2 == hubtok && x1 != hubtok), pair_ax = (x1 == hubtok && x2 != hubtok);
            const int x = pair_xa ? x1 : x2;
            if (!(pair_xa || pair_ax) || x < 0 || x >= a.vocab) { o.status = SPECHUB_ST_TOKEN_RANGE; break; }
            const bool degenerate = !(Q.sx > 0.f);
            const float c = degenerate ? 0.f : Q.own / Q.sx;
            float crho = c * rho;
            const float qa = Q.own * invZq, rest = Q.sx * invZq;
            const int hubvec = hubtok >> 3, hubel = hubtok & 7;
            const int ix = pair_xa ? 0 : 1;   // the draft that is not the hub
            float px = prob_p(ix);
            const float qx = prob_q(ix);
            if (!a.beta && !a.rate) {
                // No probability is asked for: the first test needs scalars only, and if it accepts
                // the transport sums decide nothing.
                const bool acc1 = pair_xa ? accept_test(r1, px, qx, o.beta[0], true, o.status)
                                          : accept_test(r1, fmaxf(__fsub_rn(px, qx), 0.f), c * qx, o.beta[0], true, o.status);
                if (acc1) {
                    o.accept_idx = pair_xa ? 0 : 1;
                    o.token = x;
                    if (degenerate) o.status |= SPECHUB_ST_DEGENERATE_Q;
                    break;
                }
                o.status = 0;  // the full path below sets the flags again
            }
            // pass B: S1, S2, R over ids != a (Section 4, Appendix B.1)
            // (packed: the low lane takes the even ids of a vector, the high lane the odd ones)
            F2 s1, s2, rr;
            auto pass_b = [&]() {
            s1 = s2 = rr = f2_make(0.f, 0.f);
            const F2 k2 = f2_make(k, k), ncp2 = f2_make(-cP, -cP), ncq2 = f2_make(-cQ, -cQ);
            const F2 nrho2 = f2_make(-rho, -rho), ncrho2 = f2_make(-crho, -crho);
            auto vec_b = [&](int vi, V cp, V cq) {
                if (STATS) diff |= cp.differs(cq);
                if (vi == hubvec) {   // the hub's own pair is no part of the sums over y != a: -inf, mass 0
                    cp.drop(hubel);
                    cq.drop(hubel);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const F2 ep = f2_exp(cp.pair(i), k2, ncp2), eq = f2_exp(cq.pair(i), k2, ncq2);
                    const F2 d = f2_fma(nrho2, eq, ep);       // Z_p (p - q)
                    const F2 m = f2_max0(d);
                    const F2 t = f2_fma(ncrho2, eq, m);       // Z_p (max(p - q, 0) - c q)
                    const F2 w = f2_max0(t);
                    s1 = f2_add(s1, f2_sub(m, d));            // max(-d, 0) = max(d, 0) - d, exactly
                    s2 = f2_add(s2, f2_sub(w, t));
                    rr = f2_add(rr, w);
                }
            };
            // This is the last use of both rows: the loads tell L2 to let these lines go first (one
            // CTA per row: 1.38 -> 1.30 ms on V = 128256; from draft statistics, where pass A also told
            // L2 to keep the target row's lines, 1.07 -> 1.02 ms.  Keep-hints on pass A of the kernel
            // that reads both rows twice cost it 7-13 %).
            if constexpr (CS == 1) stream_pairs_last<-1>(vp, vq, lo, hi, lane, vec_b);
            else stream_pairs<-1>(vp, vq, lo, hi, lane, vec_b);
            };
            pass_b();
            float acc[3] = {f2_sum(s1), f2_sum(s2), f2_sum(rr)};
            float part[3][CS];
            lean_row_sums<CS, 3, 0, STATS>(acc, part, sh, &diff);  // [2]
            const float *mass_r = sh.acc[2];
            if (STATS && !diff) {
                take_q_normaliser();
                crho = c;
                px = qx;
                pass_b();
                acc[0] = f2_sum(s1); acc[1] = f2_sum(s2); acc[2] = f2_sum(rr);
                lean_row_sums<CS, 3, 3>(acc, part, sh);
                mass_r = sh.acc[5];
            }
            // the sums are in units of 1 / Z_p; Rraw stays in them for the residual draw
            const float Rraw = acc[2];
            const float S1 = acc[0] * invZp, S2 = degenerate ? qa : acc[1] * invZp, R = Rraw * invZp;
            const float pa = prob_p(1 - ix);
            const float hub_left = fmaxf(pa - S2, 0.f);
            o.rate[0] = fmaxf(rest - S1, 0.f) + fminf(pa, S2);
            o.rate[1] = (degenerate ? 0.f : fmaxf(qa - S2, 0.f)) + fminf(hub_left, S1);
            o.rate[2] = R;
            if (degenerate) o.status |= SPECHUB_ST_DEGENERATE_Q;
            bool acc1, acc2;
            if (pair_xa) {
                acc1 = accept_test(r1, px, qx, o.beta[0], true, o.status);
                if (acc1) { o.accept_idx = 0; o.token = x; }
                acc2 = accept_test(r2, hub_left, S1, o.beta[1], !acc1, o.status);
                if (!acc1 && acc2) { o.accept_idx = 1; o.token = hubtok; }
            } else {
                acc1 = accept_test(r1, fmaxf(__fsub_rn(px, qx), 0.f), c * qx, o.beta[0], true, o.status);
                if (acc1) { o.accept_idx = 1; o.token = x; }
                acc2 = accept_test(r2, pa, S2, o.beta[1], !acc1, o.status);
                if (!acc1 && acc2) { o.accept_idx = 0; o.token = hubtok; }
            }
            if (!(acc1 || acc2)) {
                o.accept_idx = -1;
                const double target = static_cast<double>(ures) * Rraw;   // (CS > 1)
                double base = 0.;
                const int sel = (Rraw > 0.f) ? pick_part(part[2], CS, target, base) : -1;
                if (sel < 0) {
                    o.status |= SPECHUB_ST_ZERO_RESIDUAL;
                    draw_from_p();
                } else {
                    token_elsewhere = true;
                    if (sel == me) {
                        auto wf = [&](int vi, float(&w)[8]) {
                            const V fp = vp[vi], fq = vq[vi];
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                float d, t;
                                lean_terms(lean_exp(fp.get(i), k, cP), lean_exp(fq.get(i), k, cQ), rho, crho, d, t);
                                w[i] = (vi * 8 + i == hubtok) ? 0.f : fmaxf(t, 0.f);
                            }
                        };
                        const int tok = block_sample3<CS == 1>(g, wf, mass_r, sh, CS == 1 ? ures : static_cast<float>(target - base));
                        if (threadIdx.x == 0) a.token[r] = tok;
                    }
                }
            }
        } else {
            if (x1 < 0 || x1 >= a.vocab || x2 < 0 || x2 >= a.vocab) { o.status = SPECHUB_ST_TOKEN_RANGE; break; }
            if (!a.beta && !a.rate) {
                // no probability asked for: an accepted first draft needs no sum at all
                if (accept_test(r1, prob_p(0), prob_q(0), o.beta[0], true, o.status)) {
                    o.accept_idx = 0;
                    o.token = x1;
                    break;
                }
                o.status = 0;
            }
            // RRS on bf16 rows in whole words takes plain loops unrolled twice, two pairs of loads at once, through passes B
            // and C.  With one pair ahead instead: from draft statistics 7936 rows of 128256 ids 1412 -> 1543 us, of 32000
            // 397 -> 399, without them 1920 rows of 50048 195 -> 199; but fp32 rows, 992 of 128256, 444 -> 432, 1920 of 32000
            // 199 -> 184, and RRSw, whose pass B also keeps x1's place, 2.21 -> 2.03 ms on 7936 rows of 128256.
            constexpr bool kTwoAtOnce = METHOD == kRRS && !SHIFT && sizeof(LT) == 2;
            // pass B: A1 = sum max(p - q, 0); RRSw also sums q outside x1 directly
            const int x1vec = x1 >> 3, x1el = x1 & 7;
            float dna = 0.f, dnb = 0.f;
            F2 a1;   // (packed: low lane = even ids of a vector, high lane = odd ids)
            const F2 k2 = f2_make(k, k), ncq2 = f2_make(-cQ, -cQ);
            F2 ncp2, nrho2;
            auto vec_b = [&](int vi, const V &cp, const V &cq) {
                if (STATS) diff |= cp.differs(cq);
                F2 eq[4];   // e_q of the vector, by words
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    eq[i] = f2_exp(cq.pair(i), k2, ncq2);
                    a1 = f2_add(a1, f2_max0(f2_fma(nrho2, eq[i], f2_exp(cp.pair(i), k2, ncp2))));
                }
                if (METHOD == kRRSw && !STATS) {   // (from draft statistics: sum_without, below)
                    float qq[8];
#pragma unroll
                    for (int i = 0; i < 4; ++i) f2_get(eq[i], qq[2 * i], qq[2 * i + 1]);
                    if (vi == x1vec) {
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if (i == x1el) qq[i] = 0.f;
                    }
                    dna += (qq[0] + qq[1]) + (qq[2] + qq[3]);
                    dnb += (qq[4] + qq[5]) + (qq[6] + qq[7]);
                }
            };
            auto pass_b = [&](bool from_ring) {
            a1 = f2_make(0.f, 0.f); dna = 0.f; dnb = 0.f;
            ncp2 = f2_make(-cP, -cP); nrho2 = f2_make(-rho, -rho);
            if constexpr (RING) {
            if (from_ring) {
#pragma unroll 1
                for (int c = R.nc - 1; c >= 0; --c) {
                    ring_wait(R);
                    const int v0 = lo + lane + c * kRingChunkVecs;
#pragma unroll
                    for (int j = kRingCh - 1; j >= 0; --j) {
                        V x, y;
                        ring_load(R, j, lane, x, y);
                        if (j == 0) ring_release(R, lane);
                        if (v0 + j * 32 < hi) vec_b(v0 + j * 32, x, y);
                    }
                }
                return;
            }
            }
            if constexpr (kTwoAtOnce) {
                const int n = (hi - lo - lane + 31) >> 5;   // this lane's vectors
#pragma unroll 2
                for (int vi = lo + lane + 32 * (n - 1); vi >= lo; vi -= 32) vec_b(vi, vp[vi], vq[vi]);
            } else {
                stream_pairs<-1>(vp, vq, lo, hi, lane, vec_b);
            }
            };
            pass_b(true);
            float acc[2] = {f2_sum(a1), dna + dnb};
            float part2[2][CS];
            lean_row_sums<CS, 2, 0, STATS>(acc, part2, sh, &diff);  // [2]
            if (STATS && !diff) {
                take_q_normaliser();
                pass_b(false);
                acc[0] = f2_sum(a1); acc[1] = dna + dnb;
                lean_row_sums<CS, 2, 4>(acc, part2, sh);
            }
            if (STATS && METHOD == kRRSw) acc[1] = sum_without(Q, vq, x1, k);
            const float A1 = acc[0] * invZp, den = acc[1] * invZq;   // the sums are of exponentials
            const bool q1_zero = (METHOD == kRRSw) && !(den > 0.f);
            const float gq = (METHOD == kRRSw) ? (q1_zero ? 0.f : 1.f / den) : 1.f;
            const float A1g = A1 * gq;
            const float A1grho = A1g * rho;
            // pass C: mass of the residual after two rejections
            F2 w2 = f2_make(0.f, 0.f);
            const F2 nsc2 = f2_make(-A1grho, -A1grho);
            auto vec_c = [&](int vi, const V &cp, const V &cq) {
                if (METHOD == kRRSw && vi == x1vec) {   // (one vector of the row) q1(x1) = 0: that lane's scale is 0
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        F2 nsc = nsc2;
                        if (i == (x1el >> 1)) nsc = (x1el & 1) ? f2_make(-A1grho, 0.f) : f2_make(0.f, -A1grho);
                        const F2 eq = f2_exp(cq.pair(i), k2, ncq2);
                        const F2 m = f2_max0(f2_fma(nrho2, eq, f2_exp(cp.pair(i), k2, ncp2)));
                        w2 = f2_add(w2, f2_max0(f2_fma(nsc, eq, m)));
                    }
                    return;
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const F2 eq = f2_exp(cq.pair(i), k2, ncq2);
                    const F2 m = f2_max0(f2_fma(nrho2, eq, f2_exp(cp.pair(i), k2, ncp2)));
                    w2 = f2_add(w2, f2_max0(f2_fma(nsc2, eq, m)));
                }
            };
            if constexpr (RING) {
#pragma unroll 1
                for (int c = 0; c < R.nc; ++c) {
                    ring_wait(R);
                    const int v0 = lo + lane + c * kRingChunkVecs;
#pragma unroll
                    for (int j = 0; j < kRingCh; ++j) {
                        V x, y;
                        ring_load(R, j, lane, x, y);
                        if (j == kRingCh - 1) ring_release(R, lane);
                        if (v0 + j * 32 < hi) vec_c(v0 + j * 32, x, y);
                    }
                }
            } else if constexpr (kTwoAtOnce) {
                uint64_t pol = 0;   // one CTA per row: the rows' last use, as in stream_pairs_last
                if (CS == 1) asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
#pragma unroll 2
                for (int vi = lo + lane; vi < hi; vi += 32) {
                    if (CS == 1) vec_c(vi, vp.fetch(vi, pol), vq.fetch(vi, pol));
                    else vec_c(vi, vp[vi], vq[vi]);
                }
            } else if constexpr (CS == 1) {
                stream_pairs_last<1>(vp, vq, lo, hi, lane, vec_c);
            } else {
                stream_pairs<1>(vp, vq, lo, hi, lane, vec_c);
            }
            float w2a, w2b;
            f2_get(w2, w2a, w2b);
            float w2s[1] = {w2a + w2b};
            float part1[1][CS];
            lean_row_sums<CS, 1, 2>(w2s, part1, sh);  // [3]
            const float W2raw = w2s[0], W2 = W2raw * invZp;
            o.rate[0] = fmaxf(1.f - A1, 0.f);
            o.rate[1] = fmaxf(A1 - W2, 0.f);
            o.rate[2] = W2;
            const float px1 = prob_p(0), qx1 = prob_q(0), px2 = prob_p(1), qx2 = prob_q(1);
            const bool acc1 = accept_test(r1, px1, qx1, o.beta[0], true, o.status);
            if (acc1) { o.accept_idx = 0; o.token = x1; }
            if (!acc1 && q1_zero) o.status |= SPECHUB_ST_DEGENERATE_Q;
            bool acc2 = false;
            if (A1 > 0.f) {
                const float q1x2 = (METHOD == kRRSw && x2 == x1) ? 0.f : A1g * qx2;
                acc2 = accept_test(r2, fmaxf(__fsub_rn(px2, qx2), 0.f), q1x2, o.beta[1], !acc1, o.status);
            }
            if (!acc1 && acc2) { o.accept_idx = 1; o.token = x2; }
            if (!(acc1 || acc2)) {
                o.accept_idx = -1;
                const double target = static_cast<double>(ures) * W2raw;   // (CS > 1)
                double base = 0.;
                const int sel = (A1 > 0.f && W2raw > 0.f) ? pick_part(part1[0], CS, target, base) : -1;
                if (sel < 0) {
                    o.status |= SPECHUB_ST_ZERO_RESIDUAL;
                    draw_from_p();
                } else {
                    token_elsewhere = true;
                    if (sel == me) {
                        auto wf = [&](int vi, float(&w)[8]) {
                            const V fp = vp[vi], fq = vq[vi];
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                float d, t;
                                const float s = (METHOD == kRRSw && vi * 8 + i == x1) ? 0.f : A1grho;
                                lean_terms(lean_exp(fp.get(i), k, cP), lean_exp(fq.get(i), k, cQ), rho, s, d, t);
                                w[i] = fmaxf(t, 0.f);
                            }
                        };
                        const int tok = block_sample3<CS == 1>(g, wf, sh.acc[2], sh, CS == 1 ? ures : static_cast<float>(target - base));
                        if (threadIdx.x == 0) a.token[r] = tok;
                    }
                }
            }
        }
    } while (false);
    if (RING) {
        // no copy may be on its way into this CTA's shared memory when it ends; a stage that never arrived
        // (every wait is bounded) is reported with the row
        ring_drain(R);
        if (__syncthreads_or(R.timed_out)) o.status |= SPECHUB_ST_INTERNAL;
    }
    if (writer) {
        a.accept_idx[r] = o.accept_idx;
        if (!token_elsewhere) a.token[r] = o.token;
        if (a.hub) a.hub[r] = o.hub;
        if (a.beta) { a.beta[2 * r] = o.beta[0]; a.beta[2 * r + 1] = o.beta[1]; }
        if (a.rate) { a.rate[3 * r] = o.rate[0]; a.rate[3 * r + 1] = o.rate[1]; a.rate[3 * r + 2] = o.rate[2]; }
        if (a.status) a.status[r] = o.status;
    }
    if (CS > 1) RowGroup<CS>::sync();  // no CTA leaves while another may still read its shared memory
}

// ------------------------------------------------------------------------------------------------
// Draft step (Section 4 / Algorithm 3 for SpecHub; Algorithm 1 for RRS, RRSw).
// ------------------------------------------------------------------------------------------------
template <int THREADS, int CS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) lean_draft_kernel(RowArgs a, int method) {
    __shared__ LeanShared sh;
    pdl_begin();
    const int me = RowGroup<CS>::rank();
    const long long r = blockIdx.x / CS;
    const int b = static_cast<int>(r / a.nodes), n = static_cast<int>(r % a.nodes);
    const __nv_bfloat16 *rowq = static_cast<const __nv_bfloat16 *>(a.draft) + b * a.stride_seq + n * a.stride_node;
    const StreamRow<__nv_bfloat16, false> vq(rowq, a.vocab);
    const Geo g = make_geo(a.vocab, 8, CS, me);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int lo = g.seg_lo(warp), hi = g.seg_hi(warp);
    const float k = kLog2e / temperature_of(a, b);
    const float u1 = a.uniforms[r * 5 + 0], u2 = a.uniforms[r * 5 + 1];
    const bool writer = (me == 0 && threadIdx.x == 0);

    LeanAcc<__nv_bfloat16> tq, unused;
    unused.init();
    lean_pass_a1<false, false>(vq, lo, hi, lane, k, tq);
    {
        ArgMaxSum q, unusedq;
        lean_reduce2<false>(tq, unused, vq, vq, lo, hi, k, sh, q, unusedq);
        if (threadIdx.x == 0) { sh.x_ml[0] = q.ml; sh.x_sx[0] = q.sx; sh.x_idx[0] = q.idx; sh.x_tok = -3; }
    }
    RowGroup<CS>::sync();  // [1]
    RowStat Q;
    merge_slices<CS>(sh, 0, k, Q);
    const float Zq = Q.sx + Q.own;
    uint32_t st = 0;
    const bool bad = !(Q.ml > neg_inf()) || !finite_pos(Zq) || !(Q.ml < -neg_inf());
    const int hubtok = bad ? -1 : Q.idx;
    if (writer) void_draft_stat(a, r);
    if (bad) {
        if (writer) {
            a.draft_tokens_out[2 * r] = -1; a.draft_tokens_out[2 * r + 1] = -1;
            if (a.hub) a.hub[r] = -1;
            if (a.draft_prob) { a.draft_prob[2 * r] = 0.f; a.draft_prob[2 * r + 1] = 0.f; }
            if (a.status) a.status[r] = SPECHUB_ST_NONFINITE;
        }
    } else {
        // x1 ~ q.  The CTA whose slice holds the target draws it and tells the others.
        const int t1 = lean_sample_row<CS>(g, vq, k, Q, me, -1, u1, 0, sh);
        int x1 = t1;
        if (CS > 1) {
            if (t1 != -2 && threadIdx.x == 0) sh.x_tok = t1;
            RowGroup<CS>::sync();  // [2]
            x1 = -1;
#pragma unroll
            for (int c = 0; c < CS; ++c) {
                const int v = RowGroup<CS>::peer(&sh, c)->x_tok;
                if (v != -3) x1 = v;
            }
        }
        float prob0 = 0.f, prob1 = 0.f;
        bool x2_elsewhere = false;  // x2 (and its probability) written by the CTA that draws it
        int x2 = -1;
        if (method == kSpecHub) {
            prob0 = Q.own / Zq;
            if (x1 != hubtok) {
                x2 = hubtok;
                prob1 = ex2(fmaf(load_one<__nv_bfloat16>(rowq, x1), k, -Q.C)) / Zq;
            } else if (!(Q.sx > 0.f)) {
                x2 = (hubtok == 0) ? 1 : 0;
                st |= SPECHUB_ST_DEGENERATE_Q;
            } else {
                int t2 = lean_sample_row<CS>(g, vq, k, Q, me, hubtok, u2, 0, sh);
                if (t2 == -1) t2 = hubtok == 0 ? 1 : 0;   // (what is left is below the smallest normal number)
                x2_elsewhere = true;
                if (t2 != -2 && threadIdx.x == 0) {
                    a.draft_tokens_out[2 * r + 1] = t2;
                    if (a.draft_prob)
                        a.draft_prob[2 * r + 1] = prob0 * ex2(fmaf(load_one<__nv_bfloat16>(rowq, t2), k, -Q.C)) / Q.sx;
                }
            }
        } else if (method == kRRS) {
            const int t2 = lean_sample_row<CS>(g, vq, k, Q, me, -1, u2, 0, sh);
            x2_elsewhere = true;
            if (t2 != -2 && threadIdx.x == 0) a.draft_tokens_out[2 * r + 1] = t2;
        } else {
            // q with q(x1) set to 0.  The mass of the slice that holds x1 is its sum minus x1's term:
            // unless x1 is that slice's argmax (which the published sum already leaves out), the
            // argmax's own term stays in, so at most half of the sum cancels.
            const int per = (g.nvec + CS - 1) / CS;
            const int ox = min((x1 >> 3) / per, CS - 1);
            const float lx1 = load_one<__nv_bfloat16>(rowq, x1);
            float m[CS];
            double total = 0.;
#pragma unroll
            for (int c = 0; c < CS; ++c) {
                m[c] = slice_mass<CS>(sh, 0, Q, c, x1, k);
                if (c == ox && RowGroup<CS>::peer(&sh, c)->x_idx[0] != x1)
                    m[c] = fmaxf(m[c] - ex2(__fmaf_rn(lx1, k, -Q.C)), 0.f);
                total += m[c];
            }
            x2_elsewhere = true;
            double base = 0.;
            const int sel = (total > 0.) ? pick_part(m, CS, u2 * total, base) : -1;
            if (sel < 0) {
                st |= SPECHUB_ST_DEGENERATE_Q;
                if (writer) a.draft_tokens_out[2 * r + 1] = (x1 == 0) ? 1 : 0;
            } else if (sel == me) {
                const int t2 = lean_sample_slice<CS>(g, vq, k, Q, x1, static_cast<float>(u2 * total - base), 0, sh);
                if (threadIdx.x == 0) a.draft_tokens_out[2 * r + 1] = t2;
            }
        }
        if (writer) {
            a.draft_tokens_out[2 * r] = x1;
            if (!x2_elsewhere) a.draft_tokens_out[2 * r + 1] = x2;
            if (a.hub) a.hub[r] = (method == kSpecHub) ? hubtok : -1;
            if (a.draft_prob) {
                a.draft_prob[2 * r] = prob0;
                if (!x2_elsewhere) a.draft_prob[2 * r + 1] = prob1;
            }
            if (a.status) a.status[r] = st;
        }
    }
    if (CS > 1) RowGroup<CS>::sync();
}

// ------------------------------------------------------------------------------------------------
// Draft step, one CTA per row (checkpointed pass A and sub-block sampler above).
// ------------------------------------------------------------------------------------------------
template <typename LT, bool SHIFT, int THREADS, RowPass PASS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) lean_draft_ck_kernel(RowArgs a, int method, bool keep_stats) {   // (shifted rows: marked ones)
    __shared__ LeanCkShared sh;
    pdl_begin();
    const long long r = blockIdx.x;
    const int b = static_cast<int>(r / a.nodes), n = static_cast<int>(r % a.nodes);
    const StreamRow<LT, SHIFT> vq(static_cast<const LT *>(a.draft) + b * a.stride_seq + n * a.stride_node, a.vocab);
    const Geo g = make_geo(a.vocab, 8);
    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int lo = g.seg_lo(warp), hi = g.seg_hi(warp);
    const float k = kLog2e / temperature_of(a, b);
    const float u1 = a.uniforms[r * 5 + 0], u2 = a.uniforms[r * 5 + 1];
    const int CK = lean_ck_interval(g), CS = lean_ck_slots(g, CK);

    LeanAcc<LT> tq, unused;
    unused.init();
    lean_pass_a_ck<SHIFT, THREADS, PASS>(vq, lo, hi, lane, k, CK, tq, sh.cks + warp * CS, sh.ckc + warp * CS, CS, sh.any[warp]);
    RowStat Q;
    {
        ArgMaxSum q, unusedq;
        lean_reduce2<false>(tq, unused, vq, vq, lo, hi, k, sh, q, unusedq);
        Q.set(q, k);
    }
    if (warp != 0) return;
    const float Zq = Q.sx + Q.own;
    uint32_t st = 0;
    const bool late = PASS == kRing && lean_late(sh, g);   // (nothing is drawn from, or recorded of, a part of the row)
    int x1 = -1, x2 = -1, hubtok = -1;
    float prob0 = 0.f, prob1 = 0.f;
    if (late) {
        st = SPECHUB_ST_INTERNAL;
    } else if (!(Q.ml > neg_inf()) || !finite_pos(Zq) || !(Q.ml < -neg_inf())) {
        st = SPECHUB_ST_NONFINITE;
    } else {
        hubtok = Q.idx;
        x1 = lean_ck_draw(g, vq, k, Q.C, CK, NoneOut{}, u1, sh);
        if (x1 < 0) x1 = hubtok;   // (a sub-block without an id, by rounding at its edge)
        if (method == kSpecHub) {
            prob0 = Q.own / Zq;
            if (x1 != hubtok) {
                x2 = hubtok;
                prob1 = ex2(fmaf(vq.one(x1), k, -Q.C)) / Zq;
            } else if (!(Q.sx > 0.f)) {
                x2 = (hubtok == 0) ? 1 : 0;
                st |= SPECHUB_ST_DEGENERATE_Q;
            }
        } else if (method == kRRS) {
            x2 = lean_ck_draw(g, vq, k, Q.C, CK, NoneOut{}, u2, sh);
            if (x2 < 0) x2 = hubtok;
        }
        if (x2 < 0 && method != kRRS) {   // q without x1 (SpecHub: x1 is the hub)
            lean_ck_drop(g, vq, k, Q.C, CK, OneOut{x1}, x1, sh);
            x2 = lean_ck_draw(g, vq, k, Q.C, CK, OneOut{x1}, u2, sh);
            if (x2 < 0) {   // nothing left once x1 is removed
                x2 = (x1 == 0) ? 1 : 0;
                st |= SPECHUB_ST_DEGENERATE_Q;
            } else if (method == kSpecHub) {
                prob1 = prob0 * ex2(fmaf(vq.one(x2), k, -Q.C)) / Q.sx;
            }
        }
    }
    unsigned mark = 0;
    if constexpr (SHIFT)
        if (keep_stats && a.draft_stats_out) mark = row_mark(vq.src.row, a.vocab);
    if (threadIdx.x == 0) {
        if (a.draft_stats_out) {
            DraftStat ds = {};
            if (keep_stats && !late) { ds.ml = Q.ml; ds.sx = Q.sx; ds.idx = Q.idx; ds.tag = stat_tag(k, mark); }
            static_cast<DraftStat *>(a.draft_stats_out)[r] = ds;
        }
        a.draft_tokens_out[2 * r] = x1;
        a.draft_tokens_out[2 * r + 1] = x2;
        if (a.hub) a.hub[r] = (method == kSpecHub) ? hubtok : -1;
        if (a.draft_prob) { a.draft_prob[2 * r] = prob0; a.draft_prob[2 * r + 1] = prob1; }
        if (a.status) a.status[r] = st;
    }
}

}  // namespace spechub
