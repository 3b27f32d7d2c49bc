// Rows held in registers: each row is read from memory once, every lane keeps up to NV logical vectors (8 ids each)
// of it, and all passes of a step run over those registers.
//
// A row is cut into contiguous parts, one per warp: W warps of a CTA, on CS CTAs of a cluster when one CTA's
// warps do not hold it.  Short rows take one warp or a few, several rows per CTA, and never meet a CTA-wide
// barrier.  Vector j of a part's lane l is the part's (32 j + l)-th: a load is one contiguous request.  (Consecutive
// vectors per lane would make draws simpler, but each load then touches up to 32 lines: 31 rows of 128256 ids, 8000
// cycles for the loads alone.)  After each pass every warp posts a small record into the shared memory of all CTAs of
// its row, one barrier follows (a warp barrier, a named barrier, or the cluster's), and every warp merges the records
// for itself in the same order: all warps hold bit-identical row values, take the same decisions, and pick the same
// part in an inverse-CDF draw, whose warp draws from its registers.
//
// What bounds these kernels is the chain load -> reduce -> barrier -> reduce -> draw, a few microseconds, not
// bandwidth.  They take the calls whose rows do not fill the GPU: a row spread over many warps instead of one
// CTA streaming it, one read of the row, and two exponentials per id and pass.
#pragma once

#include <cooperative_groups.h>

#include "spechub.h"
#include "spechub_args.cuh"
#include "spechub_common.cuh"
#include "spechub_stream.cuh"
#include "spechub_vec.cuh"

namespace spechub {
namespace cg = cooperative_groups;

constexpr int kRegMaxParts = 128;   // warps per row: 16 x a cluster of 8
constexpr int kRegThreads = 512;    // threads of a CTA, at most
constexpr int kRegPer = kRegMaxParts / 32;   // records per lane, at most: consecutive parts

struct RegGeo { int w, cs, rows_per_cta, seg; };   // warps per row and CTA, CTAs per row, rows per CTA, vectors per part

struct RegShared {
    float2 p[kRegMaxParts];        // (max logit, sum of exponentials on that maximum's scale)
    float4 q[kRegMaxParts];        // the same, the sum without the part's argmax, the argmax
    float4 sum[2][kRegMaxParts];   // sums of a pass, two buffers
    float2 drawn[kMaxK][4];        // draft step: a drawn id and what its part weighs without it, per row of the CTA
};

struct RegRow {   // this warp's place in its row
    int part, parts, slot0;    // its part, the parts of the row, the row's first record
    int lo, hi, seg;           // its vectors; vectors per part
    int nj, lv;                // vectors per lane, this lane's first (the others follow at distances of 32)
    int per;                   // records per lane
    int w, cs, rows_per_cta, group;
    unsigned r;                // the row

    __device__ __forceinline__ RegRow(const RegGeo &g, int vocab) {
        const int warp = threadIdx.x >> 5;
        w = g.w; cs = g.cs; rows_per_cta = g.rows_per_cta; seg = g.seg;
        group = warp / w;
        slot0 = group * w;   // (0 when a row has the CTA for itself)
        const int rank = cs > 1 ? static_cast<int>(cg::this_cluster().block_rank()) : 0;
        r = cs > 1 ? blockIdx.x / cs : blockIdx.x * rows_per_cta + group;
        part = rank * w + (warp - slot0);
        parts = w * cs;
        per = (parts + 31) >> 5;
        const int nvec = (vocab + 7) / 8;
        lo = min(part * seg, nvec);
        hi = min(lo + seg, nvec);
        nj = (seg + 31) >> 5;
        lv = lo + static_cast<int>(threadIdx.x & 31);
    }
    __device__ __forceinline__ bool has(int j) const { return lv + 32 * j < hi; }
    __device__ __forceinline__ bool holds(int y) const { return (y >> 3) >= lo && (y >> 3) < hi; }   // id y, the warp
    __device__ __forceinline__ int part_of(int y) const { return (y >> 3) / seg; }
    // a value into the same place of every CTA of the row (lane c writes CTA c's copy)
    template <class T>
    __device__ __forceinline__ void post(T *p, const T &v) const {
        const int lane = threadIdx.x & 31;
        if (cs == 1) {
            if (lane == 0) *p = v;
        } else if (lane < cs) {
            *cg::this_cluster().map_shared_rank(p, lane) = v;
        }
    }
    // before a CTA's first post: every CTA of the cluster has started
    __device__ __forceinline__ void arrive_start() const {
        if (cs > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    }
    __device__ __forceinline__ void wait_start() const {
        if (cs > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    }
    __device__ __forceinline__ void sync() const {
        if (cs > 1) {
            asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        } else if (w == 1) {
            __syncwarp();
        } else if (rows_per_cta == 1) {
            __syncthreads();
        } else {
            asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "r"(w * 32) : "memory");
        }
    }
};

__device__ __forceinline__ float warp_max(float x) {
    float m;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(x));
    return m;
}
__device__ __forceinline__ float warp_prefix(float x) {   // inclusive, over ascending lanes
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float up = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += up;
    }
    return x;
}

template <typename LT, int NV>
struct RegVecs {
    Vec8<LT> v[NV];
    __device__ __forceinline__ void load(const RegRow &g, const LT *row, int vocab) {
        const RowVecs<LT> src(row, vocab);
#pragma unroll
        for (int j = 0; j < NV; ++j) v[j] = Vec8<LT>::none();
        if (src.sh == 0) {
#pragma unroll
            for (int j = 0; j < NV; ++j)
                if (g.has(j) && src.whole(g.lv + 32 * j)) v[j] = src.load_aligned(g.lv + 32 * j);
        } else {
#pragma unroll
            for (int j = 0; j < NV; ++j)
                if (g.has(j) && src.whole(g.lv + 32 * j)) v[j] = src.load_shifted(g.lv + 32 * j);
        }
        if (g.lo < src.f0 || g.hi > src.f1) {   // the vectors at the edges of the row
#pragma unroll
            for (int j = 0; j < NV; ++j)
                if (g.has(j) && !src.whole(g.lv + 32 * j)) v[j] = src.load_slow(g.lv + 32 * j);
        }
    }
    __device__ __forceinline__ void drop(const RegRow &g, int y) {   // id y becomes -inf
        if (!g.holds(y)) return;
#pragma unroll
        for (int j = 0; j < NV; ++j)
            if (g.lv + 32 * j == (y >> 3)) v[j].drop(y & 7);
    }
};

// Values that a pass derives from the registers (unpacked logits, exponentials) are made again by the next one: kept,
// they would take more registers than there are.
template <int NV>
__device__ __forceinline__ void forget(RegVecs<__nv_bfloat16, NV> &x) {
#pragma unroll
    for (int j = 0; j < NV; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) asm volatile("" : "+r"(x.v[j].w[i]));
}
template <int NV>
__device__ __forceinline__ void forget(RegVecs<float, NV> &x) {
#pragma unroll
    for (int j = 0; j < NV; ++j)
#pragma unroll
        for (int i = 0; i < 8; ++i) asm volatile("" : "+f"(x.v[j].f[i]));
}

// ---- pass A of a part: maximum, sum of exponentials, (argmax and the sum without it) ----------------
// Both rows of a pair go through the same arithmetic with pinned roundings: equal rows give equal bits.
struct PartStat { float ml, s, sx; int idx; };

template <bool ARG, typename LT, int NV>
__device__ __forceinline__ PartStat part_stat(const RegRow &g, const RegVecs<LT, NV> &x, const LT *row, int vocab, float k) {
    const int lane = threadIdx.x & 31;
    auto m2 = x.v[0].packed_max();
#pragma unroll
    for (int j = 1; j < NV; ++j)
        if (j < g.nj) m2 = Vec8<LT>::max_of(m2, x.v[j].packed_max());
    const float m = Vec8<LT>::max_value(m2);
    PartStat o;
    o.ml = warp_max(m);
    const float c = shift_of(o.ml, k);
    const F2 k2 = f2_make(k, k), nc2 = f2_make(-c, -c);
    float vs[NV], mine = 0.f;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        vs[j] = 0.f;
        if (j < g.nj)
            vs[j] = f2_sum(f2_add(f2_add(f2_exp(x.v[j].pair(0), k2, nc2), f2_exp(x.v[j].pair(1), k2, nc2)),
                                  f2_add(f2_exp(x.v[j].pair(2), k2, nc2), f2_exp(x.v[j].pair(3), k2, nc2))));
        mine += vs[j];
    }
    o.s = warp_sum(mine);
    o.sx = 0.f;
    o.idx = 0x7fffffff;
    if (ARG && o.ml > neg_inf()) {
        // the lowest vector that holds the maximum, its ids over the lanes
        int jm = NV;
#pragma unroll
        for (int j = NV - 1; j >= 0; --j)
            if (j < g.nj && x.v[j].max() == o.ml) jm = j;
        const int at = __reduce_min_sync(kFull, jm * 32 + lane);   // (jm < NV in some lane)
        const int y = (g.lo + at) * 8 + lane;
        const float l = lane < 8 && y < vocab ? load_one<LT>(row, y) : neg_inf();
        const int first = __ffs(__ballot_sync(kFull, lane < 8 && l == o.ml)) - 1;
        o.idx = (g.lo + at) * 8 + first;
        float rest = lane == first ? 0.f : ex2(__fmaf_rn(l, k, -c));   // that vector without it
        rest = warp_sum(rest);
        float other = 0.f;
#pragma unroll
        for (int j = 0; j < NV; ++j) other += lane == (at & 31) && j == (at >> 5) ? rest : vs[j];
        o.sx = warp_sum(other);
    }
    return o;
}

// ---- row values from the parts' records -------------------------------------------------------------
struct RegStat { float ml, C, Z, sx, own; int idx; };
// One value per part: lane l holds those of the parts l * per, l * per + 1, ...
struct PerPart {
    float m[kRegPer];
    __device__ __forceinline__ void set(const RegRow &g, int s, float v) {
        s -= static_cast<int>(threadIdx.x & 31) * g.per;
#pragma unroll
        for (int i = 0; i < kRegPer; ++i)
            if (i < g.per && s == i) m[i] = v;
    }
    __device__ __forceinline__ void add(const RegRow &g, int s, float v) {
        s -= static_cast<int>(threadIdx.x & 31) * g.per;
#pragma unroll
        for (int i = 0; i < kRegPer; ++i)
            if (i < g.per && s == i) m[i] += v;
    }
};

// `floor_ml`: a logit that the row's maximum is not below (ids left out of the parts); -inf if none.
// MASS: also the parts' masses on the row's scale, for a draw: 0 for a part whose exponentials are all below the smallest
// normal number there, 0, so that a picked part has an id to give.
template <bool ARG, bool MASS, class REC>
__device__ __forceinline__ RegStat merge_parts(const RegRow &g, const REC *rec, float k, float floor_ml, PerPart *mass) {
    const int lane = threadIdx.x & 31;
    RegStat o;
    o.idx = 0x7fffffff;
    o.sx = 0.f;
    if (g.parts == 1) {   // the row is this warp's own: nothing to merge
        const REC a = rec[g.slot0];
        o.ml = fmaxf(a.x, floor_ml);
        o.C = shift_of(o.ml, k);
        const float f = rescale(a.x, shift_of(a.x, k), o.C);
        o.Z = __fmul_rn(a.y, f);
        if constexpr (ARG) { o.sx = a.z; o.idx = __float_as_int(a.w); }
        if (MASS) {
#pragma unroll
            for (int i = 0; i < kRegPer; ++i) mass->m[i] = i == 0 && lane == 0 ? o.Z : 0.f;
        }
        o.own = own_term(o.ml, k);
        return o;
    }
    REC a[kRegPer];
    float ml = floor_ml;
#pragma unroll
    for (int i = 0; i < kRegPer; ++i) {
        a[i] = REC{};
        a[i].x = neg_inf();
        if (i < g.per && lane * g.per + i < g.parts) a[i] = rec[g.slot0 + lane * g.per + i];
        ml = fmaxf(ml, a[i].x);
    }
    o.ml = warp_max(ml);
    o.C = shift_of(o.ml, k);
    if constexpr (ARG) {
        int idx = 0x7fffffff;
#pragma unroll
        for (int i = 0; i < kRegPer; ++i)
            if (a[i].x == o.ml) idx = min(idx, __float_as_int(a[i].w));
        o.idx = __reduce_min_sync(kFull, idx);
    }
    float z = 0.f, zx = 0.f;
#pragma unroll
    for (int i = 0; i < kRegPer; ++i) {
        if (MASS) mass->m[i] = 0.f;
        if (i < g.per) {
            const float f = rescale(a[i].x, shift_of(a[i].x, k), o.C);
            const float m = __fmul_rn(a[i].y, f);
            z = __fadd_rn(z, m);
            if (MASS) mass->m[i] = ex2(__fmaf_rn(a[i].x, k, -o.C)) > 0.f ? m : 0.f;
            if constexpr (ARG)
                zx = __fadd_rn(zx, (a[i].x == o.ml && __float_as_int(a[i].w) == o.idx) ? __fmul_rn(a[i].z, f) : m);
        }
    }
    o.Z = warp_sum(z);
    if (ARG) o.sx = warp_sum(zx);
    o.own = own_term(o.ml, k);
    return o;
}

// Pick the part that holds the target u * total of an inverse-CDF draw over the parts' masses.
// Returns the part (-1: no mass) and the target within it; the same in every warp.
__device__ __forceinline__ int pick_part_of(const RegRow &g, const PerPart &mass, float u, float &t_in) {
    t_in = 0.f;
    if (g.parts == 1) {
        const float m = __shfl_sync(kFull, mass.m[0], 0);
        t_in = u * m;
        return m > 0.f ? 0 : -1;
    }
    static_assert(kRegPer == 4, "a lane's masses");
    const int L = pair_pick((mass.m[0] + mass.m[1]) + (mass.m[2] + mass.m[3]), u, t_in);
    if (L < 0 || g.per == 1) return L;
    // the part within the lane's
    float run = 0.f, base = 0.f;
    int at = 0;
    bool found = false;
#pragma unroll
    for (int i = 0; i < kRegPer; ++i) {
        if (mass.m[i] > 0.f && !found) {
            at = i; base = run;
            found = run + mass.m[i] > t_in;
        }
        run += mass.m[i];
    }
    t_in -= __shfl_sync(kFull, base, L);
    return L * g.per + __shfl_sync(kFull, at, L);
}

// The sums of a pass from the parts' records; the third one's parts are kept for a draw.
__device__ __forceinline__ float4 sum_parts(const RegRow &g, const float4 *rec, PerPart &third) {
    const int lane = threadIdx.x & 31;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (g.parts == 1) {
        s = rec[g.slot0];
#pragma unroll
        for (int i = 0; i < kRegPer; ++i) third.m[i] = i == 0 && lane == 0 ? s.z : 0.f;
        return s;
    }
#pragma unroll
    for (int i = 0; i < kRegPer; ++i) {
        third.m[i] = 0.f;
        if (i < g.per && lane * g.per + i < g.parts) {
            const float4 a = rec[g.slot0 + lane * g.per + i];
            s.x += a.x; s.y += a.y; s.z += a.z;
            third.m[i] = a.z;
        }
    }
    s.x = warp_sum(s.x); s.y = warp_sum(s.y); s.z = warp_sum(s.z);
    return s;
}

// The draw inside a part, by its warp: vec(j) = what this lane's j-th vector weighs (registers), weight(y) the weight of
// id y (memory).  Lowest id whose inclusive prefix exceeds t; the last id with mass of the picked vector when rounding
// leaves none; -1: no mass.
template <int NV, class VF, class WF>
__device__ __forceinline__ int draw_in_part(const RegRow &g, int vocab, VF vec, WF weight, float t) {
    const int lane = threadIdx.x & 31;
    float s[NV], tot[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) s[j] = j < g.nj ? vec(j) : 0.f;
#pragma unroll
    for (int j = 0; j < NV; ++j) tot[j] = warp_sum(s[j]);
    float run = 0.f, base = 0.f, mine = 0.f;
    int row = -1;
    bool found = false;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        if (tot[j] > 0.f && !found) {
            row = j; base = run; mine = s[j];
            found = run + tot[j] > t;
        }
        run += tot[j];
    }
    if (row < 0) return -1;
    t -= base;
    const float incl = warp_prefix(mine);
    const unsigned pos = __ballot_sync(kFull, mine > 0.f), hit = __ballot_sync(kFull, mine > 0.f && incl > t);
    const int L = hit ? __ffs(hit) - 1 : 31 - __clz(pos);
    t = __shfl_sync(kFull, t - (incl - mine), L);
    const int y = (g.lo + row * 32 + L) * 8 + lane;
    const float w = lane < 8 && y < vocab ? weight(y) : 0.f;
    const float inc = warp_prefix(w);
    const unsigned p2 = __ballot_sync(kFull, w > 0.f), h2 = __ballot_sync(kFull, w > 0.f && inc > t);
    if (!p2) return -1;
    return y - lane + (h2 ? __ffs(h2) - 1 : 31 - __clz(p2));
}

// What a vector of a row weighs: its exponentials on the row's scale.
template <typename LT>
__device__ __forceinline__ float vec_mass(const Vec8<LT> &v, F2 k2, F2 nc2) {
    return f2_sum(f2_add(f2_add(f2_exp(v.pair(0), k2, nc2), f2_exp(v.pair(1), k2, nc2)),
                         f2_add(f2_exp(v.pair(2), k2, nc2), f2_exp(v.pair(3), k2, nc2))));
}

// ------------------------------------------------------------------------------------------------
// Draft step (Section 4 / Algorithm 3 for SpecHub; Algorithm 1 for RRS, RRSw with k drafts).
// KK: drafts per node when known at compile time (2), else 0.
// ------------------------------------------------------------------------------------------------
template <typename LT, int NV, int KK>
__global__ void __launch_bounds__(kRegThreads) reg_draft_kernel(KaryArgs A, int method, unsigned rows, RegGeo geo) {
    __shared__ RegShared sh;
    pdl_begin();
    const RowArgs &a = A.r;
    const RegRow g(geo, a.vocab);
    if (g.r >= rows) return;
    g.arrive_start();
    const int lane = threadIdx.x & 31, K = KK ? KK : A.k;
    const long long r = g.r;
    const unsigned b = g.r / static_cast<unsigned>(a.nodes), n = g.r - b * static_cast<unsigned>(a.nodes);
    const LT *rowq = static_cast<const LT *>(a.draft) + b * a.stride_seq + n * a.stride_node;
    RegVecs<LT, NV> q;
    q.load(g, rowq, a.vocab);
    const float k = kLog2e / temperature_of(a, b);
    const float *un = a.uniforms + r * (2 * K + 1);
    const bool lead = g.part == 0 && lane == 0;   // writes what no draw decides

    const PartStat ps = part_stat<true>(g, q, rowq, a.vocab, k);
    g.wait_start();
    g.post(&sh.q[g.slot0 + g.part], make_float4(ps.ml, ps.s, ps.sx, __int_as_float(ps.idx)));
    g.sync();
    PerPart mass;   // the parts' masses, ids drawn so far left out where the draws ask for it
    const RegStat Q = merge_parts<true, true>(g, sh.q, k, neg_inf(), &mass);
    const unsigned mark = a.draft_stats_out && A.keep_stats == kMarkedStats && g.part == 0 ? row_mark(rowq, a.vocab) : 0;
    if (lead && a.draft_stats_out) {
        DraftStat ds = {};
        if (A.keep_stats) { ds.ml = Q.ml; ds.sx = Q.sx; ds.idx = Q.idx; ds.tag = stat_tag(k, mark); }
        static_cast<DraftStat *>(a.draft_stats_out)[r] = ds;
    }
    if (!(Q.ml > neg_inf()) || !finite_pos(Q.Z) || !(Q.ml < -neg_inf())) {
        if (lead) {
            for (int i = 0; i < K; ++i) a.draft_tokens_out[K * r + i] = -1;
            if (a.hub) a.hub[r] = -1;
            if (a.draft_prob) { a.draft_prob[2 * r] = 0.f; a.draft_prob[2 * r + 1] = 0.f; }
            if (a.status) a.status[r] = SPECHUB_ST_NONFINITE;
        }
        return;
    }
    forget(q);
    uint32_t st = 0;
    const F2 k2 = f2_make(k, k), nc2 = f2_make(-Q.C, -Q.C);
    auto vec = [&](int j) { return vec_mass(q.v[j], k2, nc2); };
    auto expo = [&](int y) { return ex2(__fmaf_rn(load_one<LT>(rowq, y), k, -Q.C)); };
    auto drawn = [&](int i) { return __float_as_int(sh.drawn[i][g.group].x); };
    if (method == kRRS) {   // independent draws: the parts that hold them write them
#pragma unroll 1
        for (int i = 0; i < K; ++i) {
            float t;
            const int s = pick_part_of(g, mass, un[i], t);
            if (s == g.part) {
                const int tok = draw_in_part<NV>(g, a.vocab, vec, expo, t);
                if (lane == 0) a.draft_tokens_out[K * r + i] = tok;
            }
        }
    } else {
        // Draw i leaves out what was drawn before (RRSw), or the hub once it was drawn (SpecHub's second draw): the part
        // that holds a drawn id takes it out of its registers and tells the row the id and its own new mass, summed
        // directly.
        const int draws = method == kSpecHub ? 2 : K;
#pragma unroll 1
        for (int i = 0; i < draws; ++i) {
            float t;
            int known = -2;
            if (method == kSpecHub && i == 1) {
                if (drawn(0) != Q.idx) known = Q.idx;
                else if (!(Q.sx > 0.f)) { known = Q.idx == 0 ? 1 : 0; st |= SPECHUB_ST_DEGENERATE_Q; }
            }
            const int s = known >= 0 ? -1 : pick_part_of(g, mass, un[i], t);
            if (s < 0) {
                if (known < 0) {   // nothing left to draw from: lowest id not drawn yet
                    st |= SPECHUB_ST_DEGENERATE_Q;
                    known = 0;
                    for (bool again = true; again && known < a.vocab;) {
                        again = false;
                        for (int l = 0; l < i; ++l)
                            if (drawn(l) == known) { ++known; again = true; break; }
                    }
                    if (known >= a.vocab) known = 0;
                }
                __syncwarp();
                if (lane == 0) sh.drawn[i][g.group] = make_float2(__int_as_float(known), 0.f);   // (every warp the same)
                __syncwarp();
                continue;
            }
            if (s == g.part) {
                const int tok = draw_in_part<NV>(g, a.vocab, vec, [&](int y) {
                    bool out = false;
                    for (int l = 0; l < i; ++l) out |= drawn(l) == y;
                    return out ? 0.f : expo(y);
                }, t);
                float rest = 0.f;
                if (i + 1 < draws) {
                    q.drop(g, tok);
#pragma unroll
                    for (int j = 0; j < NV; ++j)
                        if (j < g.nj) rest += vec(j);
                    rest = warp_sum(rest);
                }
                g.post(&sh.drawn[i][g.group], make_float2(__int_as_float(tok), rest));
            }
            g.sync();
            mass.set(g, s, sh.drawn[i][g.group].y);
        }
        if (lead)
            for (int i = 0; i < K; ++i) a.draft_tokens_out[K * r + i] = drawn(i);
    }
    if (!lead) return;
    if (a.hub) a.hub[r] = method == kSpecHub ? Q.idx : -1;
    if (a.draft_prob) {
        float prob0 = 0.f, prob1 = 0.f;
        if (method == kSpecHub) {
            prob0 = Q.own / Q.Z;
            if (drawn(0) != Q.idx) prob1 = expo(drawn(0)) / Q.Z;
            else if (Q.sx > 0.f) prob1 = prob0 * expo(drawn(1)) / Q.sx;
        }
        a.draft_prob[2 * r] = prob0;
        a.draft_prob[2 * r + 1] = prob1;
    }
    if (a.status) a.status[r] = st;
}

// ------------------------------------------------------------------------------------------------
// Verification
// ------------------------------------------------------------------------------------------------
// A draw from p by the row's warps: bonus token of a leaf row, fallback of a rejection without residual mass.  `mass` =
// the parts' masses of p; out[i], i in the set `which`, are ids that were taken out of p's registers (their masses are
// in `mass`).
template <typename LT, int NV>
__device__ __forceinline__ void reg_draw_from_p(const RegRow &g, PerPart mass, const RegVecs<LT, NV> &p, const LT *rowp, int vocab,
                                                float k, float C, const int *out, unsigned which, float u, int32_t *token) {
    float t;
    if (pick_part_of(g, mass, u, t) != g.part) return;
    const F2 k2 = f2_make(k, k), nc2 = f2_make(-C, -C);
    auto weight = [&](int y) { return ex2(__fmaf_rn(load_one<LT>(rowp, y), k, -C)); };
    const int tok = draw_in_part<NV>(g, vocab, [&](int j) {
        float s = vec_mass(p.v[j], k2, nc2);
        for (unsigned m = which; m; m &= m - 1) {
            const int y = out[__ffs(m) - 1];
            if (g.lv + 32 * j == (y >> 3)) s += weight(y);
        }
        return s;
    }, weight, t);
    if ((threadIdx.x & 31) == 0) *token = tok;
}

// The record the draft step left (calls that take draft statistics): the row's own statistics are at hand
// here, so the record is only checked, as in the streaming kernels.
template <typename LT>
__device__ __forceinline__ bool draft_stat_ok(const RowArgs &a, long long r, const LT *rowq, float k) {
    const DraftStat ds = static_cast<const DraftStat *>(a.draft_stats_in)[r];
    bool ok = ds.tag == stat_tag(k);
    if (ok && ds.ml > neg_inf() && ds.ml < -neg_inf() && finite_pos(ds.sx + 1.f))
        ok = ds.idx >= 0 && ds.idx < a.vocab && load_one<LT>(rowq, ds.idx) == ds.ml;
    return ok;
}

template <typename LT, int NV>
__global__ void __launch_bounds__(kRegThreads) reg_verify_spechub_kernel(RowArgs a, unsigned rows, RegGeo geo) {
    __shared__ RegShared sh;
    pdl_begin();
    const RegRow g(geo, a.vocab);
    if (g.r >= rows) return;
    g.arrive_start();
    const int lane = threadIdx.x & 31;
    const long long r = g.r;
    const unsigned b = g.r / static_cast<unsigned>(a.nodes), n = g.r - b * static_cast<unsigned>(a.nodes);
    const LT *rowp = static_cast<const LT *>(a.target) + b * a.stride_seq + n * a.stride_node;
    const LT *rowq = static_cast<const LT *>(a.draft) + b * a.stride_seq + n * a.stride_node;
    const bool leaf = a.node_kind && a.node_kind[n] == SPECHUB_NODE_LEAF;
    RegVecs<LT, NV> p, q;
    p.load(g, rowp, a.vocab);
    if (!leaf) q.load(g, rowq, a.vocab);
    const float k = kLog2e / temperature_of(a, b);
    const float r1 = a.uniforms[r * 5 + 2], r2 = a.uniforms[r * 5 + 3], ures = a.uniforms[r * 5 + 4];
    const float pinf = -neg_inf();
    const bool lead = g.part == 0 && lane == 0;
    int x1 = -1, x2 = -1;
    float lp1 = 0.f, lp2 = 0.f, lq1 = 0.f, lq2 = 0.f;
    bool stat_ok = true;
    if (!leaf) {   // the drafts' logits, fetched while the rows are on their way
        x1 = a.draft_tokens_in[2 * r]; x2 = a.draft_tokens_in[2 * r + 1];
        if (x1 >= 0 && x1 < a.vocab) { lp1 = load_one<LT>(rowp, x1); lq1 = load_one<LT>(rowq, x1); }
        if (x2 >= 0 && x2 < a.vocab) { lp2 = load_one<LT>(rowp, x2); lq2 = load_one<LT>(rowq, x2); }
        if (a.draft_stats_in) stat_ok = draft_stat_ok(a, r, rowq, k);
    }
    NodeResult o;
    o.accept_idx = -1; o.token = -1; o.hub = -1; o.status = 0;
    o.beta[0] = o.beta[1] = 0.f; o.rate[0] = o.rate[1] = o.rate[2] = 0.f;
    bool elsewhere = false;   // the token is written by the warp that draws it
    auto write = [&]() {
        if (!lead) return;
        a.accept_idx[r] = o.accept_idx;
        if (!elsewhere) a.token[r] = o.token;
        if (a.hub) a.hub[r] = o.hub;
        if (a.beta) { a.beta[2 * r] = o.beta[0]; a.beta[2 * r + 1] = o.beta[1]; }
        if (a.rate) { a.rate[3 * r] = o.rate[0]; a.rate[3 * r + 1] = o.rate[1]; a.rate[3 * r + 2] = o.rate[2]; }
        if (a.status) a.status[r] = o.status;
    };

    const PartStat pp = part_stat<false>(g, p, rowp, a.vocab, k);
    PartStat pq = {};
    if (!leaf) pq = part_stat<true>(g, q, rowq, a.vocab, k);
    forget(p);
    forget(q);
    g.wait_start();
    g.post(&sh.p[g.slot0 + g.part], make_float2(pp.ml, pp.s));
    if (!leaf) g.post(&sh.q[g.slot0 + g.part], make_float4(pq.ml, pq.s, pq.sx, __int_as_float(pq.idx)));
    g.sync();
    const RegStat P = merge_parts<false, false>(g, sh.p, k, neg_inf(), nullptr);
    auto draw_from_p = [&](int hub, unsigned taken_out) {
        PerPart mp;
        merge_parts<false, true>(g, sh.p, k, neg_inf(), &mp);
        reg_draw_from_p(g, mp, p, rowp, a.vocab, k, P.C, &hub, taken_out, ures, a.token + r);
        elsewhere = true;
    };
    if (!stat_ok) { o.status = SPECHUB_ST_STATS; write(); return; }
    if (!(P.ml > neg_inf()) || !(P.ml < pinf) || !finite_pos(P.Z)) { o.status = SPECHUB_ST_NONFINITE; write(); return; }
    if (leaf) { draw_from_p(0, 0u); o.rate[2] = 1.f; write(); return; }
    const RegStat Q = merge_parts<true, false>(g, sh.q, k, neg_inf(), nullptr);
    if (!(Q.ml > neg_inf()) || !(Q.ml < pinf) || !finite_pos(Q.Z)) { o.status = SPECHUB_ST_NONFINITE; write(); return; }

    const int hubtok = Q.idx;
    o.hub = hubtok;
    const bool pair_xa = (x2 == hubtok && x1 != hubtok), pair_ax = (x1 == hubtok && x2 != hubtok);
    const int x = pair_xa ? x1 : x2;
    if (!(pair_xa || pair_ax) || x < 0 || x >= a.vocab) { o.status = SPECHUB_ST_TOKEN_RANGE; write(); return; }
    const float invZp = 1.f / P.Z, invZq = 1.f / Q.Z, rho = __fdiv_rn(P.Z, Q.Z);
    const bool degenerate = !(Q.sx > 0.f);
    const float c = degenerate ? 0.f : Q.own / Q.sx, crho = c * rho;
    const float qa = Q.own * invZq, rest = Q.sx * invZq;
    const float px = prob_of(pair_xa ? lp1 : lp2, k, P.C, invZp), qx = prob_of(pair_xa ? lq1 : lq2, k, Q.C, invZq);
    const float pa = prob_of(pair_xa ? lp2 : lp1, k, P.C, invZp);
    const float N1 = pair_xa ? px : fmaxf(__fsub_rn(px, qx), 0.f), D1 = pair_xa ? qx : c * qx;
    if (degenerate) o.status |= SPECHUB_ST_DEGENERATE_Q;
    const bool acc1 = accept_test(r1, N1, D1, o.beta[0], true, o.status);
    if (acc1) { o.accept_idx = pair_xa ? 0 : 1; o.token = x; }
    if (acc1 && !a.beta && !a.rate) { write(); return; }   // no probability asked for: the sums decide nothing

    // transport sums over ids != a (Section 4, Appendix B.1), in units of 1 / Z_p as in the streaming kernels
    p.drop(g, hubtok);
    q.drop(g, hubtok);
    F2 s1 = f2_make(0.f, 0.f), s2 = s1, rr = s1;
    const F2 k2 = f2_make(k, k), ncp2 = f2_make(-P.C, -P.C), ncq2 = f2_make(-Q.C, -Q.C);
    const F2 nrho2 = f2_make(-rho, -rho), ncrho2 = f2_make(-crho, -crho);
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        if (j >= g.nj) continue;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const F2 ep = f2_exp(p.v[j].pair(i), k2, ncp2), eq = f2_exp(q.v[j].pair(i), k2, ncq2);
            const F2 d = f2_fma(nrho2, eq, ep);     // Z_p (p - q)
            const F2 m = f2_max0(d);
            const F2 t = f2_fma(ncrho2, eq, m);     // Z_p (max(p - q, 0) - c q)
            const F2 w = f2_max0(t);
            s1 = f2_add(s1, f2_sub(m, d));          // max(-d, 0) = max(d, 0) - d, exactly
            s2 = f2_add(s2, f2_sub(w, t));
            rr = f2_add(rr, w);
        }
    }
    const float w1 = warp_sum(f2_sum(s1)), w2 = warp_sum(f2_sum(s2)), wr = warp_sum(f2_sum(rr));
    g.post(&sh.sum[0][g.slot0 + g.part], make_float4(w1, w2, wr, 0.f));
    g.sync();
    PerPart mass;
    const float4 sums = sum_parts(g, sh.sum[0], mass);
    const float Rraw = sums.z, S1 = sums.x * invZp, S2 = degenerate ? qa : sums.y * invZp;
    const float hub_left = fmaxf(pa - S2, 0.f);
    o.rate[0] = fmaxf(rest - S1, 0.f) + fminf(pa, S2);
    o.rate[1] = (degenerate ? 0.f : fmaxf(qa - S2, 0.f)) + fminf(hub_left, S1);
    o.rate[2] = Rraw * invZp;
    const bool acc2 = accept_test(r2, pair_xa ? hub_left : pa, pair_xa ? S1 : S2, o.beta[1], !acc1, o.status);
    if (!acc1 && acc2) { o.accept_idx = pair_xa ? 1 : 0; o.token = hubtok; }
    if (!(acc1 || acc2)) {
        if (!(Rraw > 0.f)) {
            o.status |= SPECHUB_ST_ZERO_RESIDUAL;
            draw_from_p(hubtok, 1u);
        } else {
            elsewhere = true;
            float t;
            if (pick_part_of(g, mass, ures, t) == g.part) {
                forget(p);
                forget(q);
                const int tok = draw_in_part<NV>(g, a.vocab, [&](int j) {
                    F2 w = f2_make(0.f, 0.f);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const F2 ep = f2_exp(p.v[j].pair(i), k2, ncp2), eq = f2_exp(q.v[j].pair(i), k2, ncq2);
                        w = f2_add(w, f2_max0(f2_fma(ncrho2, eq, f2_max0(f2_fma(nrho2, eq, ep)))));
                    }
                    return f2_sum(w);
                }, [&](int y) {
                    const float ep = ex2(__fmaf_rn(load_one<LT>(rowp, y), k, -P.C)), eq = ex2(__fmaf_rn(load_one<LT>(rowq, y), k, -Q.C));
                    const float d = __fmaf_rn(-rho, eq, ep);
                    return y == hubtok ? 0.f : fmaxf(__fmaf_rn(-crho, eq, fmaxf(d, 0.f)), 0.f);
                }, t);
                if (lane == 0) a.token[r] = tok;
            }
        }
    }
    write();
}

// Algorithm 1 with k drafts.  With P_0 = p, m_0 = 1, stage j (1 <= j <= k):
//   test j:  accept x_j  iff  r_j m_{j-1} q_j(x_j) < P_{j-1}(x_j);   P_j = max(P_{j-1} - m_{j-1} q_j, 0), m_j = sum P_j
// An id that no stage takes out of q sees the same subtractions one after another, so P_j(y) = max(p(y) - C_j q(y), 0)
// with C_j = sum of the stages' coefficients m g: a stage is one pass over p and q as they are.  Without replacement
// (RRSw) a draft loses its q once drawn, and its C stops growing: the drafts that can be taken out, x_1..x_{k-1}, are
// kept out of the passes and added to every sum as single terms (all terms are positive: nothing cancels).
template <typename LT, int NV, int KK>
__global__ void __launch_bounds__(kRegThreads) reg_verify_rrs_kernel(KaryArgs A, unsigned rows, RegGeo geo) {
    constexpr int MK = KK ? KK : kMaxK;
    __shared__ RegShared sh;
    pdl_begin();
    const RowArgs &a = A.r;
    const RegRow g(geo, a.vocab);
    if (g.r >= rows) return;
    g.arrive_start();
    const int lane = threadIdx.x & 31, K = KK ? KK : A.k;
    const bool wo = A.without_replacement != 0;
    const long long r = g.r;
    const unsigned b = g.r / static_cast<unsigned>(a.nodes), n = g.r - b * static_cast<unsigned>(a.nodes);
    const LT *rowp = static_cast<const LT *>(a.target) + b * a.stride_seq + n * a.stride_node;
    const LT *rowq = static_cast<const LT *>(a.draft) + b * a.stride_seq + n * a.stride_node;
    const bool leaf = a.node_kind && a.node_kind[n] == SPECHUB_NODE_LEAF;
    RegVecs<LT, NV> p, q;
    p.load(g, rowp, a.vocab);
    if (!leaf) q.load(g, rowq, a.vocab);
    const float *un = a.uniforms + r * (2 * K + 1);
    const float ures = un[2 * K], k = kLog2e / temperature_of(a, b), pinf = -neg_inf();
    const bool lead = g.part == 0 && lane == 0;
    int x[MK];
    float lpx[MK], lqx[MK];
    bool in_range = true, stat_ok = true;
    if (!leaf) {
#pragma unroll
        for (int i = 0; i < MK; ++i) {
            x[i] = i < K ? a.draft_tokens_in[K * r + i] : -1;
            const bool ok = x[i] >= 0 && x[i] < a.vocab;
            if (i < K) in_range &= ok;
            lpx[i] = ok ? load_one<LT>(rowp, x[i]) : neg_inf();
            lqx[i] = ok ? load_one<LT>(rowq, x[i]) : neg_inf();
        }
        if (a.draft_stats_in) stat_ok = draft_stat_ok(a, r, rowq, k);
    }
    // single terms: the distinct ids among x_1..x_{k-1} (RRSw)
    bool single[MK];
    float floor_p = neg_inf(), floor_q = neg_inf();
#pragma unroll
    for (int i = 0; i < MK; ++i) {
        single[i] = wo && !leaf && in_range && i + 1 < K;
#pragma unroll
        for (int l = 0; l < i; ++l) single[i] = single[i] && x[l] != x[i];
        if (single[i]) {
            p.drop(g, x[i]);
            q.drop(g, x[i]);
            floor_p = fmaxf(floor_p, lpx[i]);
            floor_q = fmaxf(floor_q, lqx[i]);
        }
    }
    int accept_idx = -1, token = -1;
    uint32_t status = 0;
    float beta[MK], rate[MK + 1];
    bool elsewhere = false;
#pragma unroll
    for (int i = 0; i < MK; ++i) beta[i] = rate[i] = 0.f;
    rate[MK] = 0.f;
    auto write = [&]() {
        if (!lead) return;
        a.accept_idx[r] = accept_idx;
        if (!elsewhere) a.token[r] = token;
        if (a.hub) a.hub[r] = -1;
#pragma unroll
        for (int i = 0; i < MK; ++i) {
            if (a.beta && i < K) a.beta[K * r + i] = beta[i];
            if (a.rate && i < K) a.rate[(K + 1) * r + i] = rate[i];
        }
        if (a.rate) a.rate[(K + 1) * r + K] = rate[MK];   // (rate[K] is kept in the last place)
        if (a.status) a.status[r] = status;
    };
    const PartStat pp = part_stat<false>(g, p, rowp, a.vocab, k);
    PartStat pq = {};
    if (!leaf) pq = part_stat<false>(g, q, rowq, a.vocab, k);
    forget(p);
    forget(q);
    g.wait_start();
    g.post(&sh.p[g.slot0 + g.part], make_float2(pp.ml, pp.s));
    if (!leaf) g.post(&sh.q[g.slot0 + g.part], make_float4(pq.ml, pq.s, 0.f, 0.f));
    g.sync();
    RegStat P = merge_parts<false, false>(g, sh.p, k, floor_p, nullptr);
    RegStat Q = {};
    if (!leaf) Q = merge_parts<false, false>(g, sh.q, k, floor_q, nullptr);
    float ep1[MK], eq1[MK];   // the drafts' exponentials
#pragma unroll
    for (int i = 0; i < MK; ++i) {
        ep1[i] = leaf ? 0.f : ex2(__fmaf_rn(lpx[i], k, -P.C));
        eq1[i] = leaf ? 0.f : ex2(__fmaf_rn(lqx[i], k, -Q.C));
    }
    const float q_rest = Q.Z;   // outside the single terms
#pragma unroll
    for (int i = 0; i < MK; ++i)
        if (single[i]) {
            P.Z = __fadd_rn(P.Z, ep1[i]);
            Q.Z = __fadd_rn(Q.Z, eq1[i]);
        }
    if (!stat_ok) { status = SPECHUB_ST_STATS; write(); return; }
    if (!(P.ml > neg_inf()) || !(P.ml < pinf) || !finite_pos(P.Z)) { status = SPECHUB_ST_NONFINITE; write(); return; }
    if (leaf) {
        PerPart mp;
        merge_parts<false, true>(g, sh.p, k, neg_inf(), &mp);
        reg_draw_from_p(g, mp, p, rowp, a.vocab, k, P.C, x, 0u, ures, a.token + r);
        elsewhere = true;
        rate[MK] = 1.f;
        write();
        return;
    }
    if (!(Q.ml > neg_inf()) || !(Q.ml < pinf) || !finite_pos(Q.Z)) { status = SPECHUB_ST_NONFINITE; write(); return; }
    if (!in_range) { status = SPECHUB_ST_TOKEN_RANGE; write(); return; }
    const float invZp = 1.f / P.Z, invZq = 1.f / Q.Z, rho = __fdiv_rn(P.Z, Q.Z);
    const bool lite = !a.beta && !a.rate;
    const F2 k2 = f2_make(k, k), ncp2 = f2_make(-P.C, -P.C), ncq2 = f2_make(-Q.C, -Q.C);

    float m = 1.f, C = 0.f;   // m_{j-1}, C_{j-1}
    float Cx[MK];             // what C came to for x_i: stops growing once x_i is drawn (RRSw)
    PerPart mass;             // of P_j
    bool accepted = false;
#pragma unroll
    for (int j = 0; j < MK; ++j) {
        if (j >= K) break;
        // mass of q outside the drafts before this stage: positive terms only
        float den = 1.f;
        if (wo && j > 0) {
            den = q_rest;
#pragma unroll
            for (int t = 0; t < MK; ++t) {
                bool in = single[t] && t >= j;
                if (in) den += eq1[t];
            }
            den *= invZq;
        }
        const bool alive = m > 0.f;
        const float coef = m * (wo ? (den > 0.f ? 1.f / den : 0.f) : 1.f);
        const float px = ep1[j] * invZp, qx = eq1[j] * invZq;
        bool gone = false;
        float Cj = C;
#pragma unroll
        for (int l = 0; l < MK; ++l)
            if (l < j && wo && x[l] == x[j] && !gone) { gone = true; Cj = Cx[l]; }
        const float N = fmaxf(__fmaf_rn(-Cj, qx, px), 0.f), D = gone ? 0.f : coef * qx;
        if (alive) beta[j] = D > 0.f ? fminf(N / D, 1.f) : 0.f;
        if (alive && !accepted) {
            if (wo && j > 0 && !(den > 0.f)) status |= SPECHUB_ST_DEGENERATE_Q;
            if (!(D > 0.f)) status |= SPECHUB_ST_ZERO_MASS_DRAFT;
            else if (un[K + j] * D < N) { accepted = true; accept_idx = j; token = x[j]; }
        }
        if (accepted && lite) break;   // no probability asked for: the later stages decide nothing
        C += coef;
        Cx[j] = C;
        const float Crho = C * rho;
        const F2 nc = f2_make(-Crho, -Crho);
        F2 s = f2_make(0.f, 0.f);
        forget(p);
        forget(q);
#pragma unroll
        for (int jj = 0; jj < NV; ++jj) {
            if (jj >= g.nj) continue;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                s = f2_add(s, f2_max0(f2_fma(nc, f2_exp(q.v[jj].pair(i), k2, ncq2), f2_exp(p.v[jj].pair(i), k2, ncp2))));
        }
        g.post(&sh.sum[j & 1][g.slot0 + g.part], make_float4(0.f, 0.f, warp_sum(f2_sum(s)), 0.f));
        g.sync();
        float m_next = sum_parts(g, sh.sum[j & 1], mass).z;
#pragma unroll
        for (int i = 0; i < MK; ++i)
            if (single[i]) {   // (a draft that is still in q has the C of all ids)
                const float v = fmaxf(__fmaf_rn(-(i <= j ? Cx[i] : C) * rho, eq1[i], ep1[i]), 0.f);
                m_next += v;
                mass.add(g, g.part_of(x[i]), v);
            }
        m_next *= invZp;
        rate[j] = alive ? fmaxf(m - m_next, 0.f) : 0.f;
        m = m_next;
    }
    rate[MK] = m;
    if (!accepted) {
        elsewhere = true;
        if (m > 0.f) {
            float t;
            if (pick_part_of(g, mass, ures, t) == g.part) {
                auto weight = [&](int y) {
                    float Cy = C;
#pragma unroll
                    for (int i = 0; i < MK; ++i)
                        if (single[i] && x[i] == y) Cy = Cx[i];
                    const float ep = ex2(__fmaf_rn(load_one<LT>(rowp, y), k, -P.C)), eq = ex2(__fmaf_rn(load_one<LT>(rowq, y), k, -Q.C));
                    return fmaxf(__fmaf_rn(-Cy * rho, eq, ep), 0.f);
                };
                const F2 nc = f2_make(-C * rho, -C * rho);
                forget(p);
                forget(q);
                const int tok = draw_in_part<NV>(g, a.vocab, [&](int j) {
                    F2 w = f2_make(0.f, 0.f);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        w = f2_add(w, f2_max0(f2_fma(nc, f2_exp(q.v[j].pair(i), k2, ncq2), f2_exp(p.v[j].pair(i), k2, ncp2))));
                    float s = f2_sum(w);
#pragma unroll
                    for (int i = 0; i < MK; ++i)
                        if (single[i] && g.lv + 32 * j == (x[i] >> 3)) s += weight(x[i]);
                    return s;
                }, weight, t);
                if (lane == 0) a.token[r] = tok;
            }
        } else {   // (rare) a draw from p
            status |= SPECHUB_ST_ZERO_RESIDUAL;
            PerPart mp;
            merge_parts<false, true>(g, sh.p, k, floor_p, &mp);
            unsigned which = 0;
#pragma unroll
            for (int i = 0; i < MK; ++i)
                if (single[i]) {
                    which |= 1u << i;
                    mp.add(g, g.part_of(x[i]), ep1[i]);
                }
            reg_draw_from_p(g, mp, p, rowp, a.vocab, k, P.C, x, which, ures, a.token + r);
        }
    }
    write();
}

}  // namespace spechub
