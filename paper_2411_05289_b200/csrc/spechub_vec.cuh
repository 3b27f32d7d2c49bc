// Rows of logits as logical vectors of eight ids, whatever the element type and the alignment of the row.
//
// Vector v of a row always holds the ids 8 v .. 8 v + 7, so which thread sums what -- and with it every
// rounding -- depends on the vocabulary size alone, not on where the row happens to start.  Rows on a 16-byte
// boundary are read with one (bf16) or two (fp32) 128-bit loads per vector.  Other rows are read in the aligned
// 16-byte words that cover the vector and shifted into place (by an amount that the whole row shares); the first
// and the last vectors of such a row, whose words reach beyond it, are read element by element.
#pragma once

#include "spechub_common.cuh"

namespace spechub {

// Two fp32 lanes per instruction (fma / add / sub .f32x2): half the issue slots of the scalar forms,
// the same roundings (round to nearest, subnormals kept), so results do not depend on which form is used.
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2_make(float lo, float hi) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_get(F2 a, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
    F2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return d;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    F2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) {
    F2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
__device__ __forceinline__ F2 f2_max0(F2 a) {
    float lo, hi;
    f2_get(a, lo, hi);
    return f2_make(fmaxf(lo, 0.f), fmaxf(hi, 0.f));
}
__device__ __forceinline__ float f2_sum(F2 a) {
    float lo, hi;
    f2_get(a, lo, hi);
    return lo + hi;
}
// the exponentials 2^(k l - c) of a pair of logits
__device__ __forceinline__ F2 f2_exp(F2 l, F2 k2, F2 nc2) {
    const F2 x = f2_fma(l, k2, nc2);
    float x0, x1;
    f2_get(x, x0, x1);
    return f2_make(ex2(x0), ex2(x1));
}

__device__ __forceinline__ unsigned bf2max(unsigned a, unsigned b) {
    unsigned d;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ float bf2_hmax(unsigned m2) {
    return fmaxf(__uint_as_float(m2 << 16), __uint_as_float(m2 & 0xffff0000u));
}
__device__ __forceinline__ void unpack_bf16x8(const uint4 &v, float (&o)[8]) {
    o[0] = __uint_as_float(v.x << 16); o[1] = __uint_as_float(v.x & 0xffff0000u);
    o[2] = __uint_as_float(v.y << 16); o[3] = __uint_as_float(v.y & 0xffff0000u);
    o[4] = __uint_as_float(v.z << 16); o[5] = __uint_as_float(v.z & 0xffff0000u);
    o[6] = __uint_as_float(v.w << 16); o[7] = __uint_as_float(v.w & 0xffff0000u);
}

// Eight consecutive logits.
template <typename LT> struct Vec8;
template <> struct Vec8<__nv_bfloat16> {
    unsigned w[4];
    __device__ __forceinline__ static Vec8 none() { return {{0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u}}; }
    __device__ __forceinline__ F2 pair(int i) const {
        return f2_make(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u));
    }
    __device__ __forceinline__ float get(int i) const {   // (i known at compile time)
        return __uint_as_float((i & 1) ? (w[i >> 1] & 0xffff0000u) : (w[i >> 1] << 16));
    }
    // packed maximum of a thread's vectors
    using Max = unsigned;
    __device__ __forceinline__ static Max max_none() { return 0xff80ff80u; }
    __device__ __forceinline__ Max packed_max() const { return bf2max(bf2max(w[0], w[1]), bf2max(w[2], w[3])); }
    __device__ __forceinline__ static Max max_of(Max a, Max b) { return bf2max(a, b); }
    __device__ __forceinline__ static float max_value(Max m) { return bf2_hmax(m); }
    __device__ __forceinline__ float max() const { return bf2_hmax(packed_max()); }
    __device__ __forceinline__ unsigned differs(const Vec8 &o) const {
        return (w[0] ^ o.w[0]) | (w[1] ^ o.w[1]) | (w[2] ^ o.w[2]) | (w[3] ^ o.w[3]);
    }
    __device__ __forceinline__ void drop(int at) {   // element `at` becomes -inf (by masks: registers are not indexed)
        const unsigned m = (at & 1) ? 0xffff0000u : 0x0000ffffu;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned sel = i == (at >> 1) ? m : 0u;
            w[i] = (w[i] & ~sel) | (0xff80ff80u & sel);
        }
    }
};
template <> struct Vec8<float> {
    float f[8];
    __device__ __forceinline__ static Vec8 none() {
        const float n = neg_inf();
        return {{n, n, n, n, n, n, n, n}};
    }
    __device__ __forceinline__ F2 pair(int i) const { return f2_make(f[2 * i], f[2 * i + 1]); }
    __device__ __forceinline__ float get(int i) const { return f[i]; }
    using Max = float;
    __device__ __forceinline__ float max() const {
        return fmaxf(fmaxf(fmaxf(f[0], f[1]), fmaxf(f[2], f[3])), fmaxf(fmaxf(f[4], f[5]), fmaxf(f[6], f[7])));
    }
    __device__ __forceinline__ static Max max_none() { return neg_inf(); }
    __device__ __forceinline__ Max packed_max() const { return max(); }
    __device__ __forceinline__ static Max max_of(Max a, Max b) { return fmaxf(a, b); }
    __device__ __forceinline__ static float max_value(Max m) { return m; }
    __device__ __forceinline__ unsigned differs(const Vec8 &o) const {
        unsigned d = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) d |= __float_as_uint(f[i]) ^ __float_as_uint(o.f[i]);
        return d;
    }
    __device__ __forceinline__ void drop(int at) {
#pragma unroll
        for (int i = 0; i < 8; ++i) f[i] = i == at ? neg_inf() : f[i];
    }
};

// A row of any alignment.
template <typename LT>
struct RowVecs {
    const LT *row;
    int V;
    int sh;       // elements between the 16-byte boundary at or below the row's start and the row
    int f0, f1;   // vectors [f0, f1) lie in whole 16-byte words of the row

    static constexpr int kPer16 = 16 / sizeof(LT);

    __device__ __forceinline__ RowVecs(const LT *r, int vocab) : row(r), V(vocab) {
        sh = static_cast<int>((reinterpret_cast<uintptr_t>(r) & 15) / sizeof(LT));
        // shifted rows take one word more than the vector has
        f0 = sh ? 1 : 0;
        f1 = sh ? (V + sh - kPer16) / 8 : V / 8;
    }
    __device__ __forceinline__ bool whole(int vi) const { return vi >= f0 && vi < f1; }
    __device__ __forceinline__ Vec8<LT> load_aligned(int vi) const;   // whole(vi), sh == 0
    __device__ __forceinline__ Vec8<LT> load_shifted(int vi) const;   // whole(vi), sh != 0
    __device__ __forceinline__ Vec8<LT> load_slow(int vi) const;      // any vi
};

// (rolled loops: this code is next to every load, and the edges of a row are all that runs it)
template <>
__device__ __forceinline__ Vec8<__nv_bfloat16> RowVecs<__nv_bfloat16>::load_slow(int vi) const {
    const unsigned short *r = reinterpret_cast<const unsigned short *>(row);
    Vec8<__nv_bfloat16> o = Vec8<__nv_bfloat16>::none();
#pragma unroll 1
    for (int y = vi * 8 + 7; y >= vi * 8; --y) {   // elements enter at the bottom, the last one first
        const unsigned e = y < V ? r[y] : 0xff80u;
#pragma unroll
        for (int i = 3; i > 0; --i) o.w[i] = __funnelshift_l(o.w[i - 1], o.w[i], 16);
        o.w[0] = (o.w[0] << 16) | e;
    }
    return o;
}
template <>
__device__ __forceinline__ Vec8<float> RowVecs<float>::load_slow(int vi) const {
    Vec8<float> o = Vec8<float>::none();
#pragma unroll 1
    for (int y = vi * 8 + 7; y >= vi * 8; --y) {
#pragma unroll
        for (int i = 7; i > 0; --i) o.f[i] = o.f[i - 1];
        o.f[0] = y < V ? row[y] : neg_inf();
    }
    return o;
}

template <>
__device__ __forceinline__ Vec8<__nv_bfloat16> RowVecs<__nv_bfloat16>::load_aligned(int vi) const {
    const uint4 a = reinterpret_cast<const uint4 *>(row)[vi];
    return {{a.x, a.y, a.z, a.w}};
}
template <>
__device__ __forceinline__ Vec8<float> RowVecs<float>::load_aligned(int vi) const {
    const float4 *p = reinterpret_cast<const float4 *>(row) + 2 * vi;
    const float4 a = p[0], b = p[1];
    return {{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}

// the vector in the words that cover it
template <int N>
__device__ __forceinline__ Vec8<__nv_bfloat16> shift_words_by(const unsigned (&w)[8], unsigned bits) {
    Vec8<__nv_bfloat16> o;
#pragma unroll
    for (int i = 0; i < 4; ++i) o.w[i] = __funnelshift_r(w[i + N], w[i + N + 1], bits);
    return o;
}
__device__ __forceinline__ Vec8<__nv_bfloat16> shift_words(const uint4 &a, const uint4 &b, int sh) {
    const unsigned w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    const unsigned bits = (sh & 1) * 16;
    switch (sh >> 1) {   // (the same for the whole row)
        case 0: return shift_words_by<0>(w, bits);
        case 1: return shift_words_by<1>(w, bits);
        case 2: return shift_words_by<2>(w, bits);
        default: return shift_words_by<3>(w, bits);
    }
}
__device__ __forceinline__ Vec8<float> shift_words(const float4 &a, const float4 &b, const float4 &c, int sh) {
    const float w[12] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
    Vec8<float> o;
    if (sh == 1) {
#pragma unroll
        for (int i = 0; i < 8; ++i) o.f[i] = w[i + 1];
    } else if (sh == 2) {
#pragma unroll
        for (int i = 0; i < 8; ++i) o.f[i] = w[i + 2];
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) o.f[i] = w[i + 3];
    }
    return o;
}
template <>
__device__ __forceinline__ Vec8<__nv_bfloat16> RowVecs<__nv_bfloat16>::load_shifted(int vi) const {
    const uint4 *p = reinterpret_cast<const uint4 *>(row - sh) + vi;
    return shift_words(p[0], p[1], sh);
}
template <>
__device__ __forceinline__ Vec8<float> RowVecs<float>::load_shifted(int vi) const {
    const float4 *p = reinterpret_cast<const float4 *>(row - sh) + 2 * vi;
    return shift_words(p[0], p[1], p[2], sh);
}

// Loads with an L2 eviction policy (createpolicy).
__device__ __forceinline__ Vec8<__nv_bfloat16> load_hint(const Vec8<__nv_bfloat16> *p, uint64_t pol) {
    Vec8<__nv_bfloat16> v;
    asm volatile("ld.global.L2::cache_hint.v4.b32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ Vec8<float> load_hint(const Vec8<float> *p, uint64_t pol) {
    Vec8<float> v;
    asm volatile("ld.global.L2::cache_hint.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8], %9;"
                 : "=f"(v.f[0]), "=f"(v.f[1]), "=f"(v.f[2]), "=f"(v.f[3]), "=f"(v.f[4]), "=f"(v.f[5]), "=f"(v.f[6]), "=f"(v.f[7])
                 : "l"(p), "l"(pol));
    return v;
}

// A row as the streaming kernels read it.  SHIFT = false: every vector is a whole aligned word (bf16: 16 bytes,
// fp32: 32 bytes); SHIFT = true: any row (see RowVecs).
template <typename LT, bool SHIFT> struct StreamRow;
template <typename LT>
struct StreamRow<LT, false> {
    using Raw = Vec8<LT>;
    static constexpr int kDepth = 8 / sizeof(LT);   // vectors per lane that a pass keeps in flight: 64 bytes
    const LT *row;
    __device__ __forceinline__ StreamRow(const LT *r, int) : row(r) {}
    __device__ __forceinline__ const Vec8<LT> *vec(int vi) const { return reinterpret_cast<const Vec8<LT> *>(row) + vi; }
    __device__ __forceinline__ Vec8<LT> operator[](int vi) const;
    __device__ __forceinline__ Raw fetch(int vi) const { return (*this)[vi]; }
    __device__ __forceinline__ Raw fetch(int vi, uint64_t pol) const { return load_hint(vec(vi), pol); }
    __device__ __forceinline__ Vec8<LT> fix(const Raw &r) const { return r; }
    __device__ __forceinline__ float one(int y) const { return load_one<LT>(row, y); }
};
template <>
__device__ __forceinline__ Vec8<__nv_bfloat16> StreamRow<__nv_bfloat16, false>::operator[](int vi) const {
    const uint4 a = reinterpret_cast<const uint4 *>(row)[vi];
    return {{a.x, a.y, a.z, a.w}};
}
template <>
__device__ __forceinline__ Vec8<float> StreamRow<float, false>::operator[](int vi) const {
    Vec8<float> v;
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v.f[0]), "=f"(v.f[1]), "=f"(v.f[2]), "=f"(v.f[3]), "=f"(v.f[4]), "=f"(v.f[5]), "=f"(v.f[6]), "=f"(v.f[7])
                 : "l"(vec(vi)));
    return v;
}
template <typename LT>
struct StreamRow<LT, true> {
    RowVecs<LT> src;
    __device__ __forceinline__ StreamRow(const LT *r, int vocab) : src(r, vocab) {}
    __device__ __forceinline__ Vec8<LT> operator[](int vi) const {
        if (!src.whole(vi)) return src.load_slow(vi);
        return src.sh == 0 ? src.load_aligned(vi) : src.load_shifted(vi);
    }
    __device__ __forceinline__ float one(int y) const { return load_one<LT>(src.row, y); }
};

// The inside of such a row (whole vectors) for the loops that keep loads in flight: they take the words of a vector
// (fetch) and make the vector of them when it is used (fix).  Shifting is arithmetic on what was loaded: done at
// once, it would wait for the load.
template <typename LT> struct ShiftRaw;
template <> struct ShiftRaw<__nv_bfloat16> { uint4 a, b; };
template <> struct ShiftRaw<float> { float4 a, b, c; };
template <typename LT>
struct AlignedInside {
    using Raw = Vec8<LT>;
    static constexpr int kDepth = 8 / sizeof(LT);
    const RowVecs<LT> &src;
    __device__ __forceinline__ Raw fetch(int vi) const { return src.load_aligned(vi); }
    __device__ __forceinline__ Vec8<LT> fix(const Raw &r) const { return r; }
};
template <typename LT>
struct ShiftedInside {
    using Raw = ShiftRaw<LT>;
    static constexpr int kDepth = 4 / sizeof(LT);   // (two or three words for one vector)
    const RowVecs<LT> &src;
    __device__ __forceinline__ Raw fetch(int vi) const;
    __device__ __forceinline__ Vec8<LT> fix(const Raw &r) const;
};
template <>
__device__ __forceinline__ ShiftRaw<__nv_bfloat16> ShiftedInside<__nv_bfloat16>::fetch(int vi) const {
    const uint4 *p = reinterpret_cast<const uint4 *>(src.row - src.sh) + vi;
    return {p[0], p[1]};
}
template <>
__device__ __forceinline__ Vec8<__nv_bfloat16> ShiftedInside<__nv_bfloat16>::fix(const Raw &r) const {
    return shift_words(r.a, r.b, src.sh);
}
template <>
__device__ __forceinline__ ShiftRaw<float> ShiftedInside<float>::fetch(int vi) const {
    const float4 *p = reinterpret_cast<const float4 *>(src.row - src.sh) + 2 * vi;
    return {p[0], p[1], p[2]};
}
template <>
__device__ __forceinline__ Vec8<float> ShiftedInside<float>::fix(const Raw &r) const {
    return shift_words(r.a, r.b, r.c, src.sh);
}

// A warp's range [lo, hi) of such rows: lane-iteration `it` takes the vectors lo + 32 it + lane; the iterations
// [i0, i1) lie inside the row (or both rows) and need no check per vector.
struct InsideIters { int i0, i1, n; };
template <typename LT>
__device__ __forceinline__ InsideIters inside_iters(const RowVecs<LT> &a, const RowVecs<LT> &b, int lo, int hi) {
    InsideIters r;
    r.n = (hi - lo + 31) >> 5;
    r.i0 = min(r.n, lo < max(a.f0, b.f0) ? 4 : 0);   // (a multiple of every loop's depth)
    r.i1 = max(r.i0, min(r.n, (min(hi, min(a.f1, b.f1)) - lo) >> 5));
    return r;
}

// Loops over the inside of one row, kDepth vectors per lane in flight: the next ones are requested before the
// current ones are used.  begin() is called once, with the first ones requested; f(vector); after(D) is called after
// every D iterations.  Returns the iteration reached.
template <class IN, class BEGIN, class F, class AFTER>
__device__ __forceinline__ int inside_ahead(const IN &row, int v0, int it, int i1, BEGIN begin, F f, AFTER after) {
    constexpr int D = IN::kDepth;
    typename IN::Raw nx[D] = {};
    if (it + D <= i1) {
#pragma unroll
        for (int i = 0; i < D; ++i) nx[i] = row.fetch(v0 + 32 * (it + i));
    }
    begin();
#pragma unroll 1
    for (; it + D <= i1; it += D) {
        typename IN::Raw a[D];
#pragma unroll
        for (int i = 0; i < D; ++i) a[i] = nx[i];
        if (it + 2 * D <= i1) {
#pragma unroll
            for (int i = 0; i < D; ++i) nx[i] = row.fetch(v0 + 32 * (it + D + i));
        }
#pragma unroll
        for (int i = 0; i < D; ++i) f(row.fix(a[i]));
        after(D);
    }
    return it;
}
// ... and over the insides of two rows, the next pair of vectors in flight; STEP = 1 or -1; f(vi, vector, vector)
template <int STEP, class IN, class F>
__device__ __forceinline__ void inside_pairs(const IN &p, const IN &q, int v0, int from, int n, F f) {
    typename IN::Raw np = {}, nq = {};
    int vi = v0 + 32 * from;
    if (n > 0) { np = p.fetch(vi); nq = q.fetch(vi); }
#pragma unroll 1
    for (; n > 0; --n, vi += 32 * STEP) {
        const typename IN::Raw cp = np, cq = nq;
        if (n > 1) { np = p.fetch(vi + 32 * STEP); nq = q.fetch(vi + 32 * STEP); }
        f(vi, p.fix(cp), q.fix(cq));
    }
}
// All vectors of a warp's range of two rows of any alignment, in ascending (STEP = 1) or descending order.
template <int STEP, typename LT, class F>
__device__ __forceinline__ void any_pairs(const StreamRow<LT, true> &p, const StreamRow<LT, true> &q, int lo, int hi, int lane, F f) {
    const InsideIters t = inside_iters(p.src, q.src, lo, hi);
    const int v0 = lo + lane;
    auto slow_run = [&](int from, int n) {
#pragma unroll 1
        for (; n > 0; --n, from += STEP) {
            const int vi = v0 + 32 * from;
            if (vi < hi) f(vi, p[vi], q[vi]);
        }
    };
    const int from = STEP > 0 ? t.i0 : t.i1 - 1, n = t.i1 - t.i0;
    if (STEP > 0) slow_run(0, t.i0);
    else slow_run(t.n - 1, t.n - t.i1);
    if (p.src.sh == 0 && q.src.sh == 0)
        inside_pairs<STEP>(AlignedInside<LT>{p.src}, AlignedInside<LT>{q.src}, v0, from, n, f);
    else if (p.src.sh != 0 && q.src.sh != 0)
        inside_pairs<STEP>(ShiftedInside<LT>{p.src}, ShiftedInside<LT>{q.src}, v0, from, n, f);
    else   // (a shifted row beside one that is not: rows of two unlike buffers)
        slow_run(from, n);
    if (STEP > 0) slow_run(t.i1, t.n - t.i1);
    else slow_run(t.i0 - 1, t.i0);
}

}  // namespace spechub
