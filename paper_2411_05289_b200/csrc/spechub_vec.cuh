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
    __device__ __forceinline__ Vec8<LT> load_edge(int vi) const;      // any vi, by a call
};

// Elements y0 .. y0 + 7 (bf16) or y0 .. y0 + 3 (fp32) of a row, -inf outside it, all requested together.
__device__ __forceinline__ uint4 edge_inline(const unsigned short *row, int y0, int V) {
    unsigned e[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) e[i] = static_cast<unsigned>(y0 + i) < static_cast<unsigned>(V) ? row[y0 + i] : 0xff80u;
    return make_uint4(e[0] | e[1] << 16, e[2] | e[3] << 16, e[4] | e[5] << 16, e[6] | e[7] << 16);
}
__device__ __forceinline__ float4 edge_inline(const float *row, int y0, int V) {
    float e[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) e[i] = static_cast<unsigned>(y0 + i) < static_cast<unsigned>(V) ? row[y0 + i] : neg_inf();
    return make_float4(e[0], e[1], e[2], e[3]);
}
// ... as a call: in the streaming kernels this is next to every load, and the edges of a row are all that runs it
static __device__ __noinline__ uint4 edge_word(const unsigned short *row, int y0, int V) { return edge_inline(row, y0, V); }
static __device__ __noinline__ float4 edge_word(const float *row, int y0, int V) { return edge_inline(row, y0, V); }
template <>
__device__ __forceinline__ Vec8<__nv_bfloat16> RowVecs<__nv_bfloat16>::load_slow(int vi) const {
    const uint4 a = edge_inline(reinterpret_cast<const unsigned short *>(row), vi * 8, V);
    return {{a.x, a.y, a.z, a.w}};
}
template <>
__device__ __forceinline__ Vec8<float> RowVecs<float>::load_slow(int vi) const {
    const float4 a = edge_inline(row, vi * 8, V), b = edge_inline(row, vi * 8 + 4, V);
    return {{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
}
template <>
__device__ __forceinline__ Vec8<__nv_bfloat16> RowVecs<__nv_bfloat16>::load_edge(int vi) const {
    const uint4 a = edge_word(reinterpret_cast<const unsigned short *>(row), vi * 8, V);
    return {{a.x, a.y, a.z, a.w}};
}
template <>
__device__ __forceinline__ Vec8<float> RowVecs<float>::load_edge(int vi) const {
    const float4 a = edge_word(row, vi * 8, V), b = edge_word(row, vi * 8 + 4, V);
    return {{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w}};
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
    using Elem = LT;
    const LT *row;
    __device__ __forceinline__ StreamRow(const LT *r, int) : row(r) {}
    __device__ __forceinline__ const Vec8<LT> *vec(int vi) const { return reinterpret_cast<const Vec8<LT> *>(row) + vi; }
    __device__ __forceinline__ Vec8<LT> operator[](int vi) const;
    __device__ __forceinline__ Vec8<LT> fetch(int vi) const { return (*this)[vi]; }
    __device__ __forceinline__ Vec8<LT> fetch(int vi, uint64_t pol) const { return load_hint(vec(vi), pol); }
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
    using Elem = LT;
    RowVecs<LT> src;
    __device__ __forceinline__ StreamRow(const LT *r, int vocab) : src(r, vocab) {}
    __device__ __forceinline__ Vec8<LT> operator[](int vi) const {
        if (!src.whole(vi)) return src.load_edge(vi);
        return src.sh == 0 ? src.load_aligned(vi) : src.load_shifted(vi);
    }
    __device__ __forceinline__ float one(int y) const { return load_one<LT>(src.row, y); }
};

// A row as the loops below take it: plain(vi) where all lanes' vectors are whole, checked(vi, hi) anywhere (-inf from
// vector hi on).  Shifted rows are kept as the words of a vector (Raw) and made into the vector when it is used (fix):
// shifting is arithmetic on what was loaded; done at once, it would wait for the load.
template <typename LT>
struct WholeIn {
    using Raw = Vec8<LT>;
    static constexpr int kDepth = 8 / sizeof(LT);   // vectors per lane that a pass over one row keeps in flight: 64 bytes
    const StreamRow<LT, false> &row;
    __device__ __forceinline__ Raw plain(int vi) const { return row[vi]; }
    __device__ __forceinline__ Raw checked(int vi, int hi) const {
        Raw v = Raw::none();
        if (vi < hi) v = plain(vi);
        return v;
    }
    __device__ __forceinline__ Vec8<LT> fix(const Raw &r) const { return r; }
};
template <typename LT>
struct HintedIn {   // ... with an L2 eviction policy
    using Raw = Vec8<LT>;
    static constexpr int kDepth = 8 / sizeof(LT);
    const StreamRow<LT, false> &row;
    uint64_t pol;
    __device__ __forceinline__ Raw plain(int vi) const { return row.fetch(vi, pol); }
    __device__ __forceinline__ Raw checked(int vi, int hi) const {
        Raw v = Raw::none();
        if (vi < hi) v = plain(vi);
        return v;
    }
    __device__ __forceinline__ Vec8<LT> fix(const Raw &r) const { return r; }
};
template <typename LT>
struct AlignedIn {   // a row on a 16-byte boundary, of any length
    using Raw = Vec8<LT>;
    static constexpr int kDepth = 8 / sizeof(LT);
    const RowVecs<LT> &src;
    __device__ __forceinline__ Raw plain(int vi) const { return src.load_aligned(vi); }
    __device__ __forceinline__ Raw checked(int vi, int hi) const {
        Raw v = Raw::none();
        if (vi < hi) v = src.whole(vi) ? src.load_aligned(vi) : src.load_edge(vi);
        return v;
    }
    __device__ __forceinline__ Vec8<LT> fix(const Raw &r) const { return r; }
};
template <typename LT> struct ShiftRaw;
template <> struct ShiftRaw<__nv_bfloat16> { uint4 a, b; };
template <> struct ShiftRaw<float> { float4 a, b, c; };
template <typename LT>
struct ShiftedIn {   // any other row
    using Raw = ShiftRaw<LT>;
    static constexpr int kDepth = 4 / sizeof(LT);   // (two or three words for one vector)
    const RowVecs<LT> &src;
    __device__ __forceinline__ Raw plain(int vi) const;
    __device__ __forceinline__ Raw checked(int vi, int hi) const;
    __device__ __forceinline__ Vec8<LT> fix(const Raw &r) const;
};
template <>
__device__ __forceinline__ ShiftRaw<__nv_bfloat16> ShiftedIn<__nv_bfloat16>::plain(int vi) const {
    const uint4 *p = reinterpret_cast<const uint4 *>(src.row - src.sh) + vi;
    return {p[0], p[1]};
}
template <>
__device__ __forceinline__ ShiftRaw<__nv_bfloat16> ShiftedIn<__nv_bfloat16>::checked(int vi, int hi) const {
    const uint4 n = make_uint4(0xff80ff80u, 0xff80ff80u, 0xff80ff80u, 0xff80ff80u);
    ShiftRaw<__nv_bfloat16> r = {n, n};
    if (vi < hi) {
        if (src.whole(vi)) {
            r = plain(vi);
        } else {
            const unsigned short *e = reinterpret_cast<const unsigned short *>(src.row);
            r.a = edge_word(e, vi * 8 - src.sh, src.V);
            r.b = edge_word(e, vi * 8 - src.sh + 8, src.V);
        }
    }
    return r;
}
template <>
__device__ __forceinline__ Vec8<__nv_bfloat16> ShiftedIn<__nv_bfloat16>::fix(const Raw &r) const {
    return shift_words(r.a, r.b, src.sh);
}
template <>
__device__ __forceinline__ ShiftRaw<float> ShiftedIn<float>::plain(int vi) const {
    const float4 *p = reinterpret_cast<const float4 *>(src.row - src.sh) + 2 * vi;
    return {p[0], p[1], p[2]};
}
template <>
__device__ __forceinline__ ShiftRaw<float> ShiftedIn<float>::checked(int vi, int hi) const {
    const float4 n = make_float4(neg_inf(), neg_inf(), neg_inf(), neg_inf());
    ShiftRaw<float> r = {n, n, n};
    if (vi < hi) {
        if (src.whole(vi)) {
            r = plain(vi);
        } else {
            r.a = edge_word(src.row, vi * 8 - src.sh, src.V);
            r.b = edge_word(src.row, vi * 8 - src.sh + 4, src.V);
            r.c = edge_word(src.row, vi * 8 - src.sh + 8, src.V);
        }
    }
    return r;
}
template <>
__device__ __forceinline__ Vec8<float> ShiftedIn<float>::fix(const Raw &r) const {
    return shift_words(r.a, r.b, r.c, src.sh);
}

// A warp's range [lo, hi) of a row: lane-iteration `it` takes the vectors lo + 32 it + lane; in the iterations [i0, i1)
// every lane has a whole vector.  The same in every lane, as the compiler can see (warp_index).
struct Iters { int i0, i1, n; };
__device__ __forceinline__ int warp_index() { return __shfl_sync(kFull, static_cast<int>(threadIdx.x >> 5), 0); }
__device__ __forceinline__ Iters whole_iters(int lo, int hi) { return {0, (hi - lo) >> 5, (hi - lo + 31) >> 5}; }
template <typename LT>
__device__ __forceinline__ Iters inside_iters(const RowVecs<LT> &a, const RowVecs<LT> &b, int lo, int hi) {
    Iters r;
    r.n = (hi - lo + 31) >> 5;
    r.i0 = min(r.n, lo < max(a.f0, b.f0) ? 1 : 0);
    r.i1 = max(r.i0, min(r.n, (min(hi, min(a.f1, b.f1)) - lo) >> 5));
    return r;
}

// One row, D vectors per lane in flight ahead of the D in use, in two sets of registers that take turns.  (With one set and
// copies, the copies were a tenth of a pass's instructions; with one set and each vector's place taken by the one D further
// on, the loads no longer come in bursts: draft step on 7936 rows of 128256 ids 352 us, 368 so, 360 with copies.)  The last
// vectors of a range, and those at the edges of a row, come with the others (one by one behind the loop they cost up to
// four load round trips per row): lanes that have none take -inf, which adds 0 to every sum.  begin(the lane's first
// vector) is called with the first loads requested, one(vector) for each vector, batch(vi) after D of them, vi the first.
// APART: the first loads are not the loop's (the same loads in the same order; in verification that keeps the passes behind
// this one free of spills, 1010 us and 1029 above, in shifted rows' draft steps it is what spills).
template <int D, bool APART, class IN, class BEGIN, class ONE, class BATCH>
__device__ __forceinline__ void row_batches(const IN &in, int v0, int hi, const Iters &t, BEGIN begin, ONE one, BATCH batch) {
    using Raw = typename IN::Raw;
    auto get = [&](int i, Raw (&x)[D]) {
        if (i >= t.i0 && i + D <= t.i1) {
#pragma unroll
            for (int d = 0; d < D; ++d) x[d] = in.plain(v0 + 32 * (i + d));
        } else {
#pragma unroll
            for (int d = 0; d < D; ++d) x[d] = in.checked(v0 + 32 * (i + d), hi);
        }
    };
    auto use = [&](int i, const Raw (&x)[D]) {
#pragma unroll
        for (int d = 0; d < D; ++d) one(in.fix(x[d]));
        batch(v0 + 32 * i);
    };
    Raw a[D], b[D];
    if constexpr (APART) {
        get(0, a);
        begin(in.fix(a[0]));
#pragma unroll 1
        for (int i = 0; i < t.n; i += 2 * D) {
            if (i + D < t.n) get(i + D, b);
            use(i, a);
            if (i + D >= t.n) break;
            if (i + 2 * D < t.n) get(i + 2 * D, a);
            use(i + D, b);
        }
    } else {
#pragma unroll 1
        for (int i = -D;;) {   // (the first turn only requests)
            if (i + D < t.n) get(i + D, b);
            if (i < 0) {
                if (t.n <= 0) break;
                begin(in.fix(b[0]));
            } else {
                use(i, a);
            }
            if ((i += D) >= t.n) break;
            if (i + D < t.n) get(i + D, a);
            use(i, b);
            if ((i += D) >= t.n) break;
        }
    }
}
// ... with one set of registers, copied behind the request of the next: longer by the copies, shorter in code and in
// registers, and the last batch goes as far as the range does.  (The order of the sums is the same one.)
template <int D, class IN, class BEGIN, class ONE, class BATCH>
__device__ __forceinline__ void row_turns(const IN &in, int v0, int hi, const Iters &t, BEGIN begin, ONE one, BATCH batch) {
    using Raw = typename IN::Raw;
    auto get = [&](int i, Raw (&x)[D]) {
        if (i >= t.i0 && i + D <= t.i1) {
#pragma unroll
            for (int d = 0; d < D; ++d) x[d] = in.plain(v0 + 32 * (i + d));
        } else {
#pragma unroll
            for (int d = 0; d < D; ++d) x[d] = in.checked(v0 + 32 * (i + d), hi);
        }
    };
    if (t.n <= 0) return;
    Raw nx[D];
    get(0, nx);
    begin(in.fix(nx[0]));
#pragma unroll 1
    for (int i = 0; i < t.n; i += D) {
        Raw a[D];
#pragma unroll
        for (int d = 0; d < D; ++d) a[d] = nx[d];
        if (i + D < t.n) get(i + D, nx);
        if (i + D <= t.n) {
#pragma unroll
            for (int d = 0; d < D; ++d) one(in.fix(a[d]));
        } else {
#pragma unroll
            for (int d = 0; d < D - 1; ++d)
                if (i + d < t.n) one(in.fix(a[d]));
        }
        batch(v0 + 32 * i);
    }
}
// Two rows, ascending (STEP = 1) or descending, the next pair of vectors in flight: f(vi, x, y) with the target's and the
// draft's vector.  (Two sets of registers that take turns, the loop's code twice: verification from draft statistics on
// 7936 rows of 128256 ids 1014 -> 1046 us, three drafts 750 -> 829; the next pair's loads behind the exponentials, in the
// registers that held this pair: 1070, 790.)
template <int STEP, class IN, class F>
__device__ __forceinline__ void pair_turns(const IN &p, const IN &q, int v0, int from, int n, F f) {
    typename IN::Raw np = {}, nq = {};
    int vi = v0 + 32 * from;
    if (n > 0) { np = p.plain(vi); nq = q.plain(vi); }
#pragma unroll 1
    for (; n > 0; --n, vi += 32 * STEP) {
        const typename IN::Raw cp = np, cq = nq;
        if (n > 1) { np = p.plain(vi + 32 * STEP); nq = q.plain(vi + 32 * STEP); }
        f(vi, p.fix(cp), q.fix(cq));
    }
}
// All vectors of a warp's range of two rows of any alignment.
template <int STEP, typename LT, class F>
__device__ __forceinline__ void any_pairs(const StreamRow<LT, true> &p, const StreamRow<LT, true> &q, int lo, int hi, int lane, F f) {
    const Iters t = inside_iters(p.src, q.src, lo, hi);
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
        pair_turns<STEP>(AlignedIn<LT>{p.src}, AlignedIn<LT>{q.src}, v0, from, n, f);
    else if (p.src.sh != 0 && q.src.sh != 0)
        pair_turns<STEP>(ShiftedIn<LT>{p.src}, ShiftedIn<LT>{q.src}, v0, from, n, f);
    else   // (a shifted row beside one that is not: rows of two unlike buffers)
        slow_run(from, n);
    if (STEP > 0) slow_run(t.i1, t.n - t.i1);
    else slow_run(t.i0 - 1, t.i0);
}

}  // namespace spechub
