// Per-warp rings of bulk copies (cp.async.bulk, global -> shared, completion on an mbarrier): of two bf16 rows, over several
// passes, for streaming verification (WarpRing), and of one, once, for the draft step (RowRing, below).
//
// Two rows: a warp owns a contiguous range [lo, hi) of 16-byte vectors of the target row and of the draft row and
// goes over it once per pass, forwards or backwards.  The passes of a row form one stream of chunks
// (kRingCh vectors per lane of each row): lane 0 keeps kRingStages chunks of that stream in flight, also
// across the boundary between two passes, so that the loads of a pass are under way while the warp still
// reduces the previous one.  The warp that consumes a stage is the one that refills it: no barrier other
// than the stage's own mbarrier and a __syncwarp() is involved, and no other warp is ever waited for.
//
// Vector v of a chunk goes to lane v % 32, as in the kernels that load from global memory directly, so a
// thread sees the same vectors in the same order and every sum keeps its association.
//
// Every wait is bounded: a stage that does not arrive within kRingSpinLimit polls marks the ring as timed
// out, the kernel finishes the row and reports SPECHUB_ST_INTERNAL for it.
#pragma once

#include <cstdint>

#include "spechub_ring_run.h"
#include "spechub_vec.cuh"

namespace spechub {

constexpr int kRingCh = 3;       // vectors per lane, row and stage (measured: 1 / 2 / 3 / 4 -> 1.60 / 1.31 / 1.23 / 1.23 ms)
constexpr int kRingStages = 2;   // (2 / 3 stages at 2 vectors: 1.31 / 1.34 ms)
constexpr int kRingChunkVecs = kRingCh * 32;
constexpr int kRingStageBytes = 2 * kRingChunkVecs * 16;          // target half, draft half
constexpr int kRingWarpBytes = kRingStages * kRingStageBytes;     // 6 KB
constexpr unsigned kRingSpinLimit = 1u << 22;

__device__ __forceinline__ uint32_t ring_saddr(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

struct WarpRing {
    uint32_t data;   // shared-window address of this warp's stages
    uint32_t bars;   // shared-window address of its kRingStages mbarriers
    const uint4 *vp, *vq;
    int lo, hi;
    int nc;          // chunks per pass
    int ng;          // chunks of the whole stream
    int g;           // next chunk of the stream to consume
    int issued;      // chunks requested so far (the same in every lane; lane 0 issues)
    int ipass, ileft, iv0, istep;   // lane 0: the next chunk to request (its pass, chunks left in it, first vector, stride)
    unsigned back;   // bit i: pass i runs from the top of the range down
    bool timed_out;
};

// lane 0: request chunk `R.issued` of the stream
__device__ __forceinline__ void ring_issue(WarpRing &R) {
    const uint32_t bytes = static_cast<uint32_t>(min(kRingChunkVecs, R.hi - R.iv0)) * 16u;
    const uint32_t st = static_cast<uint32_t>(R.issued) & (kRingStages - 1);
    const uint32_t bar = R.bars + 8u * st, dst = R.data + st * kRingStageBytes;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(2u * bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(R.vp + R.iv0), "r"(bytes), "r"(bar) : "memory");
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst + kRingChunkVecs * 16), "l"(R.vq + R.iv0), "r"(bytes), "r"(bar) : "memory");
    // the chunk after this one: the next of this pass, or the first of the next pass
    if (--R.ileft > 0) R.iv0 += R.istep;
    else {
        ++R.ipass;
        R.ileft = R.nc;
        const bool down = (R.back >> R.ipass) & 1u;
        R.istep = down ? -kRingChunkVecs : kRingChunkVecs;
        R.iv0 = down ? R.lo + (R.nc - 1) * kRingChunkVecs : R.lo;
    }
}

// All lanes of the warp.  `data` / `bars`: this warp's kRingWarpBytes (16-byte aligned) and its kRingStages
// mbarriers in shared memory.  `passes` passes over [lo, hi); bit i of `back` makes pass i run backwards.
__device__ __forceinline__ void ring_begin(WarpRing &R, void *data, uint64_t *bars, const uint4 *vp, const uint4 *vq,
                                           int lo, int hi, int passes, unsigned back, int lane) {
    R.data = ring_saddr(data); R.bars = ring_saddr(bars);
    R.vp = vp; R.vq = vq; R.lo = lo; R.hi = hi;
    R.nc = hi > lo ? (hi - lo + kRingChunkVecs - 1) / kRingChunkVecs : 0;
    R.ng = passes * R.nc;
    R.g = 0; R.issued = 0; R.back = back; R.timed_out = false;
    R.ipass = 0; R.ileft = R.nc;
    R.istep = (back & 1u) ? -kRingChunkVecs : kRingChunkVecs;
    R.iv0 = (back & 1u) ? lo + (R.nc - 1) * kRingChunkVecs : lo;
    if (lane == 0) {
#pragma unroll
        for (int s = 0; s < kRingStages; ++s)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(R.bars + 8u * s) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
#pragma unroll
    for (int s = 0; s < kRingStages; ++s) {
        if (R.issued < R.ng) {
            if (lane == 0) ring_issue(R);
            ++R.issued;
        }
    }
}

// wait (bounded) until chunk R.g has arrived
__device__ __forceinline__ void ring_wait(WarpRing &R) {
    static_assert((kRingStages & (kRingStages - 1)) == 0, "stage index by mask");
    const uint32_t bar = R.bars + 8u * (static_cast<uint32_t>(R.g) & (kRingStages - 1));
    const uint32_t parity = (static_cast<uint32_t>(R.g) / kRingStages) & 1u;
    unsigned polls = 0;
    for (;;) {
        uint32_t ok;
        asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) break;
        if (++polls > kRingSpinLimit) { R.timed_out = true; break; }
    }
}

// vector j (0 .. kRingCh - 1) of this lane in chunk R.g: target and draft
__device__ __forceinline__ void ring_load(const WarpRing &R, int j, int lane, Vec8<__nv_bfloat16> &x, Vec8<__nv_bfloat16> &y) {
    const uint32_t a = R.data + (static_cast<uint32_t>(R.g) & (kRingStages - 1)) * kRingStageBytes +
                       static_cast<uint32_t>(j * 32 + lane) * 16u;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(x.w[0]), "=r"(x.w[1]), "=r"(x.w[2]), "=r"(x.w[3]) : "r"(a));
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(y.w[0]), "=r"(y.w[1]), "=r"(y.w[2]), "=r"(y.w[3]) : "r"(a + kRingChunkVecs * 16));
}

// every lane has read chunk R.g: its stage takes the next chunk of the stream
__device__ __forceinline__ void ring_release(WarpRing &R, int lane) {
    __syncwarp();
    if (R.issued < R.ng) {
        if (lane == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            ring_issue(R);
        }
        ++R.issued;
    }
    ++R.g;
}

// before the CTA ends or gives the stream up: no copy may still be on its way into shared memory
__device__ __forceinline__ void ring_drain(WarpRing &R) {
    while (R.g < R.issued) { ring_wait(R); ++R.g; }
    R.ng = R.issued;
}

__device__ __forceinline__ Vec8<__nv_bfloat16> shared_vec(uint32_t at) {
    Vec8<__nv_bfloat16> v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]) : "r"(at) : "memory");
    return v;
}
// ---- one row, once, forwards: the draft step ------------------------------------------------------------
// Chunks of 2 KB (64 bytes per lane), two in flight per warp, in no registers and none of it in L1 (the draft step on 7936
// rows of 128256 ids 351 us from registers, 339 so, 344 with three stages; 10000 rows of 65536: 238, 228, 235; of 32000:
// 148, 141).
constexpr int kRowStages = 2;
constexpr int kRowChunkBytes = 2048;
constexpr int kRowWarpBytes = kRowStages * kRowChunkBytes;

struct RowRing {
    uint32_t data, bars;   // shared-window addresses of this warp's stages and their mbarriers
    const char *src;       // the warp's range
    int bytes;             // of it
};
__device__ __forceinline__ void row_ring_issue(const RowRing &R, int c) {   // (one lane)
    const uint32_t n = static_cast<uint32_t>(min(kRowChunkBytes, R.bytes - c * kRowChunkBytes));
    const uint32_t bar = R.bars + 8u * (c % kRowStages), dst = R.data + (c % kRowStages) * kRowChunkBytes;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(n) : "memory");
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(R.src + static_cast<long long>(c) * kRowChunkBytes), "r"(n), "r"(bar) : "memory");
}
__device__ __forceinline__ void row_ring_begin(RowRing &R, void *data, uint64_t *bars, const void *src, int bytes, int lane) {
    R.data = ring_saddr(data); R.bars = ring_saddr(bars);
    R.src = static_cast<const char *>(src); R.bytes = bytes;
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < kRowStages; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(R.bars + 8u * i) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (int c = 0; c < kRowStages && c * kRowChunkBytes < bytes; ++c) row_ring_issue(R, c);
    }
    __syncwarp();
}
// Did chunk c arrive, within a bounded wait?  The same in every lane.
__device__ __forceinline__ bool row_ring_wait(const RowRing &R, int c) {
    const uint32_t bar = R.bars + 8u * (c % kRowStages), phase = (c / kRowStages) & 1;
    uint32_t done = 0;
    for (unsigned i = 0; i < kRingSpinLimit && !done; ++i)
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(bar), "r"(phase) : "memory");
    return __all_sync(kFull, done);
}
// As row_batches: begin(first vector), one(vector), batch(vi).  False: a chunk did not arrive (within its bounded wait), and
// it and those behind it are in no sum.
template <class BEGIN, class ONE, class BATCH>
__device__ __forceinline__ bool ring_batches(const RowRing &R, int lo, int hi, int lane, BEGIN begin, ONE one, BATCH batch) {
    using V = Vec8<__nv_bfloat16>;
    constexpr int D = kRowChunkBytes / (32 * static_cast<int>(sizeof(V)));
    V x[D];
    return ring_run<kRowStages>(
        (hi - lo + 32 * D - 1) / (32 * D), [&](int c) { return row_ring_wait(R, c); },
        [&](int c) {
            const int v0 = lo + lane + 32 * D * c;
            const uint32_t at = R.data + (c % kRowStages) * kRowChunkBytes + lane * static_cast<int>(sizeof(V));
            if (v0 - lane + 32 * D <= hi) {
#pragma unroll
                for (int d = 0; d < D; ++d) x[d] = shared_vec(at + 32 * d * sizeof(V));
            } else {
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    x[d] = V::none();
                    if (v0 + 32 * d < hi) x[d] = shared_vec(at + 32 * d * sizeof(V));
                }
            }
            __syncwarp();
        },
        [&](int c) {
            if (lane != 0) return;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            row_ring_issue(R, c);
        },
        [&](int c) {
            if (c == 0) begin(x[0]);
#pragma unroll
            for (int d = 0; d < D; ++d) one(x[d]);
            batch(lo + lane + 32 * D * c);
        });
}

}  // namespace spechub
