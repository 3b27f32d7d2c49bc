// Launch functions of the kernel families, one translation unit each (they compile in parallel).  Every
// function enqueues on `s` and returns a SPECHUB_* code.
#pragma once

#include <cuda_runtime.h>

#include "spechub_args.cuh"

namespace spechub {

constexpr int kMaxDevices = 64;

inline int launch_status() { return cudaGetLastError() == cudaSuccess ? SPECHUB_OK : SPECHUB_ERR_LAUNCH; }
// ... of a launch that says itself how it went; a refused one leaves no error behind for a later call to find
inline int launch_status(cudaError_t e) {
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess ? SPECHUB_OK : SPECHUB_ERR_LAUNCH;
}

// One launch: `cs` CTAs per cluster (1: none), as a programmatic dependent of the stream's last kernel.  Only for
// kernels that begin with pdl_begin().
template <class K, class... Args>
int launch_grid(K kern, unsigned grid, int threads, int smem, int cs, cudaStream_t s, const Args &...args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cs; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = cs > 1 ? 2 : 1;
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    return launch_status(cudaLaunchKernelEx(&cfg, kern, args...));
}

// Raise a kernel's dynamic shared memory limit once per device.  `configured`: one flag per device, kept by
// the caller (one array per kernel).
int allow_smem(const void *kern, int bytes, bool *configured);

int launch_walk(const WalkKArgs &w, int n, cudaStream_t s);   // the first n

// Rows held in registers.  reg_plan: false if the row does not fit, or if the streaming kernels are the faster
// ones for so many rows.
struct RegPlan { int nv, w, cs, rows_per_cta, seg; };
bool reg_plan(bool verify, int dtype, int k, int vocab, long long rows, RegPlan *out);
int launch_reg_draft(const RegPlan &pl, int dtype, const KaryArgs &a, int method, unsigned rows, cudaStream_t s);
int launch_reg_verify(const RegPlan &pl, int dtype, const KaryArgs &a, int method, unsigned rows, cudaStream_t s);

// Streaming kernels.  How the rows are read: in whole aligned words (bf16: rows on 16-byte boundaries, fp32: on
// 32-byte boundaries, vocab % 8 == 0), or shifted into place (any row).
enum StreamFormat { kBf16, kBf16Shift, kF32, kF32Shift };
int launch_lean_draft(int format, int method, int cs, const RowArgs &a, bool keep_stats, unsigned rows, cudaStream_t s);
int launch_lean_leaf(int format, const RowArgs &a, int k, const NodeOutPtrs *outs, int n_out, unsigned rows, cudaStream_t s);
// cs = CTAs per row asked for (0: the library's choice; other than 0 and 1: kBf16 only)
int launch_lean_verify_spechub(int format, int cs, const RowArgs &a, unsigned rows, cudaStream_t s);
int launch_lean_verify_rrs(int format, int cs, const RowArgs &a, unsigned rows, cudaStream_t s);
int launch_lean_verify_rrsw(int format, int cs, const RowArgs &a, unsigned rows, cudaStream_t s);
// more than two drafts per node
int launch_kary_draft(int format, const KaryArgs &a, unsigned rows, cudaStream_t s);
int launch_kary_verify(int format, const KaryArgs &a, unsigned rows, cudaStream_t s);
int launch_fused_draft(const FusedArgs &f, int32_t *hub, float *draft_prob, unsigned rows, cudaStream_t s);
int launch_fused_verify(const FusedArgs &f, unsigned rows, cudaStream_t s);

// exponentials resident on chip.  A row is spread over `cs` CTAs; every lane keeps `nb` batches of vectors.
struct ResShape { int cs, nb; };
bool resident_fits(int vocab, ResShape *out);
int launch_resident(int mask, ResShape sh, const FusedArgs &f, unsigned rows, cudaStream_t s);
int launch_resident_kary(ResShape sh, const KaryArgs &ka, unsigned rows, cudaStream_t s);

// vocabulary-sharded phases
enum ShardPhase { kPhaseStats, kPhaseSums, kPhaseDecide, kPhaseDraft, kPhaseRrsSums, kPhaseRrsDecide, kPhaseRrsDraft };
int launch_shard_phase(int phase, int dtype, bool aligned, int th, const ShardArgs &a, unsigned rows, cudaStream_t s);
int launch_shard_draft_finish(bool rrs, const ShardArgs &a, cudaStream_t s);

}  // namespace spechub
