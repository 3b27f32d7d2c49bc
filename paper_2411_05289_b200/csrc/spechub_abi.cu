// C ABI of the library (see include/spechub.h): host-side argument checks and
// kernel launches.  Nothing here allocates or synchronises.
#include <cuda_runtime.h>
#include <math.h>
#include <stdlib.h>

#include <mutex>

#include "spechub.h"
#include "spechub_launch.h"

extern "C" size_t spechub_draft_stats_bytes(const spechub_desc *desc);

namespace {

using namespace spechub;

int check_desc(const spechub_desc *d) {
    if (!d) return SPECHUB_ERR_NULL;
    if (d->struct_size != sizeof(spechub_desc) || d->version != SPECHUB_ABI_VERSION)
        return SPECHUB_ERR_VERSION;
    if (d->batch < 0 || d->nodes < 1 || d->vocab < 2 || d->k < 2 || d->k > SPECHUB_MAX_K || d->levels < 1)
        return SPECHUB_ERR_SHAPE;
    if (d->dtype != SPECHUB_F32 && d->dtype != SPECHUB_BF16) return SPECHUB_ERR_DTYPE;
    if (d->stride_node < d->vocab) return SPECHUB_ERR_STRIDE;
    if (d->nodes > 1 && d->stride_seq < d->stride_node * (int64_t)(d->nodes - 1) + d->vocab)
        return SPECHUB_ERR_STRIDE;
    if (d->nodes == 1 && d->batch > 1 && d->stride_seq < d->vocab) return SPECHUB_ERR_STRIDE;
    if (!d->temperature_per_seq && !(d->temperature > 0.f && isfinite(d->temperature)))
        return SPECHUB_ERR_TEMPERATURE;
    const uint32_t split = d->flags & 7u;
    if ((d->flags & ~15u) != 0 || (split & (split - 1)) != 0) return SPECHUB_ERR_SHAPE;
    if ((d->flags & SPECHUB_FLAG_RESIDENT) && split) return SPECHUB_ERR_SHAPE;
    if ((int64_t)d->batch * d->nodes > 0x7fffffffLL) return SPECHUB_ERR_SHAPE;
    return SPECHUB_OK;
}

// rows whose every start is 16-byte aligned take the 128-bit load path
bool rows_aligned(const spechub_desc *d, const void *base) {
    const int esz = d->dtype == SPECHUB_BF16 ? 2 : 4;
    const int per16 = 16 / esz;
    return (reinterpret_cast<uintptr_t>(base) % 16 == 0) && (d->stride_node % per16 == 0) &&
           (d->stride_seq % per16 == 0);
}

int threads_for(const spechub_desc *d) {
    const int vw = d->dtype == SPECHUB_BF16 ? 8 : 4;
    const int nvec = (d->vocab + vw - 1) / vw;
    if (nvec >= 8192) return 512;
    if (nvec >= 2048) return 256;
    if (nvec >= 128) return 128;
    if (nvec >= 64) return 64;
    return 32;
}

RowArgs base_args(const spechub_desc *d) {
    RowArgs a = {};
    a.temperature_per_seq = d->temperature_per_seq;
    a.node_kind = d->node_kind;
    a.temperature = d->temperature;
    a.nodes = d->nodes;
    a.vocab = d->vocab;
    a.stride_seq = d->stride_seq;
    a.stride_node = d->stride_node;
    return a;
}

// CTAs per row.  With 4 CTAs per SM and 148 SMs, 592/CS rows are between their first and second
// read at any time; at CS = 4 on V = 128256 that fits L2 (DRAM reads drop from 2.0x to 1.0x the
// algorithmic bytes) but the per-CTA fixed work grows 4x, and the two cancel (1.6 vs 1.8 ms).
// 0 = no flag: one CTA per row (the per-CTA fixed work of a split row outweighs the L2 hits), whose shape
// and loads the launches choose.
int lean_split(const spechub_desc *d) {
    if (d->flags & SPECHUB_FLAG_SPLIT_1) return 1;
    if (d->flags & SPECHUB_FLAG_SPLIT_2) return 2;
    if (d->flags & SPECHUB_FLAG_SPLIT_4) return 4;
    return 0;
}

// How the streaming kernels read the rows: in whole aligned words if every row starts on the boundary of a vector
// of eight ids and has no remainder.  (`aligned`: on 16-byte boundaries.)
int stream_format(const spechub_desc *d, bool aligned, const void *base0, const void *base1) {
    if (d->dtype == SPECHUB_BF16) return aligned && d->vocab % 8 == 0 ? kBf16 : kBf16Shift;
    const uintptr_t at = reinterpret_cast<uintptr_t>(base0) | reinterpret_cast<uintptr_t>(base1);
    return at % 32 == 0 && d->stride_node % 8 == 0 && d->stride_seq % 8 == 0 && d->vocab % 8 == 0 ? kF32 : kF32Shift;
}

// Shapes of the kernels that take long bf16 rows in whole words only: split rows, the three-method kernels, rows
// resident on chip.
bool lean_ok(const spechub_desc *d, bool aligned) {
    return d->dtype == SPECHUB_BF16 && aligned && d->vocab % 8 == 0 && d->vocab >= 8192;
}

bool resident_fits(const spechub_desc *d, bool aligned, ResShape *out) {
    return lean_ok(d, aligned) && resident_fits(d->vocab, out);
}
// two drafts per node: on request (SPECHUB_FLAG_RESIDENT)
bool resident_shape(const spechub_desc *d, bool aligned, ResShape *out) {
    return (d->flags & SPECHUB_FLAG_RESIDENT) && resident_fits(d, aligned, out);
}

// Shapes whose draft step leaves records that verification reads (see spechub_draft_sample_stats): rows in whole words from
// 8192 ids, rows of any alignment from 16384.  (Shorter ones would gain too -- 3584 packed rows of 12001 ids, SpecHub step
// 154 -> 141 us, RRSw 167 -> 159 -- but that they leave void records is part of the interface.  The format is the draft rows' in a draft step and both rows' in verification:
// a shape that verification takes records of is one that every draft step leaves some for; of shifted draft rows, records
// that were left for rows in whole words carry no mark and are not taken.)
KeepStats keeps_stats(const spechub_desc *d, int format) {
    const bool words = format == kBf16 || format == kF32;
    if (d->k != 2 || d->flags != 0 || d->vocab < (words ? 8192 : 16384)) return kVoidStats;
    return words ? kPlainStats : kMarkedStats;
}

// Rows held in registers: no flag asks for another kernel.
bool use_reg(bool verify, const spechub_desc *d, bool aligned, long long rows, RegPlan *pl) {
    return (d->flags == 0 || !lean_ok(d, aligned)) && reg_plan(verify, d->dtype, d->k, d->vocab, rows, pl);
}

int draft_common(const spechub_desc *d, const void *draft_logits, const float *uniforms, int method,
                 int32_t *draft_tokens, int32_t *hub, float *draft_prob, uint32_t *status,
                 void *stream, void *draft_stats = nullptr) {
    const int rc = check_desc(d);
    if (rc != SPECHUB_OK) return rc;
    if (d->batch == 0) return SPECHUB_OK;  // nothing to do; pointers are not looked at
    if (!draft_logits || !uniforms || !draft_tokens) return SPECHUB_ERR_NULL;
    if (reinterpret_cast<uintptr_t>(draft_stats) % 16 != 0) return SPECHUB_ERR_STRIDE;
    RowArgs a = base_args(d);
    // Only the shapes of keeps_stats leave statistics; every other kernel leaves records that no verification accepts
    // (all zero), and the verification paths that pair with them do not look at the records.
    a.draft_stats_out = draft_stats;
    a.draft = draft_logits;
    a.uniforms = uniforms;
    a.draft_tokens_out = draft_tokens;
    a.hub = hub;
    a.draft_prob = draft_prob;
    a.status = status;
    const unsigned rows = (unsigned)(d->batch * (int64_t)d->nodes);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bool al = rows_aligned(d, draft_logits);
    const int fmt = stream_format(d, al, draft_logits, nullptr);
    if (d->k > 2 && method == kSpecHub) return SPECHUB_ERR_SHAPE;
    KaryArgs ka;
    ka.r = a; ka.k = d->k; ka.without_replacement = (method == kRRSw); ka.keep_stats = keeps_stats(d, fmt);
    RegPlan pl;
    if (use_reg(false, d, al, rows, &pl)) return launch_reg_draft(pl, d->dtype, ka, method, rows, s);
    if (d->k > 2) return launch_kary_draft(fmt, ka, rows, s);
    return launch_lean_draft(fmt, method, lean_ok(d, al) ? lean_split(d) : 0, a, ka.keep_stats, rows, s);
}

// The walks of n methods over the same trees, in one launch (so = nullptr: none).
int launch_walks(const spechub_desc *d, const spechub_node_out *no, const spechub_seq_out *so, int n, cudaStream_t s) {
    WalkKArgs wk;
    wk.k = d->k;
    int walks = 0;
    for (int m = 0; m < n && so; ++m) {
        if (!(so[m].n_accepted || so[m].n_emitted || so[m].path_nodes || so[m].path_tokens)) continue;
        WalkArgs &w = wk.w[walks++];
        w.accept_idx = no[m].accept_idx;
        w.token = no[m].token;
        w.child = d->child;
        w.node_kind = d->node_kind;
        w.n_accepted = so[m].n_accepted;
        w.n_emitted = so[m].n_emitted;
        w.path_nodes = so[m].path_nodes;
        w.path_tokens = so[m].path_tokens;
        w.batch = d->batch;
        w.nodes = d->nodes;
        w.levels = d->levels;
    }
    return walks ? launch_walk(wk, walks, s) : SPECHUB_OK;
}

int verify_common(const spechub_desc *d, const void *target_logits, const void *draft_logits,
                  const int32_t *draft_tokens, const float *uniforms, int method,
                  const spechub_node_out *no, const spechub_seq_out *so, void *workspace,
                  size_t workspace_bytes, void *stream, const void *draft_stats = nullptr) {
    const int rc = check_desc(d);
    if (rc != SPECHUB_OK) return rc;
    if (d->batch == 0) return SPECHUB_OK;  // nothing to do; pointers are not looked at
    if (!target_logits || !draft_logits || !draft_tokens || !uniforms || !no || !no->accept_idx ||
        !no->token)
        return SPECHUB_ERR_NULL;
    if (workspace_bytes < spechub_workspace_bytes(d)) return SPECHUB_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(draft_stats) % 16 != 0) return SPECHUB_ERR_STRIDE;
    (void)workspace;
    RowArgs a = base_args(d);
    a.draft_stats_in = draft_stats;
    a.target = target_logits;
    a.draft = draft_logits;
    a.uniforms = uniforms;
    a.draft_tokens_in = draft_tokens;
    a.hub = no->hub;
    a.accept_idx = no->accept_idx;
    a.token = no->token;
    a.beta = no->beta;
    a.rate = no->rate;
    a.status = no->status;
    const unsigned rows = (unsigned)(d->batch * (int64_t)d->nodes);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bool al = rows_aligned(d, target_logits) && rows_aligned(d, draft_logits);
    const int fmt = stream_format(d, al, target_logits, draft_logits);
    if (!keeps_stats(d, fmt)) a.draft_stats_in = nullptr;
    int lrc;
    ResShape rs;
    RegPlan pl;
    if (d->k > 2 && method == kSpecHub) return SPECHUB_ERR_SHAPE;
    KaryArgs ka;
    ka.r = a; ka.k = d->k; ka.without_replacement = (method == kRRSw);
    const int cs = lean_ok(d, al) ? lean_split(d) : 0;
    if (use_reg(true, d, al, rows, &pl)) {
        // (these kernels only check the records; beside rows of any alignment they are not refused, see lean_verify_kernel)
        if (fmt != kBf16 && fmt != kF32) ka.r.draft_stats_in = nullptr;
        lrc = launch_reg_verify(pl, d->dtype, ka, method, rows, s);
    } else if (d->k > 2) {
        if (resident_shape(d, al, &rs)) lrc = launch_resident_kary(rs, ka, rows, s);
        else lrc = launch_kary_verify(fmt, ka, rows, s);
    } else if (resident_shape(d, al, &rs)) {
        FusedArgs f = {};
        f.r = a;
        f.tok[method] = draft_tokens;
        f.out[method] = NodeOutPtrs{a.accept_idx, a.token, a.hub, a.beta, a.rate, a.status};
        lrc = launch_resident(1 << method, rs, f, rows, s);
    } else if (method == kSpecHub) {
        lrc = launch_lean_verify_spechub(fmt, cs, a, rows, s);
    } else if (method == kRRS) {
        lrc = launch_lean_verify_rrs(fmt, cs, a, rows, s);
    } else {
        lrc = launch_lean_verify_rrsw(fmt, cs, a, rows, s);
    }
    if (lrc != SPECHUB_OK) return lrc;
    return launch_walks(d, no, so, 1, s);
}

// One kernel for the three methods where the lean kernels apply, the three separate paths otherwise.
int compare_draft(const spechub_desc *d, const void *draft_logits, const float *uniforms,
                  int32_t *const draft_tokens[3], int32_t *hub, float *draft_prob,
                  uint32_t *const status[3], void *stream, void *draft_stats = nullptr) {
    const int rc = check_desc(d);
    if (rc != SPECHUB_OK) return rc;
    if (d->k != 2) return SPECHUB_ERR_SHAPE;
    if (d->batch == 0) return SPECHUB_OK;
    if (!draft_logits || !uniforms || !draft_tokens || !draft_tokens[0] || !draft_tokens[1] || !draft_tokens[2])
        return SPECHUB_ERR_NULL;
    if (reinterpret_cast<uintptr_t>(draft_stats) % 16 != 0) return SPECHUB_ERR_STRIDE;
    const unsigned rows = (unsigned)(d->batch * (int64_t)d->nodes);
    RegPlan pl;
    const bool al = rows_aligned(d, draft_logits);
    if (!lean_ok(d, al) || use_reg(false, d, al, rows, &pl)) {
        for (int m = 0; m < 3; ++m) {
            const int mrc = draft_common(d, draft_logits, uniforms, m, draft_tokens[m], m == 0 ? hub : nullptr,
                                         m == 0 ? draft_prob : nullptr, status ? status[m] : nullptr, stream,
                                         m == 0 ? draft_stats : nullptr);   // (one record serves the three)
            if (mrc != SPECHUB_OK) return mrc;
        }
        return SPECHUB_OK;
    }
    FusedArgs f = {};
    f.r = base_args(d);
    f.r.draft = draft_logits;
    f.r.uniforms = uniforms;
    // records are kept where the per-method calls keep them: no split flag
    if (draft_stats && lean_split(d) != 0 &&
        cudaMemsetAsync(draft_stats, 0, spechub_draft_stats_bytes(d), static_cast<cudaStream_t>(stream)) != cudaSuccess)
        return SPECHUB_ERR_LAUNCH;
    f.r.draft_stats_out = lean_split(d) == 0 ? draft_stats : nullptr;
    for (int m = 0; m < 3; ++m) {
        f.tok_out[m] = draft_tokens[m];
        f.dstatus[m] = status ? status[m] : nullptr;
    }
    return launch_fused_draft(f, hub, draft_prob, rows, static_cast<cudaStream_t>(stream));
}

int compare_verify(const spechub_desc *d, const void *target_logits, const void *draft_logits,
                   const int32_t *const draft_tokens[3], const float *uniforms,
                   const spechub_node_out *no, const spechub_seq_out *so, void *workspace,
                   size_t workspace_bytes, void *stream, const void *draft_stats = nullptr) {
    const int rc = check_desc(d);
    if (rc != SPECHUB_OK) return rc;
    if (d->k != 2) return SPECHUB_ERR_SHAPE;
    if (d->batch == 0) return SPECHUB_OK;
    if (!target_logits || !draft_logits || !uniforms || !no || !draft_tokens) return SPECHUB_ERR_NULL;
    for (int m = 0; m < 3; ++m)
        if (!draft_tokens[m] || !no[m].accept_idx || !no[m].token) return SPECHUB_ERR_NULL;
    if (workspace_bytes < spechub_workspace_bytes(d)) return SPECHUB_ERR_WORKSPACE;
    const bool al = rows_aligned(d, target_logits) && rows_aligned(d, draft_logits);
    const unsigned rows = (unsigned)(d->batch * (int64_t)d->nodes);
    RegPlan pl;
    if (!lean_ok(d, al) || use_reg(true, d, al, rows, &pl)) {
        for (int m = 0; m < 3; ++m) {
            const int mrc = verify_common(d, target_logits, draft_logits, draft_tokens[m], uniforms, m, &no[m],
                                          nullptr, workspace, workspace_bytes, stream, draft_stats);
            if (mrc != SPECHUB_OK) return mrc;
        }
        return launch_walks(d, no, so, 3, static_cast<cudaStream_t>(stream));
    }
    FusedArgs f = {};
    f.r = base_args(d);
    f.r.target = target_logits;
    f.r.draft = draft_logits;
    f.r.uniforms = uniforms;
    for (int m = 0; m < 3; ++m) {
        f.tok[m] = draft_tokens[m];
        f.out[m].accept_idx = no[m].accept_idx; f.out[m].token = no[m].token; f.out[m].hub = no[m].hub;
        f.out[m].beta = no[m].beta; f.out[m].rate = no[m].rate; f.out[m].status = no[m].status;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int lrc;
    if (ResShape rs; resident_shape(d, al, &rs)) {
        lrc = launch_resident(7, rs, f, rows, s);
    } else {
        if (d->node_kind) {
            const int llrc = launch_lean_leaf(kBf16, f.r, 2, f.out, 3, rows, s);
            if (llrc != SPECHUB_OK) return llrc;
        }
        if (lean_split(d) == 0) f.r.draft_stats_in = draft_stats;
        lrc = launch_fused_verify(f, rows, s);
    }
    return lrc == SPECHUB_OK ? launch_walks(d, no, so, 3, s) : lrc;
}

// ---- vocabulary-sharded phases ------------------------------------------------------------------
int check_shard(const spechub_desc *d, const spechub_shard *sh) {
    const int rc = check_desc(d);
    if (rc != SPECHUB_OK) return rc;
    if (!sh) return SPECHUB_ERR_NULL;
    if (d->k != 2) return SPECHUB_ERR_SHAPE;
    if (sh->nranks < 1 || sh->nranks > 64 || sh->rank < 0 || sh->rank >= sh->nranks || sh->id_offset < 0 ||
        sh->vocab_total < 2 || (int64_t)sh->id_offset + d->vocab > sh->vocab_total)
        return SPECHUB_ERR_SHAPE;
    return SPECHUB_OK;
}

ShardArgs shard_args(const spechub_desc *d, const spechub_shard *sh) {
    ShardArgs a = {};
    a.r = base_args(d);
    a.rank = sh->rank; a.nranks = sh->nranks; a.id_offset = sh->id_offset; a.vocab_total = sh->vocab_total;
    a.rows = d->batch * (int64_t)d->nodes;
    return a;
}

int run_shard_phase(int phase, const spechub_desc *d, const ShardArgs &a, void *stream) {
    const unsigned rows = (unsigned)a.rows;
    const int th = threads_for(d);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bool al = (!a.r.target || rows_aligned(d, a.r.target)) && (!a.r.draft || rows_aligned(d, a.r.draft));
    return launch_shard_phase(phase, d->dtype, al, th, a, rows, s);
}

}  // namespace

namespace spechub {

int allow_smem(const void *kern, int bytes, bool *configured) {
    static std::mutex mutex;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return SPECHUB_ERR_LAUNCH;
    std::lock_guard<std::mutex> lock(mutex);
    if (!configured[dev]) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) {
            cudaGetLastError();
            return SPECHUB_ERR_LAUNCH;
        }
        configured[dev] = true;
    }
    return SPECHUB_OK;
}

}  // namespace spechub

extern "C" {

int spechub_draft_sample(const spechub_desc *desc, const void *draft_logits, const float *uniforms,
                         int32_t *draft_tokens, int32_t *hub, float *draft_prob, uint32_t *status,
                         void *stream) {
    return draft_common(desc, draft_logits, uniforms, kSpecHub, draft_tokens, hub, draft_prob, status,
                        stream);
}

int rrs_draft_sample(const spechub_desc *desc, const void *draft_logits, const float *uniforms,
                     int without_replacement, int32_t *draft_tokens, uint32_t *status, void *stream) {
    if (without_replacement != 0 && without_replacement != 1) return SPECHUB_ERR_METHOD;
    return draft_common(desc, draft_logits, uniforms, without_replacement ? kRRSw : kRRS,
                        draft_tokens, nullptr, nullptr, status, stream);
}

int spechub_draft_sample_stats(const spechub_desc *desc, const void *draft_logits, const float *uniforms,
                               int32_t *draft_tokens, int32_t *hub, float *draft_prob, uint32_t *status,
                               void *draft_stats, void *stream) {
    if (!draft_stats && desc && desc->batch != 0) return SPECHUB_ERR_NULL;
    return draft_common(desc, draft_logits, uniforms, kSpecHub, draft_tokens, hub, draft_prob, status,
                        stream, draft_stats);
}

int rrs_draft_sample_stats(const spechub_desc *desc, const void *draft_logits, const float *uniforms,
                           int without_replacement, int32_t *draft_tokens, uint32_t *status,
                           void *draft_stats, void *stream) {
    if (without_replacement != 0 && without_replacement != 1) return SPECHUB_ERR_METHOD;
    if (!draft_stats && desc && desc->batch != 0) return SPECHUB_ERR_NULL;
    return draft_common(desc, draft_logits, uniforms, without_replacement ? kRRSw : kRRS,
                        draft_tokens, nullptr, nullptr, status, stream, draft_stats);
}

int spechub_verify_tree_stats(const spechub_desc *desc, const void *target_logits, const void *draft_logits,
                              const void *draft_stats, const int32_t *draft_tokens, const float *uniforms,
                              const spechub_node_out *node_out, const spechub_seq_out *seq_out,
                              void *workspace, size_t workspace_bytes, void *stream) {
    if (!draft_stats && desc && desc->batch != 0) return SPECHUB_ERR_NULL;
    return verify_common(desc, target_logits, draft_logits, draft_tokens, uniforms, kSpecHub,
                         node_out, seq_out, workspace, workspace_bytes, stream, draft_stats);
}

int rrs_verify_tree_stats(const spechub_desc *desc, const void *target_logits, const void *draft_logits,
                          const void *draft_stats, const int32_t *draft_tokens, const float *uniforms,
                          int without_replacement, const spechub_node_out *node_out,
                          const spechub_seq_out *seq_out, void *workspace, size_t workspace_bytes,
                          void *stream) {
    if (without_replacement != 0 && without_replacement != 1) return SPECHUB_ERR_METHOD;
    if (!draft_stats && desc && desc->batch != 0) return SPECHUB_ERR_NULL;
    return verify_common(desc, target_logits, draft_logits, draft_tokens, uniforms,
                         without_replacement ? kRRSw : kRRS, node_out, seq_out, workspace,
                         workspace_bytes, stream, draft_stats);
}

int spechub_verify_tree(const spechub_desc *desc, const void *target_logits,
                        const void *draft_logits, const int32_t *draft_tokens,
                        const float *uniforms, const spechub_node_out *node_out,
                        const spechub_seq_out *seq_out, void *workspace, size_t workspace_bytes,
                        void *stream) {
    return verify_common(desc, target_logits, draft_logits, draft_tokens, uniforms, kSpecHub,
                         node_out, seq_out, workspace, workspace_bytes, stream);
}

int rrs_verify_tree(const spechub_desc *desc, const void *target_logits, const void *draft_logits,
                    const int32_t *draft_tokens, const float *uniforms, int without_replacement,
                    const spechub_node_out *node_out, const spechub_seq_out *seq_out,
                    void *workspace, size_t workspace_bytes, void *stream) {
    if (without_replacement != 0 && without_replacement != 1) return SPECHUB_ERR_METHOD;
    return verify_common(desc, target_logits, draft_logits, draft_tokens, uniforms,
                         without_replacement ? kRRSw : kRRS, node_out, seq_out, workspace,
                         workspace_bytes, stream);
}

int mdsd_compare_draft_sample(const spechub_desc *desc, const void *draft_logits, const float *uniforms,
                              int32_t *const draft_tokens[3], int32_t *hub, float *draft_prob,
                              uint32_t *const status[3], void *stream) {
    return compare_draft(desc, draft_logits, uniforms, draft_tokens, hub, draft_prob, status, stream);
}

int mdsd_compare_draft_sample_stats(const spechub_desc *desc, const void *draft_logits, const float *uniforms,
                                    int32_t *const draft_tokens[3], int32_t *hub, float *draft_prob,
                                    uint32_t *const status[3], void *draft_stats, void *stream) {
    if (!draft_stats && desc && desc->batch != 0) return SPECHUB_ERR_NULL;
    return compare_draft(desc, draft_logits, uniforms, draft_tokens, hub, draft_prob, status, stream, draft_stats);
}

int mdsd_compare_verify_tree_stats(const spechub_desc *desc, const void *target_logits, const void *draft_logits,
                                   const void *draft_stats, const int32_t *const draft_tokens[3],
                                   const float *uniforms, const spechub_node_out node_out[3],
                                   const spechub_seq_out *seq_out, void *workspace, size_t workspace_bytes,
                                   void *stream) {
    if (!draft_stats && desc && desc->batch != 0) return SPECHUB_ERR_NULL;
    if (reinterpret_cast<uintptr_t>(draft_stats) % 16 != 0) return SPECHUB_ERR_STRIDE;
    return compare_verify(desc, target_logits, draft_logits, draft_tokens, uniforms, node_out, seq_out,
                          workspace, workspace_bytes, stream, draft_stats);
}

int mdsd_compare_verify_tree(const spechub_desc *desc, const void *target_logits, const void *draft_logits,
                             const int32_t *const draft_tokens[3], const float *uniforms,
                             const spechub_node_out node_out[3], const spechub_seq_out *seq_out,
                             void *workspace, size_t workspace_bytes, void *stream) {
    return compare_verify(desc, target_logits, draft_logits, draft_tokens, uniforms, node_out, seq_out,
                          workspace, workspace_bytes, stream);
}

int spechub_walk_tree(const spechub_desc *desc, const int32_t *accept_idx, const int32_t *token,
                      const spechub_seq_out *seq_out, void *stream) {
    const int rc = check_desc(desc);
    if (rc != SPECHUB_OK) return rc;
    if (desc->batch == 0) return SPECHUB_OK;
    if (!accept_idx || !token || !seq_out) return SPECHUB_ERR_NULL;
    spechub_node_out no = {};
    no.accept_idx = const_cast<int32_t *>(accept_idx);
    no.token = const_cast<int32_t *>(token);
    return launch_walks(desc, &no, seq_out, 1, static_cast<cudaStream_t>(stream));
}

int spechub_shard_stats(const spechub_desc *desc, const spechub_shard *shard, const void *target_slice,
                        const void *draft_slice, float *stats, void *stream) {
    const int rc = check_shard(desc, shard);
    if (rc != SPECHUB_OK) return rc;
    if (desc->batch == 0) return SPECHUB_OK;
    if (!draft_slice || !stats) return SPECHUB_ERR_NULL;
    ShardArgs a = shard_args(desc, shard);
    a.r.target = target_slice; a.r.draft = draft_slice; a.out = stats;
    return run_shard_phase(kPhaseStats, desc, a, stream);
}

int spechub_shard_sums(const spechub_desc *desc, const spechub_shard *shard, const void *target_slice,
                       const void *draft_slice, const int32_t *draft_tokens, const float *gathered_stats,
                       float *sums, void *stream) {
    const int rc = check_shard(desc, shard);
    if (rc != SPECHUB_OK) return rc;
    if (desc->batch == 0) return SPECHUB_OK;
    if (!target_slice || !draft_slice || !draft_tokens || !gathered_stats || !sums) return SPECHUB_ERR_NULL;
    ShardArgs a = shard_args(desc, shard);
    a.r.target = target_slice; a.r.draft = draft_slice; a.r.draft_tokens_in = draft_tokens;
    a.gstats = gathered_stats; a.out = sums;
    return run_shard_phase(kPhaseSums, desc, a, stream);
}

int spechub_shard_decide(const spechub_desc *desc, const spechub_shard *shard, const void *target_slice,
                         const void *draft_slice, const int32_t *draft_tokens, const float *uniforms,
                         const float *gathered_stats, const float *gathered_sums,
                         const spechub_node_out *no, void *stream) {
    const int rc = check_shard(desc, shard);
    if (rc != SPECHUB_OK) return rc;
    if (desc->batch == 0) return SPECHUB_OK;
    if (!target_slice || !draft_slice || !draft_tokens || !uniforms || !gathered_stats || !gathered_sums ||
        !no || !no->accept_idx || !no->token)
        return SPECHUB_ERR_NULL;
    ShardArgs a = shard_args(desc, shard);
    a.r.target = target_slice; a.r.draft = draft_slice; a.r.draft_tokens_in = draft_tokens;
    a.r.uniforms = uniforms; a.gstats = gathered_stats; a.gsums = gathered_sums;
    a.r.hub = no->hub; a.r.accept_idx = no->accept_idx; a.r.token = no->token;
    a.r.beta = no->beta; a.r.rate = no->rate; a.r.status = no->status;
    return run_shard_phase(kPhaseDecide, desc, a, stream);
}

int spechub_shard_draft(const spechub_desc *desc, const spechub_shard *shard, const void *draft_slice,
                        const float *uniforms, const float *gathered_stats, int32_t *cand, void *stream) {
    const int rc = check_shard(desc, shard);
    if (rc != SPECHUB_OK) return rc;
    if (desc->batch == 0) return SPECHUB_OK;
    if (!draft_slice || !uniforms || !gathered_stats || !cand) return SPECHUB_ERR_NULL;
    ShardArgs a = shard_args(desc, shard);
    a.r.draft = draft_slice; a.r.uniforms = uniforms; a.gstats = gathered_stats; a.cand_out = cand;
    return run_shard_phase(kPhaseDraft, desc, a, stream);
}

int spechub_shard_draft_finish(const spechub_desc *desc, const spechub_shard *shard,
                               const float *gathered_stats, const int32_t *cand_max,
                               int32_t *draft_tokens, int32_t *hub, uint32_t *status, void *stream) {
    const int rc = check_shard(desc, shard);
    if (rc != SPECHUB_OK) return rc;
    if (desc->batch == 0) return SPECHUB_OK;
    if (!gathered_stats || !cand_max || !draft_tokens) return SPECHUB_ERR_NULL;
    ShardArgs a = shard_args(desc, shard);
    a.gstats = gathered_stats; a.cand = cand_max;
    a.r.draft_tokens_out = draft_tokens; a.r.hub = hub; a.r.status = status;
    return launch_shard_draft_finish(false, a, static_cast<cudaStream_t>(stream));
}

int rrs_shard_sums(const spechub_desc *desc, const spechub_shard *shard, int without_replacement,
                   const void *target_slice, const void *draft_slice, const int32_t *draft_tokens,
                   const float *gathered_stats, const float *gathered_sums, float *out, void *stream) {
    if (without_replacement != 0 && without_replacement != 1) return SPECHUB_ERR_METHOD;
    const int rc = check_shard(desc, shard);
    if (rc != SPECHUB_OK) return rc;
    if (desc->batch == 0) return SPECHUB_OK;
    if (!target_slice || !draft_slice || !draft_tokens || !gathered_stats || !out) return SPECHUB_ERR_NULL;
    ShardArgs a = shard_args(desc, shard);
    a.without_replacement = without_replacement;
    a.r.target = target_slice; a.r.draft = draft_slice; a.r.draft_tokens_in = draft_tokens;
    a.gstats = gathered_stats; a.gsums = gathered_sums; a.out = out;
    return run_shard_phase(kPhaseRrsSums, desc, a, stream);
}

int rrs_shard_decide(const spechub_desc *desc, const spechub_shard *shard, int without_replacement,
                     const void *target_slice, const void *draft_slice, const int32_t *draft_tokens,
                     const float *uniforms, const float *gathered_stats, const float *gathered_sums,
                     const float *gathered_w2, const spechub_node_out *no, void *stream) {
    if (without_replacement != 0 && without_replacement != 1) return SPECHUB_ERR_METHOD;
    const int rc = check_shard(desc, shard);
    if (rc != SPECHUB_OK) return rc;
    if (desc->batch == 0) return SPECHUB_OK;
    if (!target_slice || !draft_slice || !draft_tokens || !uniforms || !gathered_stats || !gathered_sums ||
        !gathered_w2 || !no || !no->accept_idx || !no->token)
        return SPECHUB_ERR_NULL;
    ShardArgs a = shard_args(desc, shard);
    a.without_replacement = without_replacement;
    a.r.target = target_slice; a.r.draft = draft_slice; a.r.draft_tokens_in = draft_tokens;
    a.r.uniforms = uniforms; a.gstats = gathered_stats; a.gsums = gathered_sums; a.gw2 = gathered_w2;
    a.r.hub = no->hub; a.r.accept_idx = no->accept_idx; a.r.token = no->token;
    a.r.beta = no->beta; a.r.rate = no->rate; a.r.status = no->status;
    return run_shard_phase(kPhaseRrsDecide, desc, a, stream);
}

int rrs_shard_draft(const spechub_desc *desc, const spechub_shard *shard, int without_replacement,
                    const void *draft_slice, const float *uniforms, const float *gathered_stats,
                    const int32_t *cand_max, const float *ex1_max, int32_t *cand, float *ex1, void *stream) {
    if (without_replacement != 0 && without_replacement != 1) return SPECHUB_ERR_METHOD;
    const int rc = check_shard(desc, shard);
    if (rc != SPECHUB_OK) return rc;
    if (desc->batch == 0) return SPECHUB_OK;
    if (!draft_slice || !uniforms || !gathered_stats || !cand) return SPECHUB_ERR_NULL;
    if ((cand_max == nullptr) != (ex1_max == nullptr)) return SPECHUB_ERR_NULL;
    if (cand_max && !without_replacement) return SPECHUB_ERR_METHOD;   // only RRSw has a second round
    ShardArgs a = shard_args(desc, shard);
    a.without_replacement = without_replacement;
    a.r.draft = draft_slice; a.r.uniforms = uniforms; a.gstats = gathered_stats;
    a.x1_known = cand_max; a.ex1_known = ex1_max; a.cand_out = cand; a.ex1_out = ex1;
    return run_shard_phase(kPhaseRrsDraft, desc, a, stream);
}

int rrs_shard_draft_finish(const spechub_desc *desc, const spechub_shard *shard, int without_replacement,
                           const float *gathered_stats, const int32_t *cand_max, int32_t *draft_tokens,
                           uint32_t *status, void *stream) {
    if (without_replacement != 0 && without_replacement != 1) return SPECHUB_ERR_METHOD;
    const int rc = check_shard(desc, shard);
    if (rc != SPECHUB_OK) return rc;
    if (desc->batch == 0) return SPECHUB_OK;
    if (!gathered_stats || !cand_max || !draft_tokens) return SPECHUB_ERR_NULL;
    ShardArgs a = shard_args(desc, shard);
    a.without_replacement = without_replacement;
    a.gstats = gathered_stats; a.cand = cand_max;
    a.r.draft_tokens_out = draft_tokens; a.r.status = status;
    return launch_shard_draft_finish(true, a, static_cast<cudaStream_t>(stream));
}

size_t spechub_workspace_bytes(const spechub_desc *desc) {
    (void)desc;
    return 0;
}

size_t spechub_draft_stats_bytes(const spechub_desc *desc) {
    if (!desc || desc->batch < 0 || desc->nodes < 1) return 0;
    return sizeof(DraftStat) * static_cast<size_t>(desc->batch) * static_cast<size_t>(desc->nodes);
}

const char *spechub_status_string(int code) {
    switch (code) {
        case SPECHUB_OK: return "ok";
        case SPECHUB_ERR_NULL: return "a required pointer is NULL";
        case SPECHUB_ERR_VERSION: return "descriptor struct_size/version mismatch";
        case SPECHUB_ERR_SHAPE: return "bad shape: need batch >= 0, nodes >= 1, vocab >= 2, 2 <= k <= 8 (k == 2 for SpecHub), levels >= 1, valid flags";
        case SPECHUB_ERR_DTYPE: return "dtype must be SPECHUB_F32 or SPECHUB_BF16";
        case SPECHUB_ERR_STRIDE: return "strides too small for the given shape";
        case SPECHUB_ERR_TEMPERATURE: return "temperature must be finite and > 0";
        case SPECHUB_ERR_WORKSPACE: return "workspace smaller than spechub_workspace_bytes()";
        case SPECHUB_ERR_LAUNCH: return "kernel launch failed";
        case SPECHUB_ERR_METHOD: return "without_replacement must be 0 or 1";
        case SPECHUB_ERR_TOO_LARGE: return "batch * nodes exceeds SPECHUB_STATIC_MAX_ROWS of spechub_verify_tree_static";
        default: return "unknown status";
    }
}

int spechub_abi_version(void) { return SPECHUB_ABI_VERSION; }

}  // extern "C"

// ---- verification without any allocation ---------------------------------------------------------
// Scratch of spechub_verify_tree_static: per row the "stats" record and the "sums" record of the
// phase kernels (8 floats each).  Lives in every GPU that loads the library until the process ends.
static __device__ __align__(256) float g_static_scratch[(size_t)SPECHUB_STATIC_MAX_ROWS * 2 * spechub::kShardRecord];

namespace {

std::mutex g_static_mutex;
float *g_static_ptr[kMaxDevices] = {};

// Device address of g_static_scratch on the current device.  In host code the array's name is only
// a handle for the runtime, never an address a kernel may be given, so the address is looked up
// once per device (with that device current) and kept.
int static_scratch(float **out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return SPECHUB_ERR_LAUNCH;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_ptr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) {
            cudaGetLastError();
            return SPECHUB_ERR_LAUNCH;
        }
        g_static_ptr[dev] = static_cast<float *>(p);
    }
    *out = g_static_ptr[dev];
    return SPECHUB_OK;
}

}  // namespace

extern "C" int spechub_verify_tree_static(const spechub_desc *desc, const void *target_logits,
                                          const void *draft_logits, const int32_t *draft_tokens,
                                          const float *uniforms, const spechub_node_out *no,
                                          const spechub_seq_out *so, void *stream) {
    const int rc = check_desc(desc);
    if (rc != SPECHUB_OK) return rc;
    if (desc->k != 2) return SPECHUB_ERR_SHAPE;
    if (desc->batch == 0) return SPECHUB_OK;
    if (!target_logits || !draft_logits || !draft_tokens || !uniforms || !no || !no->accept_idx || !no->token)
        return SPECHUB_ERR_NULL;
    const int64_t rows = desc->batch * (int64_t)desc->nodes;
    if (rows > SPECHUB_STATIC_MAX_ROWS) return SPECHUB_ERR_TOO_LARGE;
    float *scratch = nullptr;
    const int src = static_scratch(&scratch);
    if (src != SPECHUB_OK) return src;
    float *stats = scratch, *sums = scratch + rows * kShardRecord;

    // one rank that holds the whole vocabulary: the phase kernels, back to back on the stream
    spechub_shard whole = {0, 1, 0, desc->vocab};
    ShardArgs a = shard_args(desc, &whole);
    a.r.target = target_logits; a.r.draft = draft_logits; a.r.draft_tokens_in = draft_tokens;
    a.r.uniforms = uniforms;
    a.out = stats;                     // every record is written in full: nothing has to start at zero
    int prc = run_shard_phase(kPhaseStats, desc, a, stream);
    if (prc != SPECHUB_OK) return prc;
    a.gstats = stats; a.out = sums;
    prc = run_shard_phase(kPhaseSums, desc, a, stream);
    if (prc != SPECHUB_OK) return prc;
    a.gsums = sums; a.out = nullptr;
    a.r.hub = no->hub; a.r.accept_idx = no->accept_idx; a.r.token = no->token;
    a.r.beta = no->beta; a.r.rate = no->rate; a.r.status = no->status;
    prc = run_shard_phase(kPhaseDecide, desc, a, stream);
    if (prc != SPECHUB_OK) return prc;
    return launch_walks(desc, no, so, 1, static_cast<cudaStream_t>(stream));
}
