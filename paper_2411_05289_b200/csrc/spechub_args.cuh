// What the launch functions hand to the kernels.
#pragma once

#include <stdint.h>

#include "spechub.h"

namespace spechub {

enum Method { kSpecHub = 0, kRRS = 1, kRRSw = 2 };

constexpr int kMaxK = SPECHUB_MAX_K;

struct RowArgs {
    const void *target;   // [B][N][V] (verify only)
    const void *draft;    // [B][N][V]
    const float *uniforms;  // [B][N][5]
    const int32_t *draft_tokens_in;  // verify: [B][N][2]
    int32_t *draft_tokens_out;       // draft: [B][N][2]
    int32_t *hub;
    float *draft_prob;
    int32_t *accept_idx;
    int32_t *token;
    float *beta;
    float *rate;
    uint32_t *status;
    const float *temperature_per_seq;
    const uint8_t *node_kind;
    float temperature;
    int nodes, vocab;
    long long stride_seq, stride_node;
    // per-row statistics of the draft logits, handed from the draft step to verification: [B][N] DraftStat
    void *draft_stats_out;       // draft step, may be NULL
    const void *draft_stats_in;  // verification through a *_stats entry point
};

// What the draft step knows about a row of draft logits once it has read it, and what verification would
// otherwise have to read the row for a second time to find out (Section 4: a = argmax q; q(a); 1 - q(a)).
struct DraftStat {
    float ml;       // the row's maximum logit
    float sx;       // sum over ids != argmax of 2^(k l - rint(k ml)), k = log2(e) / T
    int idx;        // argmax, lowest id on ties
    unsigned tag;   // stat_tag: a record of another kind or temperature (with a mark: of another row) is not taken
};
constexpr unsigned kDraftStatTag = 0x51a76u << 12;   // (another number whenever the record's meaning changes)

// The records a draft step leaves: void ones, those of rows read in whole words, those of other rows (row_mark).
enum KeepStats : int { kVoidStats, kPlainStats, kMarkedStats };

struct NodeOutPtrs {
    int32_t *accept_idx, *token, *hub;
    float *beta, *rate;
    uint32_t *status;
};
struct LeafArgs {
    RowArgs r;
    NodeOutPtrs out[3];
    int n_out, k;
};

struct FusedArgs {
    RowArgs r;                 // target, draft, uniforms, temperature, node_kind, shape
    const int32_t *tok[3];     // draft tokens of SpecHub, RRS, RRSw (verify)
    int32_t *tok_out[3];       // (draft)
    NodeOutPtrs out[3];
    uint32_t *dstatus[3];      // draft status
};

struct KaryArgs {
    RowArgs r;
    int k;
    int without_replacement;
    KeepStats keep_stats;   // draft step: the records left for verification
};

constexpr int kShardRecord = 8;  // floats per row in a phase output

struct ShardArgs {
    RowArgs r;             // r.target / r.draft: this rank's slices; r.vocab: their width
    int rank, nranks, id_offset, vocab_total;
    long long rows;
    const float *gstats;   // [nranks][rows][8]: (ml, sx, idx) of p then of q, per rank
    const float *gsums;    // [nranks][rows][8]
    const float *gw2;      // [nranks][rows][8] (RRS / RRSw: second-stage residual masses)
    int without_replacement;
    const int32_t *x1_known;  // RRSw draft, second round: [rows][2] candidates after the maximum
    const float *ex1_known;   // ... and the exponential of x1's logit, [rows]
    float *ex1_out;           // first round: that exponential from x1's owner, -1 elsewhere
    const int32_t *cand;   // [rows][2] after the element-wise maximum over ranks
    float *out;            // [rows][8] phase output
    int32_t *cand_out;     // [rows][2]
};

struct WalkArgs {
    const int32_t *accept_idx, *token, *child;
    const uint8_t *node_kind;
    int32_t *n_accepted, *n_emitted, *path_nodes, *path_tokens;
    int batch, nodes, levels;
};

struct WalkKArgs {
    WalkArgs w[3];
    int k;
};
}  // namespace spechub
