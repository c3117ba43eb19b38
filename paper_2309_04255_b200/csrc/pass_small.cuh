// Host-visible interface of the one-kernel fp32 pass (pass_small.cu).
#pragma once

#include "common.cuh"

namespace llmcad {

struct SmallPass {
    // model and packed weights (offsets in bytes, as the packing lays them out)
    int L, d, H, hd, f, V, S;
    float eps;
    const char *base;
    size_t attn_norm, wqkv, wo, ffn_norm, wgu, wdown, layer_bytes, tok_embed, final_norm, lm_head;
    float *kv;
    const double *inv_freq;
    // the tree: the nodes n_old .. n_tree-1 are computed
    const int32_t *tokens, *parent;
    int P, n_tree, n_old;
    // workspaces [node][...]: residual stream, queries, unnormalised attention outputs [range][node][d] (128 rows in
    // all) with (max, sum) [range][node][H], SwiGLU output, rotary table, best logit per node, barrier words (zero
    // between launches)
    float *x, *q, *att, *h;
    float2 *att_ml;
    float2 *rope_cs;
    unsigned long long *best;
    uint32_t *bar;
    // outputs; logits null: the decoder layers only (prefill)
    float *logits;
    int32_t *status;
    int keep_status;          // the status word of an earlier chunk of the same call stands
    int verify;               // 1: argmax, search and rollback follow
    int32_t *argmax, *path, *scalars;
    int path_fill;
    int top_k;                // > 0: the top_k most probable successors of every computed node
    int32_t *topk_ids;
    float *topk_probs;
    uint64_t wait_limit_ns;
};

// Whether a pass over n_keys keys (prefix and tree) fits this kernel; the caller sees to fp32.
bool small_pass_serves(int d, int f, int hd, int H, int n_keys);
cudaError_t launch_small_pass(const SmallPass &p, int n_sms, cudaStream_t st);

}  // namespace llmcad
