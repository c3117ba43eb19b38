// Host-visible interface of the one-kernel bf16 pass over few nodes (pass_stream.cu).
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace llmcad {

constexpr int kStreamMaxNodes = 4;      // computed nodes of a pass

// One of the five GEMM shapes of a pass. Its units (a rotary pair of rows, gate and up row of a feature, or two
// adjacent rows) are dealt out to the CTAs; a CTA's eight warps are kg groups, which take the k-blocks in turn, of
// mg warps, which share the rows.
struct StreamGemm {
    int units, K;
    int mg, kg;
    int kb_item;              // k-blocks of 64 columns per ring item
    int kb_all, n_items, x_kb;          // k-blocks and items in all, k-blocks per stage of the input
    size_t upper;             // bytes from the matrix of the units' first rows to that of their second (SwiGLU), or 0
};

enum StreamKind : int { SG_QKV, SG_O, SG_GU, SG_DOWN, SG_HEAD, SG_KINDS };

struct StreamPass {
    // model and packed weights (offsets in bytes, as the packing lays them out)
    int L, d, H, f, V, S;
    float eps;
    const char *base;
    size_t w_off[SG_KINDS];             // inside a layer; SG_HEAD: from the base
    size_t attn_norm, ffn_norm, layer_bytes, tok_embed, final_norm;
    StreamGemm g[SG_KINDS];
    int w4;                             // the layer matrices are INT4 tiles
    char *kv;
    const double *inv_freq;
    // the tree: the nodes n_old .. n_tree-1 are computed
    const int32_t *tokens, *parent;
    int P, n_tree, n_old;
    int splits;                         // key ranges per head
    // workspaces: GEMM inputs as MMA fragments (see pass_stream.cu), fp32 queries and new keys and values [3][node][d],
    // partial attention outputs [head][split][node][kStreamPartRow], sums of squares [2][node][CTA], barrier words (zero
    // between launches): grid barrier, CTAs that left, then one per head
    void *xn, *att, *h;
    float *qkv, *part, *ssq;
    uint32_t *bar;
    // outputs; logits null: the decoder layers only. head_first .. n-1: the nodes whose logits are wanted
    float *logits;
    int head_first, head_parts;         // a CTA's rows of the lm_head are taken in so many parts
    int32_t *status;
    int keep_status;                    // the status word of an earlier chunk of the same call stands
    uint64_t wait_limit_ns;
    int withhold_input;                 // self-test of the wait limit: the copies of the phases' inputs are never issued
    int slots, slot_bytes, x_stage_bytes, x_off, red_off, q_off, cs_off;    // shared memory layout
};
constexpr int kStreamHeadParts = 4;
constexpr int kStreamPartRow = 132;     // 128 outputs, max, sum

// Whether a model of these sizes can go through the kernel at all, and whether a pass of n computed nodes should.
bool stream_pass_serves(int d, int f, int hd, int H, int V, int n_sms);
bool stream_pass_prefers(int n);
size_t stream_pass_floats_qkv(int d);
size_t stream_pass_floats_part(int n_sms);
// Fills in how the work is cut; false where shared memory does not hold it.
bool plan_stream_pass(StreamPass &p, int n_sms);
cudaError_t launch_stream_pass(const StreamPass &p, int n_sms, cudaStream_t st);

}  // namespace llmcad
