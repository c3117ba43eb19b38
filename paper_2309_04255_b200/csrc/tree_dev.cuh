// Device-side pieces of the integer part of a pass, shared by the kernels of tree.cu and by the kernels
// that do this part themselves: the mask table of a tree (Sec. 3.2 "Tree decoder") and the
// verified-sequence search (Sec. 3.2 "Depth-first verified sequence searching").
//
// A tree has at most 128 nodes. Walking from a node to the root is a chain of dependent reads, 127 of
// them in a chain-shaped tree; both functions use pointer doubling instead: every node holds a pointer to
// an ancestor and what it knows about the nodes up to there, and adopts its ancestor's pointer and
// knowledge: ceil(log2(depth)) rounds, two block barriers each. All threads of the block call them (at
// least 128 threads); thread c works on node c.
#pragma once

#include "common.cuh"

namespace llmcad {

struct MaskTable {
    int32_t par[LLMCAD_MAX_TREE];
    int32_t jump[LLMCAD_MAX_TREE];
    uint32_t anc[LLMCAD_MAX_TREE][4];   // bit j of row i: node j is i or an ancestor of i
};

// Reads parent (and tokens, unless null), checks every link and token, and fills t.anc. Returns 0 or the
// error code, the same in every thread; with an error t.anc holds the node's own bit only.
__device__ __forceinline__ int mask_table(MaskTable &t, const int32_t *parent, const int32_t *tokens, int n, int vocab)
{
    const int c = threadIdx.x;
    int bad_tree = 0, bad_token = 0;
    if (c < n) {
        const int p = __ldg(parent + c);
        bad_tree = c == 0 ? p != -1 : (p < 0 || p >= c);
        if (tokens != nullptr) { const int tk = __ldg(tokens + c); bad_token = tk < 0 || tk >= vocab; }
        t.par[c] = bad_tree ? 0 : p;
        t.jump[c] = (c == 0 || bad_tree) ? 0 : p;
#pragma unroll
        for (int w = 0; w < 4; ++w) t.anc[c][w] = (c >> 5) == w ? 1u << (c & 31) : 0u;
    }
    bad_tree = __syncthreads_or(bad_tree);
    bad_token = __syncthreads_or(bad_token);
    if (bad_tree | bad_token) return bad_tree ? LLMCAD_ERR_BAD_TREE : LLMCAD_ERR_BAD_TOKEN;
    while (true) {
        uint32_t a[4];
        int j = 0, jj = 0;
        if (c < n) {
            j = t.jump[c];
            jj = t.jump[j];
#pragma unroll
            for (int w = 0; w < 4; ++w) a[w] = t.anc[c][w] | t.anc[j][w];
        }
        const int more = __syncthreads_or(j != 0);
        if (c < n) {
            t.jump[c] = jj;
#pragma unroll
            for (int w = 0; w < 4; ++w) t.anc[c][w] = a[w];
        }
        __syncthreads();
        if (!more) return 0;
    }
}

__device__ __forceinline__ int mask_depth(const uint32_t (&row)[4])
{
    return __popc(row[0]) + __popc(row[1]) + __popc(row[2]) + __popc(row[3]) - 1;
}

struct PathSearch {
    int32_t par[LLMCAD_MAX_TREE], jump[LLMCAD_MAX_TREE], ok[LLMCAD_MAX_TREE], dep[LLMCAD_MAX_TREE];
    int32_t path[LLMCAD_MAX_TREE];
    int32_t key[4], below[4];
    int32_t len, n_all, has_child;
};

// Node c is verified iff every link on its root path is correct (the child's draft token equals the
// target's output at the parent, best(p)); the verified sequence ends at the deepest verified node, ties to
// the lowest index. Fills s.path and s.len, with `report` also n_all (draft tokens on the longest branch
// through the last verified node) and has_child. The tree is valid.
template <typename Best>
__device__ __forceinline__ void path_search(PathSearch &s, const int32_t *parent, const int32_t *tokens, Best best_of, int n,
                                            bool report)
{
    const int c = threadIdx.x;
    int d = 0;
    if (c < n) {
        const int p = c == 0 ? 0 : __ldg(parent + c);
        s.par[c] = p;
        s.jump[c] = p;
        s.ok[c] = c == 0 ? 1 : (__ldg(tokens + c) == best_of(p));
        s.dep[c] = c != 0;
    }
    if (c == 0) s.has_child = 0;
    __syncthreads();
    while (true) {
        int j = 0, jj = 0, ok = 0;
        if (c < n) {
            j = s.jump[c];
            jj = s.jump[j];
            ok = s.ok[c] & s.ok[j];
            d = s.dep[c] + s.dep[j];
        }
        const int more = __syncthreads_or(j != 0);
        if (c < n) { s.jump[c] = jj; s.ok[c] = ok; s.dep[c] = d; }
        __syncthreads();
        if (!more) break;
    }
    if (c < LLMCAD_MAX_TREE) {
        int key = (c < n && s.ok[c]) ? (d << 8) | (LLMCAD_MAX_TREE - 1 - c) : -1;
        for (int o = 16; o; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
        if ((c & 31) == 0) s.key[c >> 5] = key;
    }
    __syncthreads();
    const int best = LLMCAD_MAX_TREE - 1 - (max(max(s.key[0], s.key[1]), max(s.key[2], s.key[3])) & 0xff);
    if (c == 0) {
        const int len = s.dep[best] + 1;
        s.len = len;
        for (int cur = best, j = len - 1; j >= 0; cur = s.par[cur], --j) s.path[j] = cur;
    }
    if (report && c < LLMCAD_MAX_TREE) {
        int below = -1;
        if (c < n) {
            int cur = c;
            while (cur > best) cur = s.par[cur];
            if (cur == best) below = d;
            if (c > 0 && s.par[c] == best) s.has_child = 1;
        }
        for (int o = 16; o; o >>= 1) below = max(below, __shfl_xor_sync(0xffffffffu, below, o));
        if ((c & 31) == 0) s.below[c >> 5] = below;
    }
    __syncthreads();
    if (report && c == 0) s.n_all = max(max(s.below[0], s.below[1]), max(s.below[2], s.below[3]));
}

// The outputs of a pass: the path, -1 in what its first path_len entries hold behind it, and scalars, by one block.
template <typename Best>
__device__ __forceinline__ void report_path(const PathSearch &s, Best best_of, int P, int path_len, int32_t *path, int32_t *scalars)
{
    for (int j = threadIdx.x; j < max(s.len, path_len); j += blockDim.x) path[j] = j < s.len ? s.path[j] : -1;
    if (threadIdx.x == 0) {
        scalars[LLMCAD_S_ACCEPTED_LEN] = s.len;
        scalars[LLMCAD_S_NEXT_TOKEN] = best_of(s.path[s.len - 1]);
        scalars[LLMCAD_S_NEW_PREFIX_LEN] = P + s.len;
        scalars[LLMCAD_S_N_CORRECT] = s.len - 1;
        scalars[LLMCAD_S_N_ALL] = s.n_all;
        scalars[LLMCAD_S_RECTIFIED] = s.has_child;
        scalars[LLMCAD_S_RESERVED] = 0;
    }
}
// The same for a pass that an earlier phase refused: an empty result. The status word is not written.
__device__ __forceinline__ void report_refused(int P, int path_len, int32_t *path, int32_t *scalars)
{
    for (int j = threadIdx.x; j < path_len; j += blockDim.x) path[j] = -1;
    if (threadIdx.x == 0) {
        scalars[LLMCAD_S_ACCEPTED_LEN] = 0;
        scalars[LLMCAD_S_NEXT_TOKEN] = -1;
        scalars[LLMCAD_S_NEW_PREFIX_LEN] = P;
        scalars[LLMCAD_S_N_CORRECT] = 0;
        scalars[LLMCAD_S_N_ALL] = 0;
        scalars[LLMCAD_S_RECTIFIED] = 0;
        scalars[LLMCAD_S_RESERVED] = 0;
    }
}

// Rollback (Sec. 3.2) of one 16-byte column of one head: rows P + path[j] -> P + j. path is strictly
// increasing with path[j] >= j, so an ascending copy never reads a slot that it has overwritten; eight rows
// are read before they are written to keep loads in flight. `base` points at slot P of the column.
__device__ __forceinline__ void rollback_column(uint4 *base, int chunks, const int32_t *path, int len)
{
    int j0 = 0;
    while (j0 < len && path[j0] == j0) ++j0;  // rows already in place
    for (int j = j0; j < len; j += 8) {
        uint4 tmp[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (j + u < len) tmp[u] = __ldcg(base + (size_t)path[j + u] * chunks);
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (j + u < len) base[(size_t)(j + u) * chunks] = tmp[u];
    }
}

}  // namespace llmcad
