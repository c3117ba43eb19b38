// A whole fp32 pass in one cooperative kernel.
//
// The fp32 configuration is a small model: a pass is a chain of 5 L + 3 steps of a microsecond or two each. As
// one kernel per step it was bound by the hand-over between kernels and by steps that kept few loads in flight
// (2 layers, d 256: 33 kernels, 203 us at 15 nodes; 2.4 ms at 128 nodes and 2000 prefix keys). Here one CTA per
// SM stays for the whole pass, steps are separated by grid barriers (1.1-1.3 us each on 148 SMs, the slowest
// CTA's lead included), and what a step can fetch without the previous one, its first weights, it requests
// before the barrier: 59 us and 0.35 ms (4 layers of d 512 to 2048, 1 to 128 nodes: 1.3 to 23 times as fast;
// level at d 4096 with one node and a short prefix). What bounds it now is latency: a GEMM step is a barrier, one
// round trip to L2 for its input rows, ~1 us of arithmetic, and the stores.
//
//   GEMM steps    input rows are staged in shared memory (RMSNorm gain applied and sums of squares taken on the
//                 way in; the norm factor multiplies the finished sums). A warp owns two output rows (a rotary
//                 pair, or gate and up of one feature) on eight nodes, its lanes split K. One copy of the step's
//                 code with the epilogue chosen at run time: five copies spilled registers and ran cold.
//   attention     a CTA owns (head, one or two nodes, a range of keys): scores with eight threads per key,
//                 softmax, P V; the ranges are merged where the O GEMM stages its input.
//   tail          argmax (packed 64-bit maxima), verified-path search and rollback, or top-k.
//
// (The same kernel was built for bf16 models with mma.sync: 80 us against 79 us through the tensor-core kernels
// at d 512, 12 nodes, and slower above; not kept.)
//
// What another CTA wrote in this kernel is read past L1 (ld.cg). The barrier wait is bounded; when it runs out
// the CTA sets the status word and leaves, and so do the others.
#include "pass_small.cuh"
#include "topk_dev.cuh"
#include "tree_dev.cuh"

namespace llmcad {

namespace {

constexpr int kSpThreads = 256;             // 255 registers each: beside 200 KB of shared memory L1 has no room for spills
constexpr int kSpWarps = kSpThreads / 32;
constexpr size_t kSpSmem = 200 * 1024;      // dynamic shared memory, whatever the model

constexpr int kSpMaxSplits = 8;             // key ranges of an attention task
constexpr int kSpMaxAttW = 4096;            // (range, node, head) triples

enum Src : int { SRC_NORM, SRC_PLAIN, SRC_ATT };

// threadIdx.x as a value the compiler knows nothing about: every step derives its thread's share from its own, or
// address arithmetic of all steps would be moved in front of the loop over the layers and spilled there.
__device__ __forceinline__ int step_tid()
{
    int t = threadIdx.x;
    asm volatile("" : "+r"(t));
    return t;
}

struct SpShared {
    union {
        MaskTable table;                    // stays for the attention steps
        PathSearch search;
        TopkSmem topk;
    };
    float rs[LLMCAD_MAX_TREE];              // norm factors of the staged nodes
    unsigned long long best[LLMCAD_MAX_TREE];
    float m[kSpWarps], l[kSpWarps];
    float att_w[kSpMaxAttW];                // factors of the key ranges [range][node][head]
    int abort_flag;
};

// Grid barrier number k (1, 2, ...): all CTAs are resident (cooperative launch). False when the wait ran out.
struct GridBarrier {
    uint32_t *ctr;
    uint32_t target;
    uint64_t limit;
    int32_t *status;
    __device__ bool sync(SpShared &sh)
    {
        target += gridDim.x;
        __syncthreads();
        if (threadIdx.x == 0) {
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr) : "memory");
            uint64_t t0 = 0;
            int late = 0;
            for (uint32_t it = 1; ld_acquire_gpu_u32(ctr) < target; ++it) {
                if ((it & 255u) == 0) {
                    const uint64_t now = global_timer_ns();
                    if (t0 == 0) t0 = now;
                    else if (now - t0 > limit) { late = 1; break; }
                }
            }
            if (late) {
                atomicCAS(status, 0, LLMCAD_ERR_TIMEOUT);
                sh.abort_flag = 1;
            }
        }
        __syncthreads();
        return sh.abort_flag == 0;
    }
};

__device__ __forceinline__ unsigned long long pack_best(float v, int idx)
{
    const uint32_t u = __float_as_uint(v + 0.0f);           // -0 counts as +0
    const uint32_t ord = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return ((unsigned long long)ord << 32) | (0xffffffffu - (uint32_t)idx);
}
__device__ __forceinline__ int unpack_best(unsigned long long k) { return (int)(0xffffffffu - (uint32_t)k); }

// One GEMM step.
struct Gemm {
    const float *w;
    int n_out, K;            // output rows (SwiGLU: features), columns
    const float *gain;       // SRC_NORM
    int splits;              // SRC_ATT: key ranges to merge
    int layer;
    int epi, src;            // EpiMode, Src: run-time values, so that the kernel holds one copy of a step
};

// Input rows c0 .. c0 + nc - 1 into shared memory (nc, even, counts padding rows too, which become zero). A warp
// takes two rows at a time and has all their loads of 512 columns in flight: what this costs is round trips to L2.
__device__ __forceinline__ void stage_rows(const SmallPass &p, const Gemm &g, SpShared &sh, float *act, int c0, int nc, int n)
{
    const int tid = step_tid(), warp = tid >> 5, lane = tid & 31;
    for (int r = 2 * warp; r < nc; r += 2 * kSpWarps) {
        float ss[2] = {0.f, 0.f};
        for (int kb = 0; kb < g.K; kb += 512) {
            float4 v[2][4], gn[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = kb + u * 128 + lane * 4;
                if (g.src == SRC_NORM) gn[u] = k < g.K ? __ldg(reinterpret_cast<const float4 *>(g.gain + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int node = c0 + r + q;
                    const float *src = g.src == SRC_NORM ? p.x : g.src == SRC_PLAIN ? p.h : p.att;
                    v[q][u] = node < n && k < g.K ? __ldcg(reinterpret_cast<const float4 *>(src + (size_t)node * g.K + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
            if (g.src == SRC_ATT) {
                // the key ranges' outputs, weighted (att_weights): range 0 is in v
                for (int s = 0; s < g.splits; ++s) {
                    float4 o[2][4];
                    if (s > 0) {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                const int node = c0 + r + q, k = kb + u * 128 + lane * 4;
                                o[q][u] = node < n && k < g.K ? __ldcg(reinterpret_cast<const float4 *>(p.att + (size_t)(s * n + node) * g.K + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
                            }
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            const int node = min(c0 + r + q, n - 1), k = min(kb + u * 128 + lane * 4, g.K - 4);
                            const float w = sh.att_w[(s * n + node) * p.H + k / p.hd];
                            if (s == 0) { v[q][u].x *= w; v[q][u].y *= w; v[q][u].z *= w; v[q][u].w *= w; }
                            else { v[q][u].x += o[q][u].x * w; v[q][u].y += o[q][u].y * w; v[q][u].z += o[q][u].z * w; v[q][u].w += o[q][u].w * w; }
                        }
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = kb + u * 128 + lane * 4;
                if (k >= g.K) continue;
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    float4 a = v[q][u];
                    if (g.src == SRC_NORM) {
                        ss[q] += a.x * a.x + a.y * a.y + a.z * a.z + a.w * a.w;
                        a.x *= gn[u].x; a.y *= gn[u].y; a.z *= gn[u].z; a.w *= gn[u].w;
                    }
                    *reinterpret_cast<float4 *>(act + (size_t)(r + q) * g.K + k) = a;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (g.src == SRC_NORM)
                for (int o = 16; o; o >>= 1) ss[q] += __shfl_xor_sync(0xffffffffu, ss[q], o);
            if (lane == 0) sh.rs[r + q] = g.src == SRC_NORM ? rsqrtf(ss[q] / (float)g.K + p.eps) : 1.f;
        }
    }
}

// Merge of the key ranges: the factor of range s is 2^(m_s - M) / sum_s 2^(m_s - M) l_s.
__device__ __forceinline__ void att_weights(const SmallPass &p, SpShared &sh, int splits, int n)
{
    for (int i = step_tid(); i < n * p.H; i += kSpThreads) {
        float2 ml[kSpMaxSplits];
#pragma unroll
        for (int s = 0; s < kSpMaxSplits; ++s) ml[s] = s < splits ? __ldcg(p.att_ml + (size_t)s * n * p.H + i) : make_float2(-INFINITY, 0.f);
        float M = -INFINITY, L = 0.f;
#pragma unroll
        for (int s = 0; s < kSpMaxSplits; ++s) M = fmaxf(M, ml[s].x);
#pragma unroll
        for (int s = 0; s < kSpMaxSplits; ++s) {
            ml[s].x = ml[s].x == -INFINITY ? 0.f : exp2f(ml[s].x - M);
            L += ml[s].x * ml[s].y;
        }
        const float inv = L > 0.f ? 1.f / L : 0.f;
#pragma unroll
        for (int s = 0; s < kSpMaxSplits; ++s)
            if (s < splits) sh.att_w[s * n * p.H + i] = ml[s].x * inv;
    }
    __syncthreads();
}

// What a finished pair needs besides its sums, requested while the sums are still being made: the rotary
// (cos, sin), or the residual.
__device__ __forceinline__ float2 pair_aux(const SmallPass &p, const Gemm &g, int pair, int node)
{
    const int r0 = 2 * pair;
    if (g.epi == EPI_QKV && r0 < 2 * p.d) return __ldcg(p.rope_cs + (size_t)node * (p.hd >> 1) + ((r0 % p.hd) >> 1));
    if (g.epi == EPI_RESID) return __ldcg(reinterpret_cast<const float2 *>(p.x + (size_t)node * g.n_out + r0));
    return make_float2(1.f, 0.f);
}

// A finished pair of sums of one node: output rows 2 * pair and 2 * pair + 1, or gate and up of feature `pair`.
__device__ __forceinline__ void finish_pair(const SmallPass &p, const Gemm &g, SpShared &sh, int pair, int node, float v0, float v1, float2 aux)
{
    const int r0 = 2 * pair;
    if (g.epi == EPI_QKV) {
        const int sec = r0 / p.d, c = r0 - sec * p.d, head = c / p.hd, e = c - head * p.hd;
        const float o0 = v0 * aux.x - v1 * aux.y, o1 = v0 * aux.y + v1 * aux.x;      // values pass through with (1, 0)
        if (sec == 0) *reinterpret_cast<float2 *>(p.q + (size_t)node * p.d + c) = make_float2(o0, o1);
        else {
            const int slot = p.P + p.n_old + node;
            if (!LLMCAD_CHECK(slot < p.S && head < p.H, p.status)) return;
            float *dst = p.kv + (((size_t)g.layer * 2 + (sec - 1)) * p.H + head) * (size_t)p.S * p.hd + (size_t)slot * p.hd + e;
            *reinterpret_cast<float2 *>(dst) = make_float2(o0, o1);
        }
    } else if (g.epi == EPI_RESID) {
        *reinterpret_cast<float2 *>(p.x + (size_t)node * g.n_out + r0) = make_float2(aux.x + v0, aux.y + v1);
    } else if (g.epi == EPI_SWIGLU) {
        p.h[(size_t)node * g.n_out + pair] = v0 / (1.0f + expf(-v0)) * v1;
    } else {
        float *y = p.logits + (size_t)node * g.n_out + r0;
        const bool has1 = r0 + 1 < g.n_out;
        y[0] = v0;
        if (has1) y[1] = v1;
        if (p.verify) {
            if (v0 != v0 || (has1 && v1 != v1)) atomicCAS(p.status, 0, LLMCAD_ERR_NAN);
            unsigned long long b = pack_best(v0, r0);
            if (has1) { const unsigned long long b1 = pack_best(v1, r0 + 1); b = b1 > b ? b1 : b; }
            atomicMax(&sh.best[node], b);
        }
    }
}

// ---- a GEMM step: a warp per pair of output rows and eight nodes
__device__ __forceinline__ void pair_rows_f32(const Gemm &g, int epi, int pair, const float *&wa, const float *&wb)
{
    const float *W = g.w;
    if (epi == EPI_SWIGLU) {
        wa = W + (size_t)pair * g.K;
        wb = W + (size_t)(g.n_out + pair) * g.K;
    } else {
        wa = W + (size_t)(2 * pair) * g.K;
        wb = 2 * pair + 1 < g.n_out ? wa + g.K : wa;
    }
}

// columns k0 .. k0 + 255 of two rows: two 16-byte loads of each per lane
__device__ __forceinline__ void load_w_f32(float4 (&w)[2][2], const float *wa, const float *wb, int k0, int K, int lane)
{
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int k = k0 + u * 128 + lane * 4;
        const bool ok = k < K;
        w[0][u] = ok ? __ldg(reinterpret_cast<const float4 *>(wa + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
        w[1][u] = ok ? __ldg(reinterpret_cast<const float4 *>(wb + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

__device__ __forceinline__ bool gemm_step(const SmallPass &p, const Gemm &g, SpShared &sh, float *smem, GridBarrier &bar)
{
    const int tid = step_tid(), warp = tid >> 5, lane = tid & 31;
    const int n = p.n_tree - p.n_old;
    const int n_pairs = g.epi == EPI_SWIGLU ? g.n_out : (g.n_out + 1) / 2;
    const int total_warps = (int)gridDim.x * kSpWarps;
    const int first = warp * (int)gridDim.x + (int)blockIdx.x;      // neighbouring tasks on different SMs
    const int ld = g.K;                                             // floats
    const int cap = (int)(kSpSmem / ((size_t)g.K * 4)) / 8 * 8;
    const int chunk = min((n + 7) / 8 * 8, min(cap, LLMCAD_MAX_TREE));
    const float *wa = nullptr, *wb = nullptr;
    float4 pre[2][2];
    if (first < n_pairs) {                                          // the first task of a chunk of up to n_pairs * (chunk / 8) tasks
        pair_rows_f32(g, g.epi, first, wa, wb);
        load_w_f32(pre, wa, wb, 0, g.K, lane);
    }
    if (!bar.sync(sh)) return false;
    if (g.src == SRC_ATT) att_weights(p, sh, g.splits, n);
    for (int c0 = 0; c0 < n; c0 += chunk) {
        const int nc = min(chunk, (n - c0 + 7) / 8 * 8), n_tasks = n_pairs * (nc / 8);
        if (c0 > 0) __syncthreads();                                // the rows of the previous chunk have been used
        if ((int)blockIdx.x < n_tasks) stage_rows(p, g, sh, smem, c0, nc, n);
        __syncthreads();
        // a task = a pair of rows on eight nodes; the pairs first, so that a warp's first task is the preloaded one
        for (int task = first; task < n_tasks; task += total_warps) {
            const int b8 = task / n_pairs, pair = task - b8 * n_pairs, b = 8 * b8;
            const int node = c0 + b + (lane & 7);
            const float2 aux = lane < 8 && node < n ? pair_aux(p, g, pair, node) : make_float2(0.f, 0.f);
            pair_rows_f32(g, g.epi, pair, wa, wb);
            float acc[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) acc[i] = 0.f;
            float4 w[2][2];
            if (task == first && first < n_pairs && c0 == 0) {
#pragma unroll
                for (int u = 0; u < 2; ++u) { w[0][u] = pre[0][u]; w[1][u] = pre[1][u]; }
            } else load_w_f32(w, wa, wb, 0, g.K, lane);
            for (int k0 = 0; k0 < g.K; k0 += 256) {
                float4 nx[2][2];
                load_w_f32(nx, wa, wb, k0 + 256, g.K, lane);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int k = min(k0 + u * 128 + lane * 4, g.K - 4);        // past the row the weights are zero
                    const float *xs = smem + (size_t)b * ld + k;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float4 x = *reinterpret_cast<const float4 *>(xs + (size_t)i * ld);
                        acc[i] = fmaf(w[0][u].x, x.x, fmaf(w[0][u].y, x.y, fmaf(w[0][u].z, x.z, fmaf(w[0][u].w, x.w, acc[i]))));
                        acc[8 + i] = fmaf(w[1][u].x, x.x, fmaf(w[1][u].y, x.y, fmaf(w[1][u].z, x.z, fmaf(w[1][u].w, x.w, acc[8 + i]))));
                    }
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) { w[0][u] = nx[0][u]; w[1][u] = nx[1][u]; }
            }
            // sums over the lanes, scattered: lanes 8 * row + node (and + 16) end with their own, 16 shuffles for 16 sums
#pragma unroll
            for (int o = 8; o; o >>= 1) {
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int i = 0; i < o; ++i) {
                    const float send = up ? acc[i] : acc[i + o], keep = up ? acc[i + o] : acc[i];
                    acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
            acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 16);
            const float other = __shfl_xor_sync(0xffffffffu, acc[0], 8);
            if (lane < 8 && node < n) {
                const float rs = sh.rs[b + lane];
                finish_pair(p, g, sh, pair, node, acc[0] * rs, other * rs, aux);
            }
        }
    }
    return true;
}

// ---- attention: how the (head, nodes, key range) tasks are cut. More nodes per task only when there are more
// (head, node) pairs than CTAs; the keys are split when there are fewer, down to 64 keys a range.
struct AttnCut {
    int nodes, groups, splits;      // nodes per task, node groups, key ranges
};
__device__ __forceinline__ AttnCut attn_cut(const SmallPass &p)
{
    const int n = p.n_tree - p.n_old, n_keys = p.P + p.n_tree;
    AttnCut c;
    c.nodes = n * p.H > (int)gridDim.x ? 2 : 1;
    c.groups = (n + c.nodes - 1) / c.nodes;
    // (splits * n <= 128 rows of outputs)
    c.splits = min(min((int)gridDim.x / (c.groups * p.H), n_keys / 64), min(kSpMaxSplits, LLMCAD_MAX_TREE / n));
    if (c.splits < 1) c.splits = 1;
    return c;
}

// CPT: 16-byte chunks of a K row per thread (eight threads share a row)
template <int G, int CPT>
__device__ __forceinline__ void attention_tasks(const SmallPass &p, SpShared &sh, float *smem, const AttnCut &cut, int layer)
{
    constexpr int U = CPT == 4 ? 2 : 4, kGroupsOf8 = kSpThreads / 8;
    const int tid = step_tid(), warp = tid >> 5, lane = tid & 31;
    const int n = p.n_tree - p.n_old, hd = p.hd, n_keys = p.P + p.n_tree;
    const int tpr = hd / 4, parts = kSpThreads / tpr;             // threads per V row, keys in flight
    float *s_o = smem;                     // [parts][G][hd]
    float *s_sc = s_o + (size_t)parts * G * hd;                      // [G][keys of the range]
    const int range = (n_keys + cut.splits - 1) / cut.splits;
    const float scale = 1.4426950408889634f * rsqrtf((float)hd);
    const float *kl = p.kv + (size_t)layer * 2 * p.H * p.S * hd;
    const int n_tasks = p.H * cut.groups * cut.splits;
    for (int task = (int)blockIdx.x; task < n_tasks; task += (int)gridDim.x) {
        const int split = task / (p.H * cut.groups), rest = task - split * p.H * cut.groups;
        const int head = rest / cut.groups, node0 = (rest - head * cut.groups) * G;
        const int k0 = split * range, k1 = min(n_keys, k0 + range), nk = max(0, k1 - k0);
        const float *K = kl + (size_t)head * p.S * hd, *V = K + (size_t)p.H * p.S * hd;
        // ---- scores, in units of log2
        const int j = tid & 7;
        float4 q[G][CPT];
#pragma unroll
        for (int g = 0; g < G; ++g)
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                const float4 v = __ldcg(reinterpret_cast<const float4 *>(p.q + (size_t)min(node0 + g, n - 1) * p.d + head * hd) + j + 8 * c);
                q[g][c] = make_float4(v.x * scale, v.y * scale, v.z * scale, v.w * scale);
            }
        for (int kb = k0; kb < k1; kb += U * kGroupsOf8) {
            float4 r[U][CPT];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int c = 0; c < CPT; ++c)
                    r[u][c] = __ldcg(reinterpret_cast<const float4 *>(K + (size_t)min(kb + (tid >> 3) + u * kGroupsOf8, k1 - 1) * hd) + j + 8 * c);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int key = kb + (tid >> 3) + u * kGroupsOf8;
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    float dot = 0.f;
#pragma unroll
                    for (int c = 0; c < CPT; ++c)
                        dot = fmaf(q[g][c].x, r[u][c].x, fmaf(q[g][c].y, r[u][c].y, fmaf(q[g][c].z, r[u][c].z, fmaf(q[g][c].w, r[u][c].w, dot))));
                    for (int o = 4; o; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
                    if (j == 0 && key < k1) {
                        const int node = key - p.P, row = p.n_old + min(node0 + g, n - 1);
                        const bool vis = node < 0 || ((sh.table.anc[row][node >> 5] >> (node & 31)) & 1u);
                        s_sc[(size_t)g * range + key - k0] = vis ? dot : -INFINITY;
                    }
                }
            }
        }
        __syncthreads();
        // ---- softmax of the range: warp w works on node w % G
        const int wg = warp % G;
        float *sc = s_sc + (size_t)wg * range;
        float mx = -INFINITY;
        for (int i = (warp / G) * 32 + lane; i < nk; i += 32 * (kSpWarps / G)) mx = fmaxf(mx, sc[i]);
        for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) sh.m[warp] = mx;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kSpWarps / G; ++w) mx = fmaxf(mx, sh.m[w * G + wg]);
        const float ref = mx == -INFINITY ? 0.f : mx;
        float sum = 0.f;
        for (int i = (warp / G) * 32 + lane; i < nk; i += 32 * (kSpWarps / G)) {
            const float e = exp2f(sc[i] - ref);
            sc[i] = e;
            sum += e;
        }
        for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) sh.l[warp] = sum;
        __syncthreads();
        // ---- P V: a thread owns four of the head's dims and every parts-th key
        const int part = tid / tpr, c = tid - part * tpr;
        float4 acc[G];
#pragma unroll
        for (int g = 0; g < G; ++g) acc[g] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int i0 = part; i0 < nk; i0 += 8 * parts) {
            float4 r[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) r[u] = __ldcg(reinterpret_cast<const float4 *>(V + (size_t)(k0 + min(i0 + u * parts, nk - 1)) * hd) + c);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = i0 + u * parts;
                if (i >= nk) break;
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const float w = s_sc[(size_t)g * range + i];
                    acc[g].x = fmaf(w, r[u].x, acc[g].x); acc[g].y = fmaf(w, r[u].y, acc[g].y);
                    acc[g].z = fmaf(w, r[u].z, acc[g].z); acc[g].w = fmaf(w, r[u].w, acc[g].w);
                }
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g) *reinterpret_cast<float4 *>(s_o + ((size_t)part * G + g) * hd + c * 4) = acc[g];
        __syncthreads();
        for (int i = tid; i < G * hd; i += kSpThreads) {
            const int g = i / hd, e = i - g * hd, node = node0 + g;
            if (node >= n) continue;
            float o = 0.f;
            for (int q2 = 0; q2 < parts; ++q2) o += s_o[((size_t)q2 * G + g) * hd + e];
            p.att[(size_t)(split * n + node) * p.d + head * hd + e] = o;
            if (e == 0) {
                float m = -INFINITY, l = 0.f;
                for (int w = g; w < kSpWarps; w += G) { m = fmaxf(m, sh.m[w]); l += sh.l[w]; }
                p.att_ml[(size_t)(split * n + node) * p.H + head] = make_float2(m, l);
            }
        }
        __syncthreads();
    }
}

template <int CPT>
__device__ __forceinline__ void attention_step(const SmallPass &p, SpShared &sh, float *smem, const AttnCut &cut, int layer)
{
    if (cut.nodes == 1) attention_tasks<1, CPT>(p, sh, smem, cut, layer);
    else attention_tasks<2, CPT>(p, sh, smem, cut, layer);
}

// ---- the pass. False when a barrier wait ran out.
__device__ __forceinline__ bool run_pass(const SmallPass &p, SpShared &sh, float *smem, GridBarrier &bar)
{
    const int tid = threadIdx.x, n = p.n_tree - p.n_old, d = p.d;
    const int gt = (int)blockIdx.x * kSpThreads + tid, n_threads = (int)gridDim.x * kSpThreads;
    // every CTA checks the tree itself, and all agree
    const int err = mask_table(sh.table, p.parent, p.tokens, p.n_tree, p.V);
    int stands = 0;
    if (p.keep_status) stands = *reinterpret_cast<volatile int32_t *>(p.status);     // written by an earlier launch
    else if (gt == 0) *p.status = err;
    if (err || stands) {
        if (gt == 0 && p.keep_status && err) atomicCAS(p.status, 0, err);
        if (p.verify && blockIdx.x == 0) report_refused(p.P, p.path_fill, p.path, p.scalars);
        return true;
    }
    auto weights = [&](size_t off) { return reinterpret_cast<const float *>(p.base + off); };
    for (int i = gt; i < n * d; i += n_threads) {
        const int node = i / d, k = i - node * d;
        p.x[i] = __ldg(weights(p.tok_embed) + (size_t)__ldg(p.tokens + p.n_old + node) * d + k);
    }
    for (int i = gt; i < n * (p.hd / 2); i += n_threads) {
        const int node = i / (p.hd / 2), t = i - node * (p.hd / 2);
        double sn, cs;
        sincos((double)(p.P + mask_depth(sh.table.anc[p.n_old + node])) * p.inv_freq[t], &sn, &cs);
        p.rope_cs[i] = make_float2((float)cs, (float)sn);
    }
    if (gt < LLMCAD_MAX_TREE) p.best[gt] = 0;
    for (int i = tid; i < LLMCAD_MAX_TREE; i += kSpThreads) sh.best[i] = 0;

    const AttnCut cut = attn_cut(p);
    // the GEMM steps in order, four per layer, then the lm_head; attention runs before the second of each layer
    for (int step = 0; step < 4 * p.L + (p.logits != nullptr ? 1 : 0); ++step) {
        const int l = step >> 2;
        const size_t lb = p.layer_bytes * (size_t)l;
        Gemm g{weights(p.lm_head), p.V, d, weights(p.final_norm), 1, l, EPI_PLAIN, SRC_NORM};
        if (l < p.L) {
            switch (step & 3) {
            case 0: g = Gemm{weights(lb + p.wqkv), 3 * d, d, weights(lb + p.attn_norm), 1, l, EPI_QKV, SRC_NORM}; break;
            case 1: g = Gemm{weights(lb + p.wo), d, d, nullptr, cut.splits, l, EPI_RESID, SRC_ATT}; break;
            case 2: g = Gemm{weights(lb + p.wgu), p.f, d, weights(lb + p.ffn_norm), 1, l, EPI_SWIGLU, SRC_NORM}; break;
            default: g = Gemm{weights(lb + p.wdown), d, p.f, nullptr, 1, l, EPI_RESID, SRC_PLAIN}; break;
            }
        }
        if (g.src == SRC_ATT) {
            if (!bar.sync(sh)) return false;
            if (p.hd == 64) attention_step<2>(p, sh, smem, cut, l);
            else attention_step<4>(p, sh, smem, cut, l);
        }
        if (!gemm_step(p, g, sh, smem, bar)) return false;
    }
    if (p.logits == nullptr) return true;
    if (p.verify) {
        __syncthreads();
        for (int i = tid; i < n; i += kSpThreads)
            if (sh.best[i] != 0) atomicMax(p.best + i, sh.best[i]);
    }
    if (!p.verify && p.top_k == 0) return true;
    if (!bar.sync(sh)) return false;
    if (p.top_k > 0) {
        for (int i = (int)blockIdx.x; i < n; i += (int)gridDim.x)
            topk_row<kSpThreads, 8>(sh.topk, p.logits + (size_t)i * p.V, p.V, p.top_k, p.topk_ids + (size_t)i * p.top_k,
                                    p.topk_probs + (size_t)i * p.top_k, p.status);
    }
    if (!p.verify) return true;
    auto best_of = [&](int i) { return unpack_best(__ldcg(p.best + i)); };
    if (blockIdx.x == 0)
        for (int i = tid; i < n; i += kSpThreads) p.argmax[i] = best_of(i);
    if (*reinterpret_cast<volatile int32_t *>(p.status)) {          // a logit was NaN
        if (blockIdx.x == 0) report_refused(p.P, p.path_fill, p.path, p.scalars);
        return true;
    }
    path_search(sh.search, p.parent, p.tokens, best_of, n, blockIdx.x == 0);
    if (blockIdx.x == 0) report_path(sh.search, best_of, p.P, p.path_fill, p.path, p.scalars);
    const int chunks = p.hd / 4;
    for (int w = gt; w < p.L * 2 * p.H * chunks; w += n_threads) {
        const int lkh = w / chunks, ch = w - lkh * chunks;
        rollback_column(reinterpret_cast<uint4 *>(p.kv) + ((size_t)lkh * p.S + p.P) * chunks + ch, chunks, sh.search.path, sh.search.len);
    }
    return true;
}

}  // namespace

__global__ void __launch_bounds__(kSpThreads, 1)
small_pass_kernel(const __grid_constant__ SmallPass p)
{
    extern __shared__ __align__(16) float smem[];
    __shared__ SpShared sh;
    if (threadIdx.x == 0) sh.abort_flag = 0;
    GridBarrier bar{p.bar, 0, p.wait_limit_ns, p.status};
    const bool ok = run_pass(p, sh, smem, bar);
    if (!ok && p.verify && blockIdx.x == 0) report_refused(p.P, p.path_fill, p.path, p.scalars);
    // the last CTA to leave puts the barrier words back to zero for the next launch
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(p.bar + 1, 1u) == gridDim.x - 1) {
            p.bar[0] = 0;
            p.bar[1] = 0;
        }
    }
}

// Whether a pass fits: eight rows of the widest GEMM input staged, the scores of two nodes beside the partial
// outputs, the merge factors. There is no lower or upper line on the work: the other fp32 path runs plain FMAs too.
bool small_pass_serves(int d, int f, int hd, int H, int n_keys)
{
    const int widest = d > f ? d : f;
    return 8 * (size_t)widest * sizeof(float) <= kSpSmem && H <= kSpMaxAttW / LLMCAD_MAX_TREE &&
           sizeof(float) * 2 * ((size_t)(kSpThreads / (hd / 4)) * hd + n_keys) <= kSpSmem;
}

cudaError_t launch_small_pass(const SmallPass &p, int n_sms, cudaStream_t st)
{
    static PerDeviceOnce attr_set;
    if (attr_set.needed()) {
        const cudaError_t e = cudaFuncSetAttribute(small_pass_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSpSmem);
        if (e != cudaSuccess) return e;
        attr_set.mark();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_sms);
    cfg.blockDim = dim3(kSpThreads);
    cfg.dynamicSmemBytes = kSpSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, small_pass_kernel, p);
}

}  // namespace llmcad
