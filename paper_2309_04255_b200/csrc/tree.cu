// Integer side of the pass: mask table, embedding gather, argmax, verified-path search,
// cache rollback. Everything here is bit-exact by construction.
#include "common.cuh"
#include "topk_dev.cuh"
#include "tree_dev.cuh"

namespace llmcad {

// ------------------------------------------------------------------------------------------
// Start of a pass: mask table (Sec. 3.2 "Tree decoder") and embedding gather in one kernel, block i = node
// i. Every block checks the whole tree itself (n <= 128 links and tokens, one load each), so that all of
// them agree on the outcome without talking to each other, and block 0 states it in the status word: no
// memset and no second kernel in front of the first GEMM. `keep` (later chunks of a prefill) leaves a
// status word set by an earlier phase alone. Nodes from n_old on also get their rotary table row, in fp64
// at position prefix_len + depth, their row of the residual stream and, with gain != null (the tensor-core
// path folds the first RMSNorm into the QKV GEMM), gain * x as a GEMM input (hi and, if comp, lo plane)
// and the row's sum of squares.
//
// This kernel lets its dependents go only after its own dependency has resolved: the first GEMM requests
// weights before its own, and those may have been written right before the call, on this stream.
template <typename T>
__global__ void __launch_bounds__(256)
prep_embed_kernel(const int32_t *__restrict__ parent, const int32_t *__restrict__ tokens, int n_tree, int n_old, int P, int vocab,
                  int hd, const double *__restrict__ inv_freq, TreeBuffers tb, const T *__restrict__ E, int d,
                  const T *__restrict__ gain, float *x, T *xg, float *ssq, int comp, int32_t *status, int keep)
{
    __shared__ MaskTable t;
    __shared__ float red[8];
    const int i = blockIdx.x;
    pdl_wait();
    pdl_launch_dependents();
    const int err = mask_table(t, parent, tokens, n_tree, vocab);
    if (i == 0 && threadIdx.x == 0) {
        if (!keep) *status = err;
        else if (err) atomicCAS(status, 0, err);
    }
    const uint32_t row_bits[4] = {t.anc[i][0], t.anc[i][1], t.anc[i][2], t.anc[i][3]};
    const int depth = err ? 0 : mask_depth(row_bits);
    if (threadIdx.x == 0) {
        tb.depth[i] = depth;
        tb.pos[i] = P + depth;
#pragma unroll
        for (int w = 0; w < 4; ++w) tb.anc[i * 4 + w] = row_bits[w];
    }
    if (E == nullptr || i < n_old || err || (keep && *reinterpret_cast<volatile int32_t *>(status))) return;
    const double p = (double)(P + depth);
    for (int k = threadIdx.x; k < hd / 2; k += 256) {
        double sn, cs;
        sincos(p * inv_freq[k], &sn, &cs);
        tb.rope_cs[(size_t)i * (hd / 2) + k] = make_float2((float)cs, (float)sn);
    }
    const int r = i - n_old;
    const T *row = E + (size_t)__ldg(tokens + i) * d;
    float ss = 0.f;
    for (int k = threadIdx.x; k < d; k += 256) {
        const float v = to_f32<T>(row[k]);
        x[(size_t)r * d + k] = v;
        if (gain != nullptr) {
            store_split<T>(xg + (size_t)r * d + k, (size_t)kLoRows * d, v * to_f32<T>(gain[k]), comp != 0);
            ss += v * v;
        }
    }
    if (gain == nullptr) return;
    for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    if (threadIdx.x == 0) {
        float tot = 0.f;
        for (int w = 0; w < 8; ++w) tot += red[w];
        ssq[r] = tot;
    }
}

cudaError_t launch_tree_prep(const int32_t *parent, const int32_t *tokens, int n, int P, int vocab, TreeBuffers tb, int32_t *status,
                             cudaStream_t st)
{
    LaunchCfg lc(n, 256, 0, st);
    return cudaLaunchKernelEx(&lc.cfg, prep_embed_kernel<float>, parent, tokens, n, 0, P, vocab, 0, (const double *)nullptr, tb,
                              (const float *)nullptr, 0, (const float *)nullptr, (float *)nullptr, (float *)nullptr, (float *)nullptr, 0,
                              status, 0);
}

cudaError_t launch_prep_embed(const int32_t *parent, const int32_t *tokens, int n_tree, int n_old, int P, int vocab, int hd,
                              const double *inv_freq, TreeBuffers tb, const void *E, int dtype, int d, const void *gain, float *x,
                              void *xg, float *ssq, int comp, int32_t *status, int keep, cudaStream_t st)
{
    LaunchCfg lc(n_tree, 256, 0, st);
    if (dtype == LLMCAD_F32)
        return cudaLaunchKernelEx(&lc.cfg, prep_embed_kernel<float>, parent, tokens, n_tree, n_old, P, vocab, hd, inv_freq, tb,
                                  (const float *)E, d, (const float *)gain, x, (float *)xg, ssq, comp, status, keep);
    return cudaLaunchKernelEx(&lc.cfg, prep_embed_kernel<__nv_bfloat16>, parent, tokens, n_tree, n_old, P, vocab, hd, inv_freq, tb,
                              (const __nv_bfloat16 *)E, d, (const __nv_bfloat16 *)gain, x, (__nv_bfloat16 *)xg, ssq, comp, status, keep);
}

// Start of a prompt chunk of more than 128 tokens, block i = token i; as above with the tree known to be a chain.
__global__ void __launch_bounds__(256)
chain_embed_kernel(const int32_t *__restrict__ tokens, int n, int P, int vocab, int hd, const double *__restrict__ inv_freq, TreeBuffers tb,
                   const __nv_bfloat16 *__restrict__ E, int d, const __nv_bfloat16 *__restrict__ gain, float *x, __nv_bfloat16 *xg, float *ssq,
                   int32_t *status, int keep)
{
    __shared__ float red[8];
    const int i = blockIdx.x;
    pdl_wait();
    pdl_launch_dependents();
    int bad = 0;
    for (int c = threadIdx.x; c < n; c += 256) { const int tk = __ldg(tokens + c); bad |= tk < 0 || tk >= vocab; }
    const int err = __syncthreads_or(bad) ? LLMCAD_ERR_BAD_TOKEN : 0;
    if (i == 0 && threadIdx.x == 0) {
        if (!keep) *status = err;
        else if (err) atomicCAS(status, 0, err);
    }
    if (i < LLMCAD_MAX_TREE && threadIdx.x < 4) {
        const int left = i + 1 - 32 * (int)threadIdx.x;      // bits 0 .. i of the row
        tb.anc[i * 4 + threadIdx.x] = left >= 32 ? 0xffffffffu : (left <= 0 ? 0u : (1u << left) - 1u);
    }
    if (err || (keep && *reinterpret_cast<volatile int32_t *>(status))) return;
    for (int k = threadIdx.x; k < hd / 2; k += 256) {
        double sn, cs;
        sincos((double)(P + i) * inv_freq[k], &sn, &cs);
        tb.rope_cs[(size_t)i * (hd / 2) + k] = make_float2((float)cs, (float)sn);
    }
    const __nv_bfloat16 *row = E + (size_t)__ldg(tokens + i) * d;
    float ss = 0.f;
    for (int k = threadIdx.x; k < d; k += 256) {
        const float v = __bfloat162float(row[k]);
        x[(size_t)i * d + k] = v;
        store_split<__nv_bfloat16>(xg + (size_t)i * d + k, (size_t)kLoRows * d, v * __bfloat162float(gain[k]), true);
        ss += v * v;
    }
    for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    if (threadIdx.x == 0) {
        float tot = 0.f;
        for (int w = 0; w < 8; ++w) tot += red[w];
        ssq[i] = tot;
    }
}

cudaError_t launch_chain_embed(const int32_t *tokens, int n, int P, int vocab, int hd, const double *inv_freq, TreeBuffers tb, const void *E,
                               int d, const void *gain, float *x, void *xg, float *ssq, int32_t *status, int keep, cudaStream_t st)
{
    LaunchCfg lc(n, 256, 0, st);
    return cudaLaunchKernelEx(&lc.cfg, chain_embed_kernel, tokens, n, P, vocab, hd, inv_freq, tb, (const __nv_bfloat16 *)E, d,
                              (const __nv_bfloat16 *)gain, x, (__nv_bfloat16 *)xg, ssq, status, keep);
}

// ------------------------------------------------------------------------------------------
// RMSNorm of the fp32 residual stream into the GEMM input dtype. One block per node; the row is
// read once with 16-byte loads and kept in registers between the reduction and the scaling
// (rows longer than 4 * kNormVec * blockDim fall back to re-reading).
constexpr int kNormThreads = 512;
constexpr int kNormVec = 4;   // float4 per thread held in registers -> d <= 8192

template <typename T> __device__ __forceinline__ void store4(T *p, float a, float b, float c, float d);
template <> __device__ __forceinline__ void store4<float>(float *p, float a, float b, float c, float d)
{
    *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d);
}
template <> __device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16 *p, float a, float b, float c, float d)
{
    __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
    uint2 u;
    u.x = *reinterpret_cast<uint32_t *>(&lo);
    u.y = *reinterpret_cast<uint32_t *>(&hi);
    *reinterpret_cast<uint2 *>(p) = u;
}

template <typename T>
__global__ void __launch_bounds__(kNormThreads)
rmsnorm_kernel(const float *__restrict__ x, const T *__restrict__ g, int d, float eps, T *__restrict__ out,
               const int32_t *status)
{
    pdl_launch_dependents();
    pdl_wait();
    if (*status) return;
    __shared__ float red[kNormThreads / 32];
    const int i = blockIdx.x, tid = threadIdx.x;
    const float4 *xi = reinterpret_cast<const float4 *>(x + (size_t)i * d);
    const int nv = d >> 2;                      // d is a multiple of 8
    float4 r[kNormVec];
    float ss = 0.f;
#pragma unroll
    for (int u = 0; u < kNormVec; ++u) {
        const int k = tid + u * kNormThreads;
        r[u] = k < nv ? __ldcg(xi + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        ss += r[u].x * r[u].x + r[u].y * r[u].y + r[u].z * r[u].z + r[u].w * r[u].w;
    }
    for (int k = tid + kNormVec * kNormThreads; k < nv; k += kNormThreads) {
        const float4 t = __ldcg(xi + k);
        ss += t.x * t.x + t.y * t.y + t.z * t.z + t.w * t.w;
    }
    for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if ((tid & 31) == 0) red[tid >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < kNormThreads / 32; ++w) tot += red[w];
    const float rs = rsqrtf(tot / d + eps);
    T *oi = out + (size_t)i * d;
#pragma unroll
    for (int u = 0; u < kNormVec; ++u) {
        const int k = tid + u * kNormThreads;
        if (k < nv) {
            const T *gk = g + 4 * k;
            store4<T>(oi + 4 * k, r[u].x * rs * to_f32<T>(gk[0]), r[u].y * rs * to_f32<T>(gk[1]),
                      r[u].z * rs * to_f32<T>(gk[2]), r[u].w * rs * to_f32<T>(gk[3]));
        }
    }
    for (int k = tid + kNormVec * kNormThreads; k < nv; k += kNormThreads) {
        const float4 t = __ldcg(xi + k);
        const T *gk = g + 4 * k;
        store4<T>(oi + 4 * k, t.x * rs * to_f32<T>(gk[0]), t.y * rs * to_f32<T>(gk[1]), t.z * rs * to_f32<T>(gk[2]),
                  t.w * rs * to_f32<T>(gk[3]));
    }
}

cudaError_t launch_rmsnorm(const float *x, const void *g, int dtype, int n, int d, float eps, void *out,
                           const int32_t *status, cudaStream_t st)
{
    LaunchCfg lc(n, kNormThreads, 0, st);
    if (dtype == LLMCAD_F32)
        return cudaLaunchKernelEx(&lc.cfg, rmsnorm_kernel<float>, x, (const float *)g, d, eps, (float *)out, status);
    return cudaLaunchKernelEx(&lc.cfg, rmsnorm_kernel<__nv_bfloat16>, x, (const __nv_bfloat16 *)g, d, eps,
                              (__nv_bfloat16 *)out, status);
}

// ------------------------------------------------------------------------------------------
// Greedy choice of the target at every node: lowest index of the maximum; a NaN sets status.
constexpr int kArgmaxThreads = 1024;

__global__ void __launch_bounds__(kArgmaxThreads)
argmax_kernel(const float *__restrict__ logits, int vocab, int32_t *argmax, int32_t *status)
{
    pdl_launch_dependents();
    pdl_wait();
    if (*status) return;
    __shared__ float s_v[32];
    __shared__ int s_i[32];
    const int i = blockIdx.x;
    const float *row = logits + (size_t)i * vocab;
    float best = -INFINITY;
    int bi = 0x7fffffff;
    bool nan = false;
    if ((vocab & 3) == 0) {
        const float4 *r4 = reinterpret_cast<const float4 *>(row);
        for (int t = threadIdx.x; t < (vocab >> 2); t += kArgmaxThreads) {
            const float4 q = __ldcg(r4 + t);
            argmax_take(q.x, 4 * t, best, bi, nan);
            argmax_take(q.y, 4 * t + 1, best, bi, nan);
            argmax_take(q.z, 4 * t + 2, best, bi, nan);
            argmax_take(q.w, 4 * t + 3, best, bi, nan);
        }
    } else {
        for (int t = threadIdx.x; t < vocab; t += kArgmaxThreads) argmax_take(row[t], t, best, bi, nan);
    }
    if (nan) atomicCAS(status, 0, LLMCAD_ERR_NAN);
    for (int o = 16; o; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
    }
    if ((threadIdx.x & 31) == 0) { s_v[threadIdx.x >> 5] = best; s_i[threadIdx.x >> 5] = bi; }
    __syncthreads();
    if (threadIdx.x < 32) {
        best = s_v[threadIdx.x];
        bi = s_i[threadIdx.x];
        for (int o = 16; o; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, best, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
        }
        if (threadIdx.x == 0) argmax[i] = (bi == 0x7fffffff) ? 0 : bi;
    }
}

cudaError_t launch_argmax(const float *logits, int n, int vocab, int32_t *argmax, int32_t *status, cudaStream_t st)
{
    LaunchCfg lc(n, kArgmaxThreads, 0, st);
    return cudaLaunchKernelEx(&lc.cfg, argmax_kernel, logits, vocab, argmax, status);
}

// ------------------------------------------------------------------------------------------
// Confidences of the generating side (topk_dev.cuh), one block per node. A row of 32000 logits sits in
// registers (32 a thread), where k rounds over L2 used to read it k + 2 times.
constexpr int kTopkThreads = 1024;

__global__ void __launch_bounds__(kTopkThreads)
topk_softmax_kernel(const float *__restrict__ logits, int vocab, int k, int32_t *ids, float *probs, int32_t *status)
{
    __shared__ TopkSmem s;
    pdl_launch_dependents();
    pdl_wait();
    if (*status) return;
    topk_row<kTopkThreads, 32>(s, logits + (size_t)blockIdx.x * vocab, vocab, k, ids + (size_t)blockIdx.x * k, probs + (size_t)blockIdx.x * k,
                               status);
}

cudaError_t launch_topk_softmax(const float *logits, int n, int vocab, int k, int32_t *ids, float *probs, int32_t *status,
                                cudaStream_t st)
{
    LaunchCfg lc(n, kTopkThreads, 0, st);
    return cudaLaunchKernelEx(&lc.cfg, topk_softmax_kernel, logits, vocab, k, ids, probs, status);
}

// ------------------------------------------------------------------------------------------
// Verified-sequence search and rollback (Sec. 3.2) in one kernel: every block finds the path itself (a few
// loads and some rounds in shared memory) and moves its own columns of the cache, block 0 also reports. As
// two kernels the second waited for the first only to read a dozen numbers. `check`: the tree has not been
// validated yet (the stand-alone call); otherwise an error of an earlier phase stands in the status word.
constexpr int kSearchThreads = 128;

__global__ void __launch_bounds__(kSearchThreads)
search_rollback_kernel(const int32_t *__restrict__ parent, const int32_t *__restrict__ tokens, const int32_t *argmax, int n, int P,
                       int vocab, int check, int32_t *path, int path_len, int32_t *scalars, uint4 *kv, int n_lkh, int S, int chunks)
{
    __shared__ union { MaskTable t; PathSearch s; } sh;
    pdl_launch_dependents();
    pdl_wait();
    int status;
    if (check) {
        status = mask_table(sh.t, parent, tokens, n, vocab);
        if (blockIdx.x == 0 && threadIdx.x == 0) scalars[LLMCAD_S_STATUS] = status;
    } else status = *reinterpret_cast<volatile int32_t *>(scalars + LLMCAD_S_STATUS);
    if (status) {  // report an empty result, leave the cache as it was
        if (blockIdx.x == 0) report_refused(P, path_len, path, scalars);
        return;
    }
    auto best_of = [&](int p) { return __ldcg(argmax + p); };
    path_search(sh.s, parent, tokens, best_of, n, blockIdx.x == 0);
    if (blockIdx.x == 0) report_path(sh.s, best_of, P, path_len, path, scalars);
    if (kv == nullptr) return;
    int len = sh.s.len;
    if (!LLMCAD_CHECK(len >= 1 && P + len <= S && len <= n, scalars + LLMCAD_S_STATUS)) return;
    for (int j = threadIdx.x; j < len; j += kSearchThreads)
        if (!LLMCAD_CHECK(sh.s.path[j] >= j && sh.s.path[j] < n, scalars + LLMCAD_S_STATUS)) len = 0;
    const long long w = (long long)blockIdx.x * kSearchThreads + threadIdx.x;
    if (w >= (long long)n_lkh * chunks) return;
    const int lkh = (int)(w / chunks), ch = (int)(w % chunks);
    rollback_column(kv + ((size_t)lkh * S + P) * chunks + ch, chunks, sh.s.path, len);
}

cudaError_t launch_search_rollback(const int32_t *parent, const int32_t *tokens, const int32_t *argmax, int n, int P, int vocab,
                                   int check, int32_t *path, int path_len, int32_t *scalars, void *kv, int dtype, int n_layers,
                                   int n_heads, int S, int hd, cudaStream_t st)
{
    const int elem = dtype == LLMCAD_F32 ? 4 : 2;
    const int chunks = hd * elem / 16;
    const int n_lkh = n_layers * 2 * n_heads;
    const long long total = kv != nullptr ? (long long)n_lkh * chunks : 1;
    const unsigned grid = (unsigned)((total + kSearchThreads - 1) / kSearchThreads);
    LaunchCfg lc(grid > 0 ? grid : 1, kSearchThreads, 0, st);
    return cudaLaunchKernelEx(&lc.cfg, search_rollback_kernel, parent, tokens, argmax, n, P, vocab, check, path, path_len, scalars,
                              (uint4 *)kv, n_lkh, S, chunks);
}

}  // namespace llmcad
