// Top-k of one row of logits with softmax probabilities, by one block (Sec. 3.2: a candidate above a
// confidence threshold opens a branch). Shared by the stand-alone kernel and by the small-model pass.
//
// What bounds it is round trips: the row is read once, into registers (up to kRegs values a thread), and the
// k rounds only compare what the threads hold: a thread knows its best value that has not been taken, a round
// finds the best of those over the block, and only the thread that owned the winner looks for its next one.
// Rows too long for the registers are read again from L2 where a thread has to look for its next best.
#pragma once

#include "common.cuh"

namespace llmcad {

struct TopkSmem {
    float v[32];
    int i[32];
    float best_v, sum;
    int best_i;
};

__device__ __forceinline__ void argmax_take(float v, int t, float &best, int &bi, bool &nan)
{
    nan |= (v != v);
    if (v > best || (v == best && t < bi)) { best = v; bi = t; }
}

// Largest value over the block, ties to the lower index; the same in every thread.
template <int THREADS>
__device__ __forceinline__ void block_argmax(TopkSmem &s, float v, int i, float &out_v, int &out_i)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, v, o);
        const int oi = __shfl_xor_sync(0xffffffffu, i, o);
        if (ov > v || (ov == v && oi < i)) { v = ov; i = oi; }
    }
    if (lane == 0) { s.v[warp] = v; s.i[warp] = i; }
    __syncthreads();
    if (warp == 0) {
        v = lane < THREADS / 32 ? s.v[lane] : -INFINITY;
        i = lane < THREADS / 32 ? s.i[lane] : 0x7fffffff;
        for (int o = 16; o; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, v, o);
            const int oi = __shfl_xor_sync(0xffffffffu, i, o);
            if (ov > v || (ov == v && oi < i)) { v = ov; i = oi; }
        }
        if (lane == 0) { s.best_v = v; s.best_i = i; }
    }
    __syncthreads();
    out_v = s.best_v; out_i = s.best_i;
}

// ids[k], probs[k]: descending, ties to the lower id; a NaN in the row sets *status.
template <int THREADS, int kRegs>
__device__ __forceinline__ void topk_row(TopkSmem &s, const float *row, int vocab, int k, int32_t *ids, float *probs, int32_t *status)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool held = vocab <= kRegs * THREADS;
    float x[kRegs];
    float best = -INFINITY;
    int bi = 0x7fffffff;
    bool nan = false;
#pragma unroll
    for (int u = 0; u < kRegs; ++u) x[u] = tid + u * THREADS < vocab ? __ldcg(row + tid + u * THREADS) : -INFINITY;
#pragma unroll
    for (int u = 0; u < kRegs; ++u)
        if (tid + u * THREADS < vocab) argmax_take(x[u], tid + u * THREADS, best, bi, nan);
    for (int t = tid + kRegs * THREADS; t < vocab; t += THREADS) argmax_take(__ldcg(row + t), t, best, bi, nan);
    if (nan) atomicCAS(status, 0, LLMCAD_ERR_NAN);

    float bv; int bidx;
    block_argmax<THREADS>(s, best, bi, bv, bidx);
    const float mx = bv;
    float sum = 0.f;
#pragma unroll
    for (int u = 0; u < kRegs; ++u)
        if (tid + u * THREADS < vocab) sum += expf(x[u] - mx);
    for (int t = tid + kRegs * THREADS; t < vocab; t += THREADS) sum += expf(__ldcg(row + t) - mx);
    for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) s.v[warp] = sum;
    __syncthreads();
    if (warp == 0) {
        float t = lane < THREADS / 32 ? s.v[lane] : 0.f;
        for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) s.sum = t;
    }
    __syncthreads();
    const float inv = 1.0f / s.sum;

    // a thread's own values in the order it would give them up: everything before (last_v, last_i) is taken
    for (int r = 0; r < k; ++r) {
        if (r > 0) block_argmax<THREADS>(s, best, bi, bv, bidx);
        if (tid == 0) {
            ids[r] = bidx == 0x7fffffff ? 0 : bidx;
            probs[r] = expf(bv - mx) * inv;
        }
        if (bidx == bi && r + 1 < k) {          // mine: the next one is the largest below (bv, bidx) in the order of the result
            best = -INFINITY;
            bi = 0x7fffffff;
            auto next = [&](float v, int t) {
                const bool left = v < bv || (v == bv && t > bidx);
                if (left && (v > best || (v == best && t < bi))) { best = v; bi = t; }
            };
            if (held) {
#pragma unroll
                for (int u = 0; u < kRegs; ++u)
                    if (tid + u * THREADS < vocab) next(x[u], tid + u * THREADS);
            } else {
                for (int t = tid; t < vocab; t += THREADS) next(__ldcg(row + t), t);
            }
        }
    }
    __syncthreads();
}

}  // namespace llmcad
