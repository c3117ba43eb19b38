// Weight-streaming skinny GEMMs on the sm_100a tensor cores.
//
// The one-shot verification of Sec. 3.2 visits every parameter once for all N <= 128 tree nodes,
// so each GEMM is D[n_out][N] = W[n_out][K] * X[N][K]^T with a tiny N: it is bound by the bytes
// of W coming from HBM. The streaming kernel therefore puts W on the M side of tcgen05.mma (128
// weight rows per tile = the 128 TMEM lanes) and the tree nodes on the N side (padded to a multiple
// of 16; with hi + lo activation planes the MMA sees every node twice), and streams W exactly once
// through a ring in shared memory: the weights are stored as pre-swizzled 16 KB tiles (pack.cu), so
// a ring item (one tile, two k-blocks) is one contiguous 32 KB bulk copy.
//
// A GEMM is two kernels, chained by programmatic dependent launch.
//
// gemm_stream_kernel: persistent grid, one CTA per SM. The (tile, k-block pair, half) items of the
// GEMM are split evenly over the CTAs (stream-K): a CTA's range may start and end inside a tile.
// For every tile that a CTA holds items of (a "segment") it leaves its accumulators, hi and lo
// columns added, in a workspace slot (slot = tile + CTA, unique because the CTAs' ranges are
// ordered), and exits. Nothing in it waits for another CTA.
//
// gemm_finish_kernel: all warps of the GPU add the segments of every tile in CTA order (so the
// result does not depend on timing) and apply the fused epilogue (rotary + K/V cache write,
// residual + the next norm's gain * x and sums of squares, SwiGLU, or plain fp32 rows). It needs
// next to no shared memory, so the NEXT GEMM's streaming CTAs become resident as soon as this
// GEMM's streaming CTAs leave, and fill their weight rings while the finishing runs: the HBM
// stream pauses only for as long as a ring lasts, not for the whole tail of a GEMM.
//
// Warp roles of the streaming kernel (224 threads): warp 0 = weight producer, warp 1 = TMEM
// allocator + MMA issuer, warps 2..5 = accumulator dump (tcgen05.ld of their 32 lanes each),
// warp 6 = activation loader (TMA). Accumulators are double-buffered in TMEM, so that the dump of one
// segment overlaps the MMAs of the next.
//
// Programmatic stream serialization: the ring is filled with weight tiles while the previous
// kernels of the pass are still running; activations and the workspace wait for the grid
// dependency. The streaming kernel lets its dependents go only after its own dependency has
// resolved, so the finishing kernel may read what earlier GEMMs produced (norm sums, gains) before
// its own dependency, the streaming kernel, completes. A status word left by an earlier phase is
// not looked at here: the GEMMs then work on stale but finite activations and write only scratch
// and tree slots, and the search/rollback kernels at the end of the pass report the error.
//
// Every wait of the streaming kernel (mbarriers only) is bounded by a deadline; on expiry the
// kernel sets the status word to LLMCAD_ERR_TIMEOUT, lets every role fall out of its loop, frees
// TMEM and returns.
#include <cuda.h>

#include <cstdlib>

#include "common.cuh"
#include "gemm_tc.cuh"
#include "mbar.cuh"

namespace llmcad {

namespace {

constexpr int kTileM = 128;     // weight rows per tile
constexpr int kBlockK = 64;     // bf16 elements per k-block = one 128-byte swizzle row
constexpr int kThreads = 224;   // producer, MMA issuer, 4 epilogue warps, activation loader
constexpr int kFinThreads = 384;  // finishing kernel: 12 warps, three per scheduler
// An SM's registers come in four banks of 16K, one per warp scheduler: beside the streaming CTA's two warps per
// scheduler (96 registers a thread) three finishing warps fit with up to 106 each.
constexpr int kFinMaxRegs = 96;
constexpr size_t kFinSmem = 24 * 1024;   // dynamic shared memory the finishing kernel asks for (and does not use):
                                         // it keeps two of its CTAs from settling on one SM, which would leave no room
                                         // there for the next GEMM's streaming CTA
constexpr int kATileBytes = kTileM * kBlockK * 2;  // 16 KB
constexpr int kMaxStages = 16;
constexpr int kMaxPairK = 2;     // k-blocks per ring item (GemmDesc::pair_k): 2 = one 32 KB weight copy feeds 8 MMAs;
                                 // 1 for wide activation tiles, which would leave too few ring stages otherwise

// ---------------------------------------------------------------- mbarrier
// Bounded wait: gives up after wait_limit ns or as soon as another role has raised `abort`.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, uint64_t wait_limit)
{
    if (mbar_try(bar, parity)) return true;
    uint64_t t0 = 0;
    for (uint32_t it = 1;; ++it) {
        // (try_wait itself suspends the thread for a while when the phase is not complete; a __nanosleep between the
        // tries, meant to leave issue slots to the warp that shares the scheduler, measured 0.6 % slower per pass)
        if (mbar_try(bar, parity)) return true;
        if ((it & 255u) == 0) {
            if (*abort_flag) return false;
            if (t0 == 0) t0 = global_timer_ns();
            else if (global_timer_ns() - t0 > wait_limit) return false;
        }
    }
}

// Whole-warp wait for roles that are not on the critical path of the weight stream: one lane
// polls and the warp follows. A warp of 32 pollers per barrier would saturate the shared-memory
// pipeline that the producer's copies and barrier operations also go through.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int *abort_flag, int lane, uint64_t wait_limit)
{
    int ok = 1;
    if (lane == 0 && !mbar_try(bar, parity)) {
        const uint64_t t0 = global_timer_ns();
        for (uint32_t it = 1;; ++it) {
            if (mbar_try(bar, parity)) break;
            if ((it & 63u) == 0 && (*abort_flag || global_timer_ns() - t0 > wait_limit)) { ok = 0; break; }
        }
    }
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

// ---------------------------------------------------------------- TMA
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar,
                                            uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%2, %3}], [%4], %5;"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(bar), "l"(policy)
        : "memory");
}

// Activation box (64 columns x rows x planes) at column c0, row 0, plane 0.
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int c0, uint32_t bar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%2, %3, %3}], [%4], %5;"
        ::"r"(dst), "l"(map), "r"(c0), "r"(0), "r"(bar), "l"(policy)
        : "memory");
}

// One contiguous run of global memory into shared memory (both 16-byte aligned, size a multiple of 16).
__device__ __forceinline__ void bulk_load_1d(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
        ::"r"(dst), "l"(src), "r"(bytes), "r"(bar), "l"(policy)
        : "memory");
}

// ---------------------------------------------------------------- tcgen05
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// D[tmem] (+)= A[smem] * B[smem]^T, bf16 inputs, fp32 accumulate, issued by one thread.
__device__ __forceinline__ void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// 16 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float *v)
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// 32 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float *v)
{
    uint32_t a[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]), "=r"(a[15]), "=r"(a[16]), "=r"(a[17]), "=r"(a[18]), "=r"(a[19]), "=r"(a[20]), "=r"(a[21]), "=r"(a[22]), "=r"(a[23]), "=r"(a[24]), "=r"(a[25]), "=r"(a[26]), "=r"(a[27]), "=r"(a[28]), "=r"(a[29]), "=r"(a[30]), "=r"(a[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(a[j]);
}

// 32 consecutive fp32 columns of this thread's TMEM lane at each of two addresses, summed. A load plus
// its wait costs ~0.15 us whatever the width, so the two loads share one wait; everything sits in one
// statement so that no register of the result can be touched before the wait.
__device__ __forceinline__ void tc_ld32_sum2(uint32_t taddr_a, uint32_t taddr_b, float *v)
{
    uint32_t a[32], b[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%64];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%65];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]), "=r"(a[15]), "=r"(a[16]), "=r"(a[17]), "=r"(a[18]), "=r"(a[19]), "=r"(a[20]), "=r"(a[21]), "=r"(a[22]), "=r"(a[23]), "=r"(a[24]), "=r"(a[25]), "=r"(a[26]), "=r"(a[27]), "=r"(a[28]), "=r"(a[29]), "=r"(a[30]), "=r"(a[31]), "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7]), "=r"(b[8]), "=r"(b[9]), "=r"(b[10]), "=r"(b[11]), "=r"(b[12]), "=r"(b[13]), "=r"(b[14]), "=r"(b[15]), "=r"(b[16]), "=r"(b[17]), "=r"(b[18]), "=r"(b[19]), "=r"(b[20]), "=r"(b[21]), "=r"(b[22]), "=r"(b[23]), "=r"(b[24]), "=r"(b[25]), "=r"(b[26]), "=r"(b[27]), "=r"(b[28]), "=r"(b[29]), "=r"(b[30]), "=r"(b[31])
        : "r"(taddr_a), "r"(taddr_b)
        : "memory");
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(a[j]) + __uint_as_float(b[j]);
}

// Shared-memory matrix descriptor: K-major tile of 128-byte rows, 128-byte swizzle, 8-row groups
// 1024 bytes apart (the layout a TMA box of 64 bf16 x rows with CU_TENSOR_MAP_SWIZZLE_128B
// produces). Fields: start address >> 4 [0,14), leading byte offset >> 4 [16,30) (unused for
// swizzled K-major, set to 1), stride byte offset >> 4 [32,46), version 1 [46,48), layout type
// [61,64) = 2 (128-byte swizzle).
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t smem_addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr >> 4) & 0x3fffu);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor of kind::f16: fp32 accumulator (bits 4-5 = 1), A and B bf16 (bits 7-9,
// 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22, M >> 4 at bits 24-28.
__host__ __device__ constexpr uint32_t make_idesc(int m, int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

struct SharedCtl {
    uint64_t full[kMaxStages];
    uint64_t empty[kMaxStages];
    uint64_t tmem_full[2];
    uint64_t tmem_empty[2];
    uint32_t tmem_base;
    volatile int abort_flag;
    volatile uint32_t a_issued;     // ring items whose weight copy (and expect_tx) has been issued
};

// A weight tile is 128 rows of the packed matrix. An output tile has one of them, or two (SwiGLU: gate and up),
// which are streamed one after the other like the tiles of different outputs: tile v belongs to output tile
// v / halves. A ring item is (tile, k-block pair): up to two consecutive 64-wide k-blocks of a tile (32 KB,
// contiguous in the tiled layout) and the matching activation tiles.
__host__ __device__ __forceinline__ int pairs_per_tile(const GemmDesc &g) { return (g.kb_per_tile + g.pair_k - 1) / g.pair_k; }
// the same with the k-blocks per item as a compile-time constant (the kernel is instantiated for 1 and 2)
template <int PK> __device__ __forceinline__ int pairs_per_tile_c(const GemmDesc &g) { return (g.kb_per_tile + PK - 1) / PK; }
// position of tile v in the packed matrix (all gate tiles, then all up tiles)
__host__ __device__ __forceinline__ int packed_tile(const GemmDesc &g, int v)
{
    return g.halves == 2 ? (v >> 1) + (v & 1) * g.up_tile_offset : v;
}

// CTA cta's share of the GEMM: items [begin, end) of its item list.
struct Range {
    int begin, end;
};
template <int PK>
__device__ __forceinline__ Range cta_range(const GemmDesc &g, int cta)
{
    const int total = g.n_tiles * g.halves * pairs_per_tile_c<PK>(g);
    Range r;
    r.begin = min(total, cta * g.items_per_cta);
    r.end = min(total, r.begin + g.items_per_cta);
    return r;
}

// Cursor over this CTA's items, in order. Coordinates are kept incrementally: the single-thread
// roles have well under a microsecond per item.
template <int PK>
struct Cursor {
    int tile, kp;          // coordinates of the current item (kp: k-block pair)
    int left;              // items left in this CTA's range, the current one included
    int ppt, kbpt;
    __device__ void init(const GemmDesc &d)
    {
        const Range r = cta_range<PK>(d, (int)blockIdx.x);
        left = r.end - r.begin;
        kbpt = d.kb_per_tile;
        ppt = pairs_per_tile_c<PK>(d);
        tile = r.begin / ppt;
        kp = r.begin - tile * ppt;
    }
    __device__ bool done() const { return left <= 0; }
    __device__ int kb0() const { return kp * PK; }
    __device__ int nk() const { return min(PK, kbpt - kp * PK); }   // k-blocks in this item
    __device__ void advance()
    {
        --left;
        if (++kp == ppt) { kp = 0; ++tile; }
    }
};

// Floats of one segment slot of the workspace: [4 row groups][n_pad / 4 node groups][32 rows][4 nodes], so that the
// dumping warps (thread = row) store four nodes at once: with one node per store the last segment of a CTA took 4-5 us
// to leave at 128-256 nodes, four times as many instructions.
__host__ __device__ __forceinline__ size_t slot_floats(int n_pad) { return (size_t)n_pad * kTileM; }

// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ void dump4(float *dst, const float *v) { *reinterpret_cast<float4 *>(dst) = make_float4(v[0], v[1], v[2], v[3]); }

// Finishing (the work of gemm_finish_kernel). Every streaming CTA that holds items of a tile has left
// its accumulators in the workspace as [row group][node group][32 rows][4 nodes] fp32 (a "segment").
// A warp reads a node group with lane = row; turned so that a lane has four rows of one node (below):
// four rounds of shuffles, in which lane L = 4r + k sends the value of node k - s in round s.
__device__ __forceinline__ float4 rotate4(float4 v, int by)       // component j of the result = component (j - by) mod 4
{
    if (by & 1) v = make_float4(v.w, v.x, v.y, v.z);
    if (by & 2) v = make_float4(v.z, v.w, v.x, v.y);
    return v;
}
__device__ __forceinline__ float4 rows_of_node(float4 v, int lane)
{
    const int ns = lane >> 3, from = 4 * (lane & 7);
    const float4 r = rotate4(make_float4(v.x, v.w, v.z, v.y), lane & 3);
    float4 g;
    g.x = __shfl_sync(0xffffffffu, r.x, from + (ns & 3));
    g.y = __shfl_sync(0xffffffffu, r.y, from + ((ns + 1) & 3));
    g.z = __shfl_sync(0xffffffffu, r.z, from + ((ns + 2) & 3));
    g.w = __shfl_sync(0xffffffffu, r.w, from + ((ns + 3) & 3));
    return rotate4(g, ns);
}

__device__ __forceinline__ uint2 pack4_bf16(const __nv_bfloat16 (&h)[4])
{
    uint2 r;
    r.x = (uint32_t)__bfloat16_as_ushort(h[0]) | ((uint32_t)__bfloat16_as_ushort(h[1]) << 16);
    r.y = (uint32_t)__bfloat16_as_ushort(h[2]) | ((uint32_t)__bfloat16_as_ushort(h[3]) << 16);
    return r;
}

// Where CTA (or CTA pair) cc left its segment of tile v, rows of row group lane_grp: slot v + cc (v + 2 cc).
__device__ __forceinline__ const float *share_ptr(const GemmParams &p, const GemmDesc &d, int cc, int v, int lane_grp)
{
    return p.partials + (size_t)(v + d.group * cc) * slot_floats(p.n_pad) + (size_t)lane_grp * p.n_pad * 32;
}

// The CTAs (pairs) that hold items of tile v: first .. first + n - 1.
struct Holders {
    int first, n;
};
__device__ __forceinline__ Holders holders_of(const GemmDesc &d, int ppt, int v)
{
    Holders h;
    const int t = d.group == 2 ? v >> 1 : v;
    h.first = t * ppt / d.items_per_cta;
    h.n = ((t + 1) * ppt - 1) / d.items_per_cta - h.first + 1;
    return h;
}

// What a warp of the finishing kernel works on.
struct FinishArgs {
    const GemmParams *p;
    const GemmDesc *d;              // in shared memory
    const float *rs;                // per-node factors of the folded input norm (shared memory)
    int tile, lane_grp;             // output tile, 32-row group
    Holders a, b;                   // who holds it (b: the up projection of a SwiGLU)
    int it_first, it_step;          // this warp finishes node groups it_first, it_first + it_step, ...
};

// Finishing a 32-row group of an output tile: add the segments of all CTAs that hold part of the
// tile, in CTA order (so the result does not depend on timing), and apply the fused epilogue. What
// this costs is the length of its dependent chain, round trips to L2 and plain instruction latency,
// not bytes. Hence: lane = (node sub-index ns = lane / 8, row quad r4 = lane % 8), iteration `it`
// handles the four output rows 4 * r4 .. + 3 of node 4 * it + ns (after rows_of_node), everything moves as 16- or 8-byte
// vectors, a rotary pair sits in one thread; the iterations of a group are dealt out to several
// warps of the grid (it_first, it_step); G node groups travel together and kB segments of each are
// loaded at a time, all loads issued before the first use. With `dry` nothing is stored: the
// finishing kernel walks through its code once that way before its input exists (see there).
// One instantiation per epilogue mode: the code is cold whenever it runs, and what that costs is
// the code walked through, not the code that exists.
template <int G, int kB, int MODE>
__device__ __forceinline__ void finish_rows_t(const FinishArgs &fa, int lane, const bool dry)
{
    typedef __nv_bfloat16 T;
    const GemmParams &p = *fa.p;
    const GemmDesc &d = *fa.d;
    const EpiParams &ep = d.ep;
    constexpr int mode = MODE;
    const int n_nodes = ep.n, n_out = ep.n_out, n_pad = p.n_pad;
    constexpr bool dual = MODE == EPI_SWIGLU;      // the one mode with two accumulators per tile (gate, up)
    const bool comp = ep.comp != 0, has_rs = ep.ssq_in != nullptr, has_xg = ep.xg_out != nullptr;
    constexpr bool resid = mode == EPI_RESID;
    const int tile = fa.tile, lane_grp = fa.lane_grp;
    const int ns = lane >> 3, r4 = lane & 7;
    const int row0 = tile * kTileM + lane_grp * 32 + 4 * r4;   // first of this lane's four output rows
    const int n_valid = min(4, n_out - row0);                  // how many of them exist
    const bool rows_ok = n_valid == 4;                         // all modes but EPI_PLAIN have n_out % 4 == 0
    const int n_parts = dual ? max(fa.a.n, fa.b.n) : fa.a.n;
    const int va = dual ? 2 * tile : tile;                     // the tile (of the gate; the up projection's is the next)
    if (!LLMCAD_CHECK(fa.a.first >= 0 && d.group * (fa.a.first + fa.a.n) <= d.grid && tile < d.n_tiles && row0 >= 0, p.status)) return;
    if (mode == EPI_QKV && !LLMCAD_CHECK(ep.P + n_nodes <= ep.S && row0 < 3 * ep.d, p.status)) return;

    // per-lane constants of the mode
    float gain[4] = {0.f, 0.f, 0.f, 0.f};
    int sec = 0, head = 0, e = 0, cidx = 0;
    if (resid && has_xg && rows_ok) {
        const uint2 g4 = __ldg(reinterpret_cast<const uint2 *>(reinterpret_cast<const T *>(ep.gain_next) + row0));
        gain[0] = __uint_as_float(g4.x << 16); gain[1] = __uint_as_float(g4.x & 0xffff0000u);
        gain[2] = __uint_as_float(g4.y << 16); gain[3] = __uint_as_float(g4.y & 0xffff0000u);
    } else if (mode == EPI_QKV) {
        sec = row0 / ep.d; cidx = row0 - sec * ep.d;
        head = cidx / ep.hd; e = cidx - head * ep.hd;
    }
    // what a node's epilogue reads besides the shares: the residual (EPI_RESID) or the rotary
    // (cos, sin) of the lane's two pairs (EPI_QKV, q and k sections)
    const float *aux = nullptr;
    int aux_stride = 0;
    if (rows_ok && resid) { aux = ep.x + row0; aux_stride = n_out; }
    if (rows_ok && mode == EPI_QKV && sec < 2) { aux = reinterpret_cast<const float *>(ep.rope_cs) + 2 * (e >> 1); aux_stride = ep.hd; }
    const float4 aux_none = resid ? make_float4(0.f, 0.f, 0.f, 0.f) : make_float4(1.f, 0.f, 1.f, 0.f);
    // where a node's outputs go in the activation format: hi and lo plane, the same stride per node. Queries get a lo
    // plane; keys and values go to the cache rounded, their remainders to kv_lo.
    T *hi_at = nullptr, *lo_at = nullptr;
    int out_stride = n_out;
    if (resid && has_xg) hi_at = reinterpret_cast<T *>(ep.xg_out) + row0;
    else if (mode == EPI_SWIGLU) hi_at = reinterpret_cast<T *>(ep.h) + row0;
    else if (mode == EPI_QKV && sec == 0) { hi_at = reinterpret_cast<T *>(ep.q_out) + cidx; out_stride = ep.d; }
    if (hi_at != nullptr) lo_at = hi_at + (size_t)kLoRows * out_stride;
    if (mode == EPI_QKV && sec > 0) {
        out_stride = ep.hd;
        hi_at = reinterpret_cast<T *>(sec == 1 ? ep.k_cache : ep.v_cache) + ((size_t)head * ep.S + ep.P) * ep.hd + e;
        lo_at = reinterpret_cast<T *>(ep.kv_lo) + (size_t)((sec - 1) * (ep.d / ep.hd) + head) * kLoRows * ep.hd + e;
    }
    if (!comp) lo_at = nullptr;
    const bool y_vec = mode == EPI_PLAIN && rows_ok && (ep.ldy & 3) == 0 && (reinterpret_cast<uintptr_t>(ep.y) & 15) == 0;

    const int iters = n_pad >> 2;
    for (int itg = fa.it_first; itg < iters; itg += G * fa.it_step) {
        // every load of the G iterations is issued before the first use
        float4 axs[G], as[G], bs[G];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int node = min(itg + g * fa.it_step, iters - 1) * 4 + ns;
            axs[g] = aux_none;
            if (aux != nullptr && node < n_nodes) axs[g] = __ldcg(reinterpret_cast<const float4 *>(aux + (size_t)node * aux_stride));
            as[g] = bs[g] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int k0 = 0; k0 < n_parts; k0 += kB) {
            float4 t[G][kB], u[G][kB];
#pragma unroll
            for (int k = 0; k < kB; ++k) {
                // (no load for a holder that does not exist: at many nodes the segments' bytes are what this costs)
                const bool has = k0 + k < fa.a.n, has_u = dual && k0 + k < fa.b.n;
                const float *sk = share_ptr(p, d, fa.a.first + k0 + k, va, lane_grp) + 4 * lane;
                const float *su = dual ? share_ptr(p, d, fa.b.first + k0 + k, va + 1, lane_grp) + 4 * lane : nullptr;
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const int it = min(itg + g * fa.it_step, iters - 1);
                    t[g][k] = has ? __ldcg(reinterpret_cast<const float4 *>(sk + (size_t)it * 128)) : make_float4(0.f, 0.f, 0.f, 0.f);
                    if (dual) u[g][k] = has_u ? __ldcg(reinterpret_cast<const float4 *>(su + (size_t)it * 128)) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
#pragma unroll
            for (int k = 0; k < kB; ++k) {
                // CTA order
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    as[g].x += t[g][k].x; as[g].y += t[g][k].y; as[g].z += t[g][k].z; as[g].w += t[g][k].w;
                    if (dual) { bs[g].x += u[g][k].x; bs[g].y += u[g][k].y; bs[g].z += u[g][k].z; bs[g].w += u[g][k].w; }
                }
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int it = itg + g * fa.it_step;
            if (it >= iters) break;
            const int node = it * 4 + ns;
            const bool ok = rows_ok && node < n_nodes;
            const float4 ax = axs[g], a = rows_of_node(as[g], lane);
            float4 b;
            if (dual) b = rows_of_node(bs[g], lane);
            const float r = has_rs ? fa.rs[node] : 1.f;
            const float v[4] = {a.x * r, a.y * r, a.z * r, a.w * r};
            float out[4];                 // what goes out in the activation format (hi and lo plane)
            if (resid) {
                const float xo[4] = {ok ? ax.x + v[0] : 0.f, ok ? ax.y + v[1] : 0.f, ok ? ax.z + v[2] : 0.f, ok ? ax.w + v[3] : 0.f};
                if (ok && !dry) *reinterpret_cast<float4 *>(ep.x + (size_t)node * n_out + row0) = make_float4(xo[0], xo[1], xo[2], xo[3]);
#pragma unroll
                for (int k = 0; k < 4; ++k) out[k] = xo[k] * gain[k];
                if (has_xg) {
                    // what the next RMSNorm needs: gain * x in the GEMM input format, and this row
                    // group's share of every node's sum of squares
                    float ss = xo[0] * xo[0] + xo[1] * xo[1] + xo[2] * xo[2] + xo[3] * xo[3];
                    ss += __shfl_xor_sync(0xffffffffu, ss, 1);
                    ss += __shfl_xor_sync(0xffffffffu, ss, 2);
                    ss += __shfl_xor_sync(0xffffffffu, ss, 4);
                    if (r4 == 0 && !dry) ep.ssq_out[(size_t)(tile * 4 + lane_grp) * kLoRows + node] = ss;
                }
            } else if (mode == EPI_SWIGLU) {
#pragma unroll
                for (int k = 0; k < 4; ++k) out[k] = v[k] / (1.0f + __expf(-v[k]));
                out[0] *= b.x * r; out[1] *= b.y * r; out[2] *= b.z * r; out[3] *= b.w * r;
            } else if (mode == EPI_QKV) {
                // rotary pairs (2t, 2t+1) = (v0, v1), (v2, v3); values pass through with (cos, sin) = (1, 0)
                out[0] = v[0] * ax.x - v[1] * ax.y; out[1] = v[0] * ax.y + v[1] * ax.x;
                out[2] = v[2] * ax.z - v[3] * ax.w; out[3] = v[2] * ax.w + v[3] * ax.z;
            } else if (node < n_nodes && !dry) {
                float *yr = ep.y + (size_t)node * ep.ldy + row0;
                if (y_vec) *reinterpret_cast<float4 *>(yr) = make_float4(v[0], v[1], v[2], v[3]);
                else {
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (k < n_valid) yr[k] = v[k];
                }
            }
            if (mode != EPI_PLAIN && hi_at != nullptr && ok && !dry) {
                T hi[4], lo[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) split_bf16(out[k], hi[k], lo[k]);
                *reinterpret_cast<uint2 *>(hi_at + (size_t)node * out_stride) = pack4_bf16(hi);
                if (lo_at != nullptr) *reinterpret_cast<uint2 *>(lo_at + (size_t)node * out_stride) = pack4_bf16(lo);
            }
        }
    }
}

}  // namespace

#define LLMCAD_TRACE(slot) do { if (p.trace && blockIdx.x < 256) p.trace[(size_t)blockIdx.x * 16 + (slot)] = global_timer_ns(); } while (0)

template <int PK>
__global__ void __launch_bounds__(kThreads, 1)
gemm_stream_kernel(const __grid_constant__ GemmMaps maps, const __grid_constant__ GemmParams p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ SharedCtl ctl;
    const GemmDesc &d = p.g;

    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp: known to be uniform
    const uint32_t nb = (uint32_t)p.n_pad * (p.comp ? 2u : 1u);   // activation rows per k-block = the MMA N: nodes (hi | lo)
    const uint32_t b_tile_bytes = nb * kBlockK * 2;
    // stage: [weights k-block 0 | weights k-block 1 | activations k-block 0 | activations k-block 1]
    const uint32_t stage_bytes = PK * (kATileBytes + b_tile_bytes);
    const uint32_t b_off = PK * kATileBytes;
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t acc_cols = nb;                         // TMEM columns of one of the two accumulator buffers
    const uint64_t wait_limit = p.wait_limit_ns;          // every wait below gives up after this many ns
    const DepWait dep{p.dep_ctr, p.dep_target, wait_limit};

    if (threadIdx.x == 0) LLMCAD_TRACE(0);

    // State of the weight producer (thread 0). It lives across the start-up barrier: the first
    // ring-full of copies goes out right after the barriers are initialised, before TMEM allocation
    // and before the other warps are even needed. Until pdl_wait() this kernel only prefetches
    // weights, which no kernel writes.
    Cursor<PK> pc;
    int ps = 0;
    uint32_t ppar = 1, pissued = 0;    // a fresh barrier passes a wait on parity 1: no special first lap
    uint64_t pol_stream = 0;
    auto issue_item = [&]() {          // the next item of the stream into ring stage ps (which must be free)
        const int nk = pc.nk();
        const uint32_t full = smem_u32(&ctl.full[ps]);
        const uint32_t dst = smem_base + ps * stage_bytes;
        mbar_expect_tx(full, (uint32_t)nk * (kATileBytes + b_tile_bytes));
        if (d.w_tiled != nullptr) {
            // consecutive k-blocks of a tile are contiguous in the tiled layout: one copy
            const size_t t = (size_t)packed_tile(d, pc.tile) * d.kb_per_tile + pc.kb0();
            bulk_load_1d(dst, d.w_tiled + t * kATileBytes, (uint32_t)nk * kATileBytes, full, pol_stream);
        } else {
            for (int k = 0; k < nk; ++k)
                tma_load_2d(dst + k * kATileBytes, &maps.w, (pc.kb0() + k) * kBlockK,
                            pc.tile * kTileM, full, pol_stream);
        }
        __threadfence_block();
        if (pissued == 0) LLMCAD_TRACE(2);
        ctl.a_issued = ++pissued;      // the activation loader may now add its bytes to this stage
        pc.advance();
        if (++ps == p.stages) { ps = 0; ppar ^= 1u; }
    };
    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(smem_u32(&ctl.full[s]), 1);
            mbar_init(smem_u32(&ctl.empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&ctl.tmem_full[b]), 1);
            mbar_init(smem_u32(&ctl.tmem_empty[b]), 4);
        }
        ctl.abort_flag = 0;
        ctl.a_issued = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol_stream));
        pc.init(d);
        while (!pc.done() && pissued < (uint32_t)p.stages) issue_item();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl.tmem_base)),
                     "r"((uint32_t)p.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl.tmem_base;
    volatile int *abort_flag = &ctl.abort_flag;
    bool timed_out = false;
    if (threadIdx.x == 0) LLMCAD_TRACE(1);

    if (warp == 0) {
        // ================================================= weight producer
        // Streams this CTA's weight tiles, in order, as fast as ring slots free up.
        if (lane == 0) {
            // (Asking L2 for weights ahead of the ring while it is blocked, or for the first items of the next GEMM
            // once this CTA's are all requested, or from the finishing kernel while HBM idles, was measured on B200
            // and costs more than it brings in every combination: 3.12 ms per pass of the 7B shape without against
            // 3.14-3.34 ms with 2-8 items ahead and 3-24 items of the next GEMM. The stream runs from HBM straight
            // into the ring.)
            uint64_t t_idle = 0;
            while (!pc.done()) {
                if (mbar_try(smem_u32(&ctl.empty[ps]), ppar)) {
                    issue_item();
                    t_idle = 0;
                    continue;
                }
                // (no sleep between the tries, here and in the activation loader: with 32 ns of it decode passes of the 7B
                // shape took 2823 instead of 2814 us, 20 layers of the 13B shape with 64 nodes 3437 instead of 3410)
                if (t_idle == 0) t_idle = global_timer_ns();
                else if (*abort_flag || global_timer_ns() - t_idle > wait_limit) { timed_out = true; break; }
            }
            LLMCAD_TRACE(6);
        }
    } else if (warp == 6) {
        // ================================================= activation loader
        // Follows the weight producer item by item and adds the (small, L2-resident) activation
        // tiles of each item, once the grid dependency says that the GEMM's input is final.
        if (lane == 0) {
            uint64_t pol_keep;
            asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol_keep));
            Cursor<PK> c;
            c.init(d);
            int s = 0;
            uint32_t i = 0;
            if (!dep_wait_thread(dep)) timed_out = true;
            fence_proxy_async();          // the activations were written by ordinary stores; the copies below read them
            pdl_launch_dependents();
            while (!c.done() && !timed_out && !p.withhold_act) {
                uint64_t t0 = 0;
                // the stage is ours: the producer has passed its "empty" wait and armed the barrier
                for (uint32_t spin = 0; (int32_t)(ctl.a_issued - (i + 1)) < 0; ++spin) {
                    if ((spin & 255u) == 255u) {
                        if (t0 == 0) t0 = global_timer_ns();
                        if (*abort_flag || global_timer_ns() - t0 > wait_limit) { timed_out = true; break; }
                    }
                }
                if (timed_out) break;
                const uint32_t full = smem_u32(&ctl.full[s]);
                const uint32_t dst = smem_base + s * stage_bytes + b_off;
                const int nk = c.nk();
                for (int k = 0; k < nk; ++k)
                    tma_load_3d(dst + k * b_tile_bytes, &maps.x, (c.kb0() + k) * kBlockK, full, pol_keep);
                c.advance();
                ++i;
                if (++s == p.stages) s = 0;
            }
        }
    } else if (warp == 1) {
        // ================================================= MMA issuer
        const uint32_t idesc = make_idesc(kTileM, (int)nb);
        const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_base, 0);
        const bool leader = elect_one();
        const Range r = cta_range<PK>(d, (int)blockIdx.x);
        const int ppt = pairs_per_tile_c<PK>(d), kbpt = d.kb_per_tile;
        uint32_t seg = 0, ph = 0;       // ph: parity to wait for on the stage's "full" barrier
        int s = 0;
        bool ready = false;             // the next item's barrier has been seen complete
        for (int i = r.begin; i < r.end && !timed_out; ++seg) {
            // one segment: the items of one tile that belong to this CTA
            const int tile = i / ppt, seg_end = min(r.end, (tile + 1) * ppt);
            int kb = (i - tile * ppt) * PK;
            const int buf = seg & 1;
            // (seg >> 1: how often this buffer has been used before)
            if (!mbar_wait_all(smem_u32(&ctl.tmem_empty[buf]), ((seg >> 1) & 1u) ^ 1u, abort_flag, wait_limit)) { timed_out = true; break; }
            const uint32_t d0 = tmem + buf * acc_cols;
            uint32_t acc = 0;
            for (; i < seg_end; ++i, kb += PK) {
                if (!ready && !mbar_wait_all(smem_u32(&ctl.full[s]), ph, abort_flag, wait_limit)) { timed_out = true; break; }
                tc_fence_after();
                const uint32_t a_addr = smem_base + s * stage_bytes, b_addr = a_addr + b_off, empty = smem_u32(&ctl.empty[s]);
                const int nk = min(PK, kbpt - kb);
                const uint64_t a_desc = make_smem_desc(a_addr), b_desc = make_smem_desc(b_addr);
                if (leader) {
#pragma unroll
                    for (int k = 0; k < PK; ++k) {
                        if (k >= nk) break;
#pragma unroll
                        for (int k4 = 0; k4 < kBlockK / 16; ++k4)
                            // advancing 16 bf16 = 32 bytes inside the swizzle row: +2 in the >>4 address field
                            tc_mma_bf16(d0, a_desc + k * (kATileBytes >> 4) + 2 * k4, b_desc + k * (b_tile_bytes >> 4) + 2 * k4, idesc,
                                        k > 0 || k4 > 0 ? 1u : acc);
                    }
                    tc_commit(empty);                        // frees the stage when these MMAs have read it
                    if (i + 1 == seg_end) tc_commit(smem_u32(&ctl.tmem_full[buf]));
                }
                acc = 1;
                if (++s == p.stages) { s = 0; ph ^= 1u; }
                ready = i + 1 < r.end && mbar_test_all(smem_u32(&ctl.full[s]), ph);    // while the tensor pipe works on this item
            }
        }
        if (lane == 0) LLMCAD_TRACE(7);
    } else {
        // ================================================= accumulator dump (warps 2..5)
        const int lane_grp = warp & 3;                 // TMEM lanes 32*lane_grp .. +31 belong to this warp
        // the workspace may still be read by the finishing kernel of the previous GEMM
        if (!dep_wait_warp(dep, lane)) timed_out = true;
        pdl_launch_dependents();
        if (threadIdx.x == 64) LLMCAD_TRACE(3);
        const Range r = cta_range<PK>(d, (int)blockIdx.x);
        const int ipt = pairs_per_tile_c<PK>(d);
        const size_t slot_stride = slot_floats(p.n_pad);
        uint32_t seg = 0;
        for (int seg_begin = r.begin; seg_begin < r.end && !timed_out; ++seg) {
            const int tile = seg_begin / ipt;
            const int seg_end = min(r.end, (tile + 1) * ipt);
            const int buf = seg & 1;
            const uint32_t use = seg >> 1;
            if (!mbar_wait_warp(smem_u32(&ctl.tmem_full[buf]), use & 1u, abort_flag, lane, wait_limit)) { timed_out = true; break; }
            tc_fence_after();
            if (threadIdx.x == 64 && seg == 0) LLMCAD_TRACE(4);
            // this CTA's segment of the tile goes to slot tile + CTA, lane = row of the 32-row group;
            // with hi + lo activations a node's two accumulator columns are added first
            const uint32_t t_lane = tmem_base + ((uint32_t)(lane_grp * 32) << 16) + buf * acc_cols;
            if (!LLMCAD_CHECK(tile >= 0 && tile < d.n_tiles * d.halves && tile + (int)blockIdx.x < d.n_tiles * d.halves + d.grid, p.status)) { timed_out = true; break; }
            float *dst = p.partials + (size_t)(tile + (int)blockIdx.x) * slot_stride + (size_t)lane_grp * p.n_pad * 32 + 4 * lane;
            int c0 = 0;
            if (p.comp) {
                // 32 nodes at a time, hi and lo columns in one round trip
                for (; c0 + 32 <= p.n_pad; c0 += 32) {
                    float v[32];
                    tc_ld32_sum2(t_lane + c0, t_lane + p.n_pad + c0, v);
#pragma unroll
                    for (int j = 0; j < 32; j += 4) dump4(dst + (size_t)(c0 + j) * 32, v + j);
                }
            }
            for (; c0 < p.n_pad; c0 += 16) {
                float v[16];
                tc_ld16(t_lane + c0, v);
                if (p.comp) {
                    float t[16];
                    tc_ld16(t_lane + p.n_pad + c0, t);
#pragma unroll
                    for (int j = 0; j < 16; ++j) v[j] += t[j];
                }
#pragma unroll
                for (int j = 0; j < 16; j += 4) dump4(dst + (size_t)(c0 + j) * 32, v + j);
            }
            // the accumulator has left TMEM: hand the buffer back to the MMA warp
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl.tmem_empty[buf]));
            seg_begin = seg_end;
        }
        if (threadIdx.x == 64) LLMCAD_TRACE(8);
    }
    __syncwarp();   // lanes that skipped their role's single-thread section rejoin their warp here
    timed_out = __any_sync(0xffffffffu, timed_out);   // keep the warp together on the way out
    // this dump warp's segments are in the workspace (also said after a wait ran out, so that nobody waits for this CTA)
    if (warp >= 2 && warp <= 5 && lane == 0) dep_arrive(p.s_done);

    if (timed_out) {
        *abort_flag = 1;
        atomicCAS(p.status, 0, LLMCAD_ERR_TIMEOUT);
        // give copies that may still be in flight time to land before the shared memory goes away
        const uint64_t t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 2000000ull) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)p.tmem_cols) : "memory");
        if (lane == 0) LLMCAD_TRACE(13);
    }
}

// ------------------------------------------------------------------------------------------------
// The streaming kernel for wide inputs, on CTA pairs (cta_group::2).
//
// With many nodes the bound moves from HBM to what an SM can take in from L2, of which gemm_stream_kernel spends
// n_pad * 256 bytes per 16 KB of weights on activation tiles (128 nodes: two thirds of the traffic), and to power
// (30B shape, 128 nodes: 1000 W, the clock drops to 1.65 GHz). Here the two CTAs of a cluster work on two weight tiles at once: one
// tcgen05.mma of 256 rows reads each CTA's own weight tile and half of the activation rows from each
// CTA's shared memory, so that every activation tile enters an SM pair once: half the traffic, and room for
// more weights in the ring (30B shape, 128 nodes, 12 layers: 4.70 -> 4.45 ms a pass; its stream alone, unthrottled,
// 53 -> 46 us for the QKV GEMM). Each CTA keeps the accumulator of its own tile and dumps it as before.
//
// Roles as in gemm_stream_kernel; the MMA warp of the first CTA of the pair issues for both. Copies of both
// CTAs complete on the first CTA's "full" barrier (its producer announces the bytes of both), the MMAs' commits
// release the stage and announce the accumulator in both CTAs, and the dump warps of both hand an
// accumulator buffer back on the first CTA's barrier. Weights travel as tensor-map boxes of 512-byte rows over
// the packed tiles: a plain bulk copy can only complete on a barrier of its own CTA.
//
// kWide (128 < nodes <= 256, prefill): hi and lo activation planes are multiplied one after the other, each into 256
// columns of its own, which is all of tensor memory: one accumulator buffer, so the next tile's MMAs wait for the dump.
// Both planes in the same columns left room for two buffers (512 tokens at 7B: 15.3 instead of 15.8 ms), but the tensor
// cores cut a sum off to its accumulator's bits at every MMA, always towards zero (5.8e-8 of the sum per k-block), and so
// did it twice as often (2 layers of the 7B shape without attention, logits against 64 bits: 1.01e-5 instead of 7.8e-6).
__device__ __forceinline__ uint32_t map_to_cta0(uint32_t addr)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
    return r;
}
__device__ __forceinline__ void tma_pair_2d(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar0, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%2, %3}], [%4], %5;"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(bar0), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void tma_pair_3d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, uint32_t bar0, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%2, %3, %4}], [%5], %6;"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar0), "l"(policy)
        : "memory");
}
// both CTAs' barriers at this offset
__device__ __forceinline__ void tc_commit_pair(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void tc_mma_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <int PK, bool kWide>
__global__ void __launch_bounds__(kThreads, 1)
gemm_pair_kernel(const __grid_constant__ GemmMaps maps, const __grid_constant__ GemmParams p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ SharedCtl ctl;
    const GemmDesc &d = p.g;

    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp: known to be uniform
    const int rank = (int)blockIdx.x & 1, group = (int)blockIdx.x >> 1;
    const int n_vtiles = d.n_tiles * d.halves;
    const uint32_t nb = (uint32_t)p.n_pad * (p.comp && !kWide ? 2u : 1u);      // MMA N
    const uint32_t b_half = nb / 2 * kBlockK * 2;                              // this CTA's activation rows of a k-block, one pass
    const uint32_t b_tile_bytes = b_half * (kWide ? 2u : 1u);
    const uint32_t stage_bytes = PK * (kATileBytes + b_tile_bytes);
    const uint32_t b_off = PK * kATileBytes;
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint64_t wait_limit = p.wait_limit_ns;
    const DepWait dep{p.dep_ctr, p.dep_target, wait_limit};
    if (threadIdx.x == 0) LLMCAD_TRACE(0);

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(smem_u32(&ctl.full[s]), 1);
            mbar_init(smem_u32(&ctl.empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&ctl.tmem_full[b]), 1);
            mbar_init(smem_u32(&ctl.tmem_empty[b]), 8);
        }
        ctl.abort_flag = 0;
        ctl.a_issued = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    // Allocating and freeing tensor memory for a pair are acts of both CTAs: neither may start before the other CTA
    // is running, nor leave before the other has done its part. (The first barrier also says that the mbarriers of
    // both exist before a copy or a commit signals them.)
    __syncwarp();
    cluster_sync_all();
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl.tmem_base)),
                     "r"((uint32_t)p.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl.tmem_base;
    volatile int *abort_flag = &ctl.abort_flag;
    bool timed_out = false;
    if (threadIdx.x == 0) LLMCAD_TRACE(1);

    // the pair's items: (pair of weight tiles, PK k-blocks), the same list in both CTAs
    const int ppt = pairs_per_tile_c<PK>(d), total = (n_vtiles + 1) / 2 * ppt;
    const int begin = min(total, group * d.items_per_cta), end = min(total, begin + d.items_per_cta);

    if (warp == 0) {
        // ================================================= weight producer
        if (lane == 0) {
            uint64_t pol_stream;
            asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol_stream));
            int s = 0, pt = begin / ppt, kp = begin - pt * ppt;
            uint32_t par = 1;
            uint64_t t_idle = 0;
            for (int i = begin; i < end;) {
                if (!mbar_try(smem_u32(&ctl.empty[s]), par)) {
                    if (t_idle == 0) t_idle = global_timer_ns();
                    else if (*abort_flag || global_timer_ns() - t_idle > wait_limit) { timed_out = true; break; }
                    continue;
                }
                t_idle = 0;
                const uint32_t full = smem_u32(&ctl.full[s]);
                if (rank == 0) mbar_expect_tx(full, 2u * stage_bytes);
                // (an odd last tile is loaded twice; an item past the end of a tile's k-blocks brings bytes nobody multiplies)
                const int v = min(2 * pt + rank, n_vtiles - 1);
                for (int k = 0; k < PK; ++k)
                    tma_pair_2d(smem_base + s * stage_bytes + k * kATileBytes, &maps.w, 0, (packed_tile(d, v) * d.kb_per_tile + kp * PK + k) * 32, map_to_cta0(full), pol_stream);
                __threadfence_block();
                if (i == begin) LLMCAD_TRACE(2);
                ctl.a_issued = (uint32_t)(++i - begin);
                if (++kp == ppt) { kp = 0; ++pt; }
                if (++s == p.stages) { s = 0; par ^= 1u; }
            }
            LLMCAD_TRACE(6);
        }
    } else if (warp == 6) {
        // ================================================= activation loader: this CTA's half of the rows
        if (lane == 0) {
            uint64_t pol_keep;
            asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol_keep));
            int s = 0, kp = begin % ppt;
            if (!dep_wait_thread(dep)) timed_out = true;
            fence_proxy_async();
            pdl_launch_dependents();
            for (int i = begin; i < end && !timed_out; ++i) {
                uint64_t t0 = 0;
                for (uint32_t spin = 0; (int32_t)(ctl.a_issued - (uint32_t)(i + 1 - begin)) < 0; ++spin) {
                    // (no sleep between the looks: 0.5 % of a pass at 30B widths with 128 nodes)
                    if ((spin & 255u) == 255u) {
                        if (t0 == 0) t0 = global_timer_ns();
                        if (*abort_flag || global_timer_ns() - t0 > wait_limit) { timed_out = true; break; }
                    }
                }
                if (timed_out) break;
                const uint32_t full = map_to_cta0(smem_u32(&ctl.full[s]));
                const uint32_t dst = smem_base + s * stage_bytes + b_off;
                // hi | lo planes: the first CTA has the hi rows, the second the lo rows; one plane, or wide: half of the rows each
                const bool by_plane = p.comp && !kWide;
                for (int k = 0; k < PK; ++k)
                    tma_pair_3d(dst + k * b_tile_bytes, &maps.x, (kp * PK + k) * kBlockK, by_plane ? 0 : rank * (int)(nb / 2), by_plane ? rank : 0, full, pol_keep);
                if (++kp == ppt) kp = 0;
                if (++s == p.stages) s = 0;
            }
        }
    } else if (warp == 1) {
        // ================================================= MMA issuer (first CTA of the pair)
        if (rank == 0) {
            const uint32_t idesc = make_idesc(2 * kTileM, (int)nb);
            const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_base, 0);
            const bool leader = elect_one();
            uint32_t seg = 0, ph = 0;
            int s = 0;
            bool ready = false;
            for (int i = begin; i < end && !timed_out; ++seg) {
                const int pt = i / ppt, seg_end = min(end, (pt + 1) * ppt);
                int kb = (i - pt * ppt) * PK;
                const int buf = kWide ? 0 : seg & 1;
                const uint32_t use = kWide ? seg : seg >> 1;
                if (!mbar_wait_all(smem_u32(&ctl.tmem_empty[buf]), (use & 1u) ^ 1u, abort_flag, wait_limit)) { timed_out = true; break; }
                const uint32_t d0 = tmem + buf * nb;
                uint32_t acc = 0;
                for (; i < seg_end; ++i, kb += PK) {
                    if (!ready && !mbar_wait_all(smem_u32(&ctl.full[s]), ph, abort_flag, wait_limit)) { timed_out = true; break; }
                    tc_fence_after();
                    const uint32_t a_addr = smem_base + s * stage_bytes, b_addr = a_addr + b_off, empty = smem_u32(&ctl.empty[s]);
                    const int nk = min(PK, d.kb_per_tile - kb);
                    const uint64_t a_desc = make_smem_desc(a_addr), b_desc = make_smem_desc(b_addr);
                    if (leader) {
#pragma unroll
                        for (int k = 0; k < PK; ++k) {
                            if (k >= nk) break;
#pragma unroll
                            for (int pl = 0; pl < (kWide ? 2 : 1); ++pl)
#pragma unroll
                                for (int k4 = 0; k4 < kBlockK / 16; ++k4)
                                    tc_mma_pair(d0 + pl * nb, a_desc + k * (kATileBytes >> 4) + 2 * k4, b_desc + ((k * b_tile_bytes + pl * b_half) >> 4) + 2 * k4, idesc,
                                                k > 0 || k4 > 0 ? 1u : acc);
                        }
                        tc_commit_pair(empty);
                        if (i + 1 == seg_end) tc_commit_pair(smem_u32(&ctl.tmem_full[buf]));
                    }
                    acc = 1;
                    if (++s == p.stages) { s = 0; ph ^= 1u; }
                    ready = i + 1 < end && mbar_test_all(smem_u32(&ctl.full[s]), ph);
                }
            }
            if (lane == 0) LLMCAD_TRACE(7);
        }
    } else {
        // ================================================= accumulator dump (warps 2..5): this CTA's weight tile
        const int lane_grp = warp & 3;
        if (!dep_wait_warp(dep, lane)) timed_out = true;
        pdl_launch_dependents();
        if (threadIdx.x == 64) LLMCAD_TRACE(3);
        const size_t slot_stride = slot_floats(p.n_pad);
        uint32_t seg = 0;
        for (int i = begin; i < end && !timed_out; ++seg) {
            const int pt = i / ppt, v = 2 * pt + rank, buf = kWide ? 0 : seg & 1;
            i = min(end, (pt + 1) * ppt);
            if (!mbar_wait_warp(smem_u32(&ctl.tmem_full[buf]), (kWide ? seg : seg >> 1) & 1u, abort_flag, lane, wait_limit)) { timed_out = true; break; }
            tc_fence_after();
            if (threadIdx.x == 64 && seg == 0) LLMCAD_TRACE(4);
            const uint32_t t_lane = tmem_base + ((uint32_t)(lane_grp * 32) << 16) + buf * nb;
            if (v < n_vtiles) {
                if (!LLMCAD_CHECK(v >= 0 && v + 2 * group < n_vtiles + d.grid, p.status)) { timed_out = true; break; }
                float *dst = p.partials + (size_t)(v + 2 * group) * slot_stride + (size_t)lane_grp * p.n_pad * 32 + 4 * lane;
                int c0 = 0;
                for (; c0 + 32 <= p.n_pad; c0 += 32) {
                    float t[32];
                    if (p.comp) tc_ld32_sum2(t_lane + c0, t_lane + p.n_pad + c0, t);
                    else tc_ld32(t_lane + c0, t);
#pragma unroll
                    for (int j = 0; j < 32; j += 4) dump4(dst + (size_t)(c0 + j) * 32, t + j);
                }
                for (; c0 < p.n_pad; c0 += 16) {
                    float t[16];
                    tc_ld16(t_lane + c0, t);
                    if (p.comp && !kWide) {
                        float u[16];
                        tc_ld16(t_lane + p.n_pad + c0, u);
#pragma unroll
                        for (int j = 0; j < 16; ++j) t[j] += u[j];
                    }
#pragma unroll
                    for (int j = 0; j < 16; j += 4) dump4(dst + (size_t)(c0 + j) * 32, t + j);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(map_to_cta0(smem_u32(&ctl.tmem_empty[buf])));
        }
        if (threadIdx.x == 64) LLMCAD_TRACE(8);
    }
    __syncwarp();
    timed_out = __any_sync(0xffffffffu, timed_out);
    if (warp >= 2 && warp <= 5 && lane == 0) dep_arrive(p.s_done);
    if (timed_out) {
        *abort_flag = 1;
        atomicCAS(p.status, 0, LLMCAD_ERR_TIMEOUT);
        const uint64_t t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 2000000ull) __nanosleep(1000);
    }
    tc_fence_before();
    __syncwarp();
    cluster_sync_all();            // the other CTA has stopped signalling this one's barriers and using its shared memory
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)p.tmem_cols) : "memory");
    __syncwarp();
    cluster_sync_all();            // and both have given their tensor memory back
    if (threadIdx.x == 32) LLMCAD_TRACE(13);
}

// ------------------------------------------------------------------------------------------------
// The streaming kernel for INT4 weights.
//
// A quarter of the bytes, so HBM no longer sets the pace: expanding the weights does (~1100 cycles per item of four
// k-blocks, against ~770 for its MMAs at 64 columns, ~48 cycles each for K = 16, and ~650 for its bytes). The weights
// are expanded straight into tensor memory and multiplied from there: thread = weight row = TMEM lane, eight codes of a
// word become four packed bf16 pairs, 32 of which are the row's share of a k-block. (Expanded into shared memory, by
// the warps that also dumped the accumulators, a pass of the 7B shape with 32 nodes took 3.53 ms; now 2.33 ms.)
//
// What an item costs beside its arithmetic, its barriers, fences and addresses, is worth as much attention: ~520
// cycles in the MMA warp, ~290 in each expanding warp. An item here is therefore two of the items that the kernels for
// bf16 weights move, 2 PK k-blocks, as far as the segment reaches.
//
// Warps: 0 producer of packed items (bulk copies), 1 TMEM allocator and MMA issuer, 2 activation loader (TMA),
// 4..11 expansion and dump: warp w works on rows 32 * (w % 4) .., the two sets of four take alternate k-blocks of an
// item and alternate 16-node chunks of a dump. More sets do not help (three: 2.58 against 2.48 ms a pass; four, with 40
// registers a thread: a third slower): the ALU and FMA pipes of the four schedulers are the bound, not latency. Three
// rings of items: packed (shared memory), expanded (tensor memory, what the accumulators leave of the 512 columns),
// activations (shared memory). Until the grid dependency the packed ring fills and the expanded ring as far as it
// reaches. At most 72 registers a thread: three warps per scheduler beside the finishing CTA's three of 96.
//
// Work is cut and ordered exactly as the kernels for bf16 weights cut theirs on the same number of nodes (CTA pairs
// included, which here only means how tiles and ranges are dealt out), so that the sums are the same to the bit.
constexpr int kW4Sets = 2, kW4Threads = 128 + 128 * kW4Sets;
constexpr int kMaxPStages = 16, kMaxXStages = 12, kMaxAStages = 12;

struct W4Ctl {
    uint64_t pfull[kMaxPStages], pempty[kMaxPStages];     // packed items
    uint64_t xfull[kMaxXStages], xempty[kMaxXStages];     // expanded items
    uint64_t afull[kMaxAStages];                          // activation items
    uint64_t tmem_full[2], tmem_empty[2];
    uint32_t tmem_base;
    volatile int abort_flag;
};

// D[tmem] (+)= A[tmem] * B[smem]^T; A: lanes = rows, one 32-bit column = two bf16 along K
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// 16 consecutive 32-bit columns of this thread's TMEM lane
__device__ __forceinline__ void tc_st16(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
          "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
// 32 codes of a row, two to a bf16 pair, into 16 columns of this thread's TMEM lane: nibble j of each half of a word by a
// shift, one (a & b) | c and one fused multiply-add. Shifts and logic run at half the issue rate and pace the kernel, so
// there must be no more of them: from the plain expression the compiler made an AND and an OR, and with `nibbles` and
// `magic` as constants it knows it is slower than with values in registers (cycles for two k-blocks: 1028 plain, 885, 839).
__device__ __forceinline__ void expand_store(const uint4 &c, uint32_t nibbles, uint32_t magic, uint32_t s2, uint32_t b2, uint32_t taddr)
{
    const uint32_t ww[4] = {c.x, c.y, c.z, c.w};
    uint32_t o[16];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t t2;
            asm("lop3.b32 %0, %1, %2, %3, 0xea;" : "=r"(t2) : "r"(ww[q] >> (4 * j)), "r"(nibbles), "r"(magic));
            asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(o[q * 4 + j]) : "r"(t2), "r"(s2), "r"(b2));
        }
    tc_st16(taddr, o);
}
__device__ __forceinline__ uint4 lds128(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ int lds_s8(uint32_t addr)
{
    int v;
    asm volatile("ld.shared.s8 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
// 16 columns at each of two addresses, summed (one wait for both loads)
__device__ __forceinline__ void tc_ld16_sum2(uint32_t taddr_a, uint32_t taddr_b, float *v)
{
    uint32_t a[16], b[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%33];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]), "=r"(a[15]),
          "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7]), "=r"(b[8]), "=r"(b[9]), "=r"(b[10]), "=r"(b[11]), "=r"(b[12]), "=r"(b[13]), "=r"(b[14]), "=r"(b[15])
        : "r"(taddr_a), "r"(taddr_b)
        : "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(a[j]) + __uint_as_float(b[j]);
}

// slot and parity of a ring of n slots
struct RingPos {
    int slot;
    uint32_t par;
    __device__ void step(int n)
    {
        if (++slot == n) { slot = 0; par ^= 1u; }
    }
};

// Walks a CTA's share [i, end) of the (tile, PK k-blocks) list in steps of up to two entries of one tile.
template <int PK>
struct W4Walk {
    int i, end, ppt, kbpt;
    int unit, kb, nk;       // tile (or pair of tiles), first k-block and number of k-blocks of the current step
    bool last;              // it ends a segment: the entries of one tile that belong to this CTA
    int n_items;
    __device__ void init(int begin, int e, int p, int k)
    {
        i = begin; end = e; ppt = p; kbpt = k;
        unit = begin / p;
        load();
    }
    __device__ void load()
    {
        const int at = i - unit * ppt, left = min(end - i, ppt - at);
        n_items = min(2, left);
        last = n_items == left;
        kb = at * PK;
        nk = min(n_items * PK, kbpt - kb);
    }
    __device__ bool done() const { return i >= end; }
    __device__ void next()
    {
        i += n_items;
        if (i == (unit + 1) * ppt) ++unit;
        load();
    }
};

// The same steps for the warps that only need to know how many k-blocks a step has: one subtraction per step.
template <int PK>
struct W4Count {
    int i, end, ppt, kbpt, unit;
    int left;               // k-blocks from the current step to the end of its segment; 0: no step left
    __device__ void init(int begin, int e, int p, int k)
    {
        i = begin; end = e; ppt = p; kbpt = k;
        unit = begin / p;
        left = 0;
        segment();
    }
    __device__ void segment()
    {
        if (i >= end) return;
        const int at = i - unit * ppt, n = min(end - i, ppt - at);
        left = min(n * PK, kbpt - at * PK);
        i += n;
        ++unit;
    }
    __device__ bool done() const { return left == 0; }
    __device__ int nk() const { return min(2 * PK, left); }
    __device__ void next(int nk)
    {
        left -= nk;
        if (left == 0) segment();
    }
};

template <int PK>
__global__ void __maxnreg__(72)
gemm_w4_kernel(const __grid_constant__ GemmMaps maps, const __grid_constant__ GemmParams p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ W4Ctl ctl;
    const GemmDesc &d = p.g;

    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp: known to be uniform
    const uint32_t nb = (uint32_t)p.n_pad * (p.comp ? 2u : 1u);
    constexpr int SK = 2 * PK;                     // k-blocks per item
    const uint32_t b_tile_bytes = nb * kBlockK * 2, astage_bytes = SK * b_tile_bytes;
    constexpr uint32_t pstage_bytes = SK * kW4TileBytes;
    const uint32_t act_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t packed_base = act_base + (uint32_t)p.astages * astage_bytes;
    const int acc_bufs = p.acc_bufs;
    const uint64_t wait_limit = p.wait_limit_ns;
    const DepWait dep{p.dep_ctr, p.dep_target, wait_limit};
    if (threadIdx.x == 0) LLMCAD_TRACE(0);

    // this CTA's items: with group == 2 two CTAs walk the same list of (pair of tiles, k-blocks), each for its tile
    const int rank = d.group == 2 ? (int)blockIdx.x & 1 : 0, group = (int)blockIdx.x / d.group;
    const int n_vtiles = d.n_tiles * d.halves, ppt = pairs_per_tile_c<PK>(d);
    const int total = (n_vtiles + d.group - 1) / d.group * ppt;
    const int begin = min(total, group * d.items_per_cta), end = min(total, begin + d.items_per_cta);
    auto tile_of = [&](int unit) { return d.group == 2 ? 2 * unit + rank : unit; };

    // ---- weight producer, across the start-up barrier: the first ring-full goes out at once
    W4Walk<PK> pw{};
    RingPos pp{0, 1};                              // a fresh barrier passes a wait on parity 1
    uint64_t pol_stream = 0;
    auto issue_item = [&]() {
        const int v = min(tile_of(pw.unit), n_vtiles - 1);
        const uint32_t full = smem_u32(&ctl.pfull[pp.slot]), bytes = (uint32_t)pw.nk * kW4TileBytes;
        mbar_expect_tx(full, bytes);
        bulk_load_1d(packed_base + pp.slot * pstage_bytes, d.w_tiled + ((size_t)packed_tile(d, v) * d.kb_per_tile + pw.kb) * kW4TileBytes,
                     bytes, full, pol_stream);
        pw.next();
        pp.step(p.pstages);
    };
    if (threadIdx.x == 0) {
        for (int s = 0; s < p.pstages; ++s) { mbar_init(smem_u32(&ctl.pfull[s]), 1); mbar_init(smem_u32(&ctl.pempty[s]), 4 * kW4Sets); }
        for (int s = 0; s < p.stages; ++s) { mbar_init(smem_u32(&ctl.xfull[s]), 4 * kW4Sets); mbar_init(smem_u32(&ctl.xempty[s]), 1); }
        for (int s = 0; s < p.astages; ++s) mbar_init(smem_u32(&ctl.afull[s]), 1);
        for (int b = 0; b < 2; ++b) { mbar_init(smem_u32(&ctl.tmem_full[b]), 1); mbar_init(smem_u32(&ctl.tmem_empty[b]), 4 * kW4Sets); }
        ctl.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol_stream));
        pw.init(begin, end, ppt, d.kb_per_tile);
        for (int q = 0; q < p.pstages && !pw.done(); ++q) issue_item();
        LLMCAD_TRACE(2);
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl.tmem_base)),
                     "r"((uint32_t)p.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl.tmem_base, x_base = tmem_base + (uint32_t)acc_bufs * nb;
    volatile int *abort_flag = &ctl.abort_flag;
    bool timed_out = false;
    if (threadIdx.x == 0) LLMCAD_TRACE(1);

    if (warp == 0) {
        if (lane == 0) {
            uint64_t t_idle = 0;
            while (!pw.done()) {
                if (mbar_try(smem_u32(&ctl.pempty[pp.slot]), pp.par)) {
                    issue_item();
                    t_idle = 0;
                    continue;
                }
                __nanosleep(32);      // (a pass of the 7B shape takes 2319 us with and 2318 without it: the expansion paces it, not this thread)
                if (t_idle == 0) t_idle = global_timer_ns();
                else if (*abort_flag || global_timer_ns() - t_idle > wait_limit) { timed_out = true; break; }
            }
            LLMCAD_TRACE(6);
        }
    } else if (warp == 2) {
        // ================================================= activation loader
        if (lane == 0) {
            uint64_t pol_keep;
            asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol_keep));
            // Item i goes where item i - astages was, once the MMAs have read that: the barrier of its expanded slot says
            // so. (There are at least as many expanded slots as activation slots: the barrier cannot be a lap further,
            // because the item that would take it there has no activations yet.)
            RingPos a{0, 0}, x{0, 0};
            W4Walk<PK> w;
            w.init(begin, end, ppt, d.kb_per_tile);
            if (!dep_wait_thread(dep)) timed_out = true;
            fence_proxy_async();          // the activations were written by ordinary stores; the copies below read them
            pdl_launch_dependents();
            for (int q = 0; !w.done() && !timed_out; ++q) {
                if (q >= p.astages) {
                    if (!mbar_wait(smem_u32(&ctl.xempty[x.slot]), x.par, abort_flag, wait_limit)) { timed_out = true; break; }
                    x.step(p.stages);
                }
                const uint32_t full = smem_u32(&ctl.afull[a.slot]), dst = act_base + a.slot * astage_bytes;
                mbar_expect_tx(full, (uint32_t)w.nk * b_tile_bytes);
                for (int k = 0; k < w.nk; ++k) tma_load_3d(dst + k * b_tile_bytes, &maps.x, (w.kb + k) * kBlockK, full, pol_keep);
                w.next();
                a.step(p.astages);
            }
        }
    } else if (warp == 1) {
        // ================================================= MMA issuer
        const uint32_t idesc = make_idesc(kTileM, (int)nb);
        const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_base, 0), xb = tmem + (uint32_t)acc_bufs * nb;
        const bool leader = elect_one();
        RingPos x{0, 0}, a{0, 0};
        W4Count<PK> w;
        w.init(begin, end, ppt, d.kb_per_tile);
        uint32_t seg = 0, acc = 0;
        int buf = 0;
        bool ready = false;
        while (!w.done()) {
            if (acc == 0) {                                  // a segment begins
                buf = acc_bufs == 2 ? (int)(seg & 1) : 0;
                const uint32_t use = acc_bufs == 2 ? seg >> 1 : seg;
                if (!mbar_wait_all(smem_u32(&ctl.tmem_empty[buf]), (use & 1u) ^ 1u, abort_flag, wait_limit)) { timed_out = true; break; }
                ++seg;
            }
            if (!ready && !(mbar_wait_all(smem_u32(&ctl.xfull[x.slot]), x.par, abort_flag, wait_limit) &&
                            mbar_wait_all(smem_u32(&ctl.afull[a.slot]), a.par, abort_flag, wait_limit))) { timed_out = true; break; }
            tc_fence_after();
            const uint32_t d0 = tmem + buf * nb, at = xb + x.slot * (SK * 32), empty = smem_u32(&ctl.xempty[x.slot]);
            const uint64_t b_desc = make_smem_desc(act_base + a.slot * astage_bytes);
            const int nk = w.nk();
            const bool last = nk == w.left;                  // the item ends its segment
            if (leader) {
#pragma unroll
                for (int k = 0; k < SK; ++k) {
                    if (k >= nk) break;
#pragma unroll
                    for (int k4 = 0; k4 < kBlockK / 16; ++k4)
                        tc_mma_ts(d0, at + k * 32 + k4 * 8, b_desc + k * (b_tile_bytes >> 4) + 2 * k4, idesc, k > 0 || k4 > 0 ? 1u : acc);
                }
                tc_commit(empty);                            // the expanded item's slot, and with it the activation item's (see the loader)
                if (last) tc_commit(smem_u32(&ctl.tmem_full[buf]));
            }
            acc = last ? 0 : 1;
            w.next(nk);
            x.step(p.stages);
            a.step(p.astages);
            ready = !w.done() && mbar_test2_all(smem_u32(&ctl.xfull[x.slot]), x.par, smem_u32(&ctl.afull[a.slot]), a.par);
        }
        if (lane == 0) LLMCAD_TRACE(7);
    } else if (warp >= 4) {
        // ================================================= expansion and dump
        const int quad = warp & 3, set = (warp - 4) >> 2, row = quad * 32 + lane;
        const uint32_t zero = (uint32_t)p.n_pad >> 24;        // (as the compiler cannot know)
        const uint32_t nibbles = 0x000f000fu | zero, magic = 0x43004300u | zero;
        const uint32_t t_quad = (uint32_t)(quad * 32) << 16;
        RingPos pk{0, 0}, x{0, 1};
        W4Count<PK> w;                             // the items to expand
        w.init(begin, end, ppt, d.kb_per_tile);
        int expanded = 0, dumpable = 0;            // items expanded; items up to and including the ones of the segment to be dumped next
        // this thread's codes and exponents in packed slot 0, and its set's columns in expanded slot 0
        const uint32_t row_codes = packed_base + set * kW4TileBytes + row * 16, row_exp = packed_base + set * kW4TileBytes + 4096 + row;
        const uint32_t x_set = x_base + t_quad + set * 32;
        bool dep_ok = false, ready = false;
        uint32_t seg = 0;
        for (int i = begin; i < end && !timed_out; ++seg) {
            const int unit = i / ppt, seg_end = min(end, (unit + 1) * ppt);
            // Items of the next segments are expanded ahead of this one's dump, as far as their slots are freed by MMAs
            // that do not wait for it: the tensor cores have work while the accumulators leave.
            dumpable += (seg_end - i + 1) / 2;
            while (!w.done() && expanded < dumpable + p.stages && !timed_out) {
                if (!ready && !(mbar_wait_all(smem_u32(&ctl.pfull[pk.slot]), pk.par, abort_flag, wait_limit) &&
                                mbar_wait_all(smem_u32(&ctl.xempty[x.slot]), x.par, abort_flag, wait_limit))) { timed_out = true; break; }
                tc_fence_after();
                // A row's 64 codes of a k-block are two 16-byte words, [half][row], its exponent follows them. A set takes every
                // other k-block; the words of its next one are loaded while it works on this one. The loop is not unrolled:
                // the expanding warps share their scheduler's instruction cache with the MMA warp, and with 400 instructions
                // here that warp's 60 were fetched anew for every item.
                uint32_t src = row_codes + pk.slot * pstage_bytes, src_e = row_exp + pk.slot * pstage_bytes, dst = x_set + x.slot * (SK * 32);
                const int nk = w.nk();
                uint4 c0 = lds128(src), c1 = lds128(src + 2048);
                int e = lds_s8(src_e);
#pragma unroll 1
                for (int k = set; k < nk; k += kW4Sets) {
                    // OR 0x4300 into each half: 128 + u (u = q + 8); (128 + u) * 2^e - 136 * 2^e = q * 2^e, exact. The bf16 bits
                    // of 2^e are (e + 127) << 7, those of -136 * 2^e are that + 0x8388.
                    const uint32_t s2 = (uint32_t)(e + 127) * 0x00800080u, b2 = s2 + 0x83888388u;
                    const uint4 h0 = c0, h1 = c1;
                    if (k + kW4Sets < nk) { src += kW4Sets * kW4TileBytes; src_e += kW4Sets * kW4TileBytes; }
                    c0 = lds128(src);
                    c1 = lds128(src + 2048);
                    e = lds_s8(src_e);
                    expand_store(h0, nibbles, magic, s2, b2, dst);
                    expand_store(h1, nibbles, magic, s2, b2, dst + 16);
                    dst += kW4Sets * 32;
                }
                const uint32_t xfull = smem_u32(&ctl.xfull[x.slot]), pempty = smem_u32(&ctl.pempty[pk.slot]);
                ++expanded;
                w.next(nk);
                pk.step(p.pstages);
                x.step(p.stages);
                ready = !w.done() && mbar_test2_all(smem_u32(&ctl.pfull[pk.slot]), pk.par, smem_u32(&ctl.xempty[x.slot]), x.par);
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
                __syncwarp();
                // The packed slot, too, is given back only here, where every word has gone through the arithmetic above: given
                // back right after the loads it was refilled before cold code (an instruction fetch of half a microsecond at
                // the start of the kernel) had got to them.
                if (lane == 0) { mbar_arrive(xfull); mbar_arrive(pempty); }
            }
            if (timed_out) break;
            // ---- dump
            if (!dep_ok) {                          // the workspace may still be read by the previous GEMM's finishing kernel
                if (!dep_wait_warp(dep, lane)) { timed_out = true; break; }
                pdl_launch_dependents();
                dep_ok = true;
                if (threadIdx.x == 128) LLMCAD_TRACE(3);
            }
            const int v = tile_of(unit), buf = acc_bufs == 2 ? (int)(seg & 1) : 0;
            const uint32_t use = acc_bufs == 2 ? seg >> 1 : seg;
            if (!mbar_wait_warp(smem_u32(&ctl.tmem_full[buf]), use & 1u, abort_flag, lane, wait_limit)) { timed_out = true; break; }
            tc_fence_after();
            if (v < n_vtiles) {
                if (!LLMCAD_CHECK(v >= 0 && v + d.group * group < n_vtiles + d.grid, p.status)) { timed_out = true; break; }
                float *dst = p.partials + (size_t)(v + d.group * group) * slot_floats(p.n_pad) + (size_t)quad * p.n_pad * 32 + 4 * lane;
                const uint32_t t_lane = tmem_base + t_quad + buf * nb;
                for (int c0 = 16 * set; c0 < p.n_pad; c0 += 16 * kW4Sets) {
                    float t[16];
                    if (p.comp) tc_ld16_sum2(t_lane + c0, t_lane + p.n_pad + c0, t);
                    else tc_ld16(t_lane + c0, t);
#pragma unroll
                    for (int j = 0; j < 16; j += 4) dump4(dst + (size_t)(c0 + j) * 32, t + j);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl.tmem_empty[buf]));
            i = seg_end;
        }
        if (threadIdx.x == 128) LLMCAD_TRACE(8);
    }
    __syncwarp();
    timed_out = __any_sync(0xffffffffu, timed_out);
    if (timed_out) {
        *abort_flag = 1;
        atomicCAS(p.status, 0, LLMCAD_ERR_TIMEOUT);
        const uint64_t t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 2000000ull) __nanosleep(1000);
    }
    tc_fence_before();
    __syncthreads();
    if (warp >= 4 && warp <= 7 && lane == 0) dep_arrive(p.s_done);      // four arrivals per CTA, behind the barrier: all sets have dumped
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)p.tmem_cols) : "memory");
        if (lane == 0) LLMCAD_TRACE(13);
    }
}

// Adds the segments of every tile and applies the fused epilogue; see the head of the file. The
// work is cut into (tile, 32-row group) pairs; k warps share a pair's node groups, k chosen so that
// all warps of the grid have work. G node groups and KB segments of each are loaded in one go
// (the launcher picks them so that a warp normally needs a single round trip to L2).
//
// Until the grid dependency (the streaming kernel) resolves, the CTA has nothing to do but sits on
// its SM already. It uses the time (a) to read what earlier GEMMs left: the description, the norm
// sums, the gains; (b) for a dry run of its own work with the stores switched off, on whatever the
// workspace holds: the code of this kernel runs once per launch and would be fetched from L2 line
// by line otherwise, which costs more than the work itself.
template <int MODE, int G, int KB>
__global__ void __maxnreg__(kFinMaxRegs)
gemm_finish_kernel(const __grid_constant__ GemmParams p)
{
    // The finishing code reads the GEMM's description (pointers, sizes, mode) all over. From the kernel
    // parameters every first touch of a constant-cache line is a miss; a copy in shared memory costs
    // nothing to read.
    __shared__ __align__(16) GemmDesc s_desc;
    __shared__ float s_part[kFinThreads / LLMCAD_MAX_TREE][LLMCAD_MAX_TREE];
    __shared__ float s_rs[kLoRows];
    {
        static_assert(sizeof(GemmDesc) % 4 == 0, "GemmDesc is copied word by word");
        const uint32_t *src = reinterpret_cast<const uint32_t *>(&p.g);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&s_desc);
        for (int i = threadIdx.x; i < (int)(sizeof(GemmDesc) / 4); i += kFinThreads) dst[i] = src[i];
    }
    pdl_launch_dependents();     // the next GEMM's streaming kernel may take the SMs as they free up
    if (threadIdx.x == 0) LLMCAD_TRACE(9);
    // what earlier GEMMs left (norm sums, residual, gains) is final: the streaming kernel of this GEMM
    // waited for the same counter before it let this kernel launch, so this returns at once
    bool late = false;
    if (threadIdx.x == 0 && p.dep_ctr != nullptr) late = !dep_wait_thread(DepWait{p.dep_ctr, p.dep_target, p.wait_limit_ns});
    __syncthreads();
    const GemmDesc &d = s_desc;
    const EpiParams &ep = d.ep;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // ---- RMSNorm of the GEMM input folded into the epilogue: the producer of the residual stream
    // left partial sums of squares per node ([parts][kLoRows]); the accumulators of node i are multiplied
    // by rsqrt(mean(x^2) + eps). Three threads per node add every third partial row, in a fixed order.
    if (ep.ssq_in != nullptr) {
        constexpr int kSlices = kFinThreads / LLMCAD_MAX_TREE;
        const int col128 = threadIdx.x & (LLMCAD_MAX_TREE - 1), slice = threadIdx.x / LLMCAD_MAX_TREE;
        for (int n0 = 0; n0 < p.n_pad; n0 += LLMCAD_MAX_TREE) {
            const int node = n0 + col128;
            float acc = 0.f;
            if (node < ep.n) {             // (the sums of a call on the last row alone start there: none lie behind them)
                const float *col = ep.ssq_in + node;
                int t = slice;
                for (; t + 7 * kSlices < ep.ssq_in_parts; t += 8 * kSlices) {
                    float v[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) v[u] = __ldcg(col + (size_t)(t + kSlices * u) * kLoRows);
#pragma unroll
                    for (int u = 0; u < 8; ++u) acc += v[u];
                }
                for (; t < ep.ssq_in_parts; t += kSlices) acc += __ldcg(col + (size_t)t * kLoRows);
            }
            s_part[slice][col128] = acc;
            __syncthreads();
            if (threadIdx.x < LLMCAD_MAX_TREE) {
                float sum = 0.f;
#pragma unroll
                for (int q = 0; q < kSlices; ++q) sum += s_part[q][threadIdx.x];
                s_rs[n0 + threadIdx.x] = rsqrtf(sum / (float)ep.norm_d + ep.eps);
            }
            __syncthreads();
        }
    }

    const int ppt = pairs_per_tile(d);
    const int pairs = d.n_tiles * 4, iters = p.n_pad >> 2;
    const int W = (int)gridDim.x * (kFinThreads / 32);
    int k = W / pairs;
    k = k < 1 ? 1 : (k > iters ? iters : k);
    const int groups = W / k;
    const int wg = warp * (int)gridDim.x + (int)blockIdx.x;      // consecutive pairs on different SMs

    for (int round = 0; round < 2; ++round) {
        const bool dry = round == 0;
        if (!dry) {
            // every segment is in the workspace
            if (p.s_done == nullptr) pdl_wait();
            else {
                if (threadIdx.x == 0) late |= !dep_wait_thread(DepWait{p.s_done, 4u * (uint32_t)d.grid, p.wait_limit_ns});
                __syncthreads();
            }
            if (threadIdx.x == 0) LLMCAD_TRACE(10);
        }
        if (wg < groups * k) {
            for (int pair = wg / k; pair < pairs; pair += groups) {
                FinishArgs fa;
                fa.p = &p; fa.d = &d; fa.rs = s_rs;
                fa.tile = pair >> 2; fa.lane_grp = pair & 3;
                fa.a = holders_of(d, ppt, fa.tile * d.halves);
                if (MODE == EPI_SWIGLU) fa.b = holders_of(d, ppt, fa.tile * 2 + 1);
                fa.it_first = wg % k; fa.it_step = k;
                finish_rows_t<G, KB, MODE>(fa, lane, dry);
                if (dry) break;          // one pair is enough to have walked through the code
            }
        }
    }
    if (p.f_done != nullptr) {
        __syncthreads();             // all of this CTA's results are written
        if (threadIdx.x == 0) {
            if (late) atomicCAS(p.status, 0, LLMCAD_ERR_TIMEOUT);
            dep_arrive(p.f_done);
        }
    }
    if (threadIdx.x == 0) LLMCAD_TRACE(12);
}

// ------------------------------------------------------------------------------------------ host

// The driver entry point is fetched through the runtime, so the library does not link libcuda.
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (fn == nullptr) {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(ptr);
    }
    return fn;
}

bool make_tensor_map_bf16(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint32_t box_rows)
{
    auto fn = get_encode_fn();
    if (fn == nullptr) return false;
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {cols * 2};
    cuuint32_t box[2] = {(cuuint32_t)kBlockK, box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

bool make_act_map_bf16(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint32_t box_rows, uint32_t planes,
                       uint64_t plane_rows, uint32_t box_planes)
{
    auto fn = get_encode_fn();
    if (fn == nullptr) return false;
    cuuint64_t dims[3] = {cols, rows, planes};
    cuuint64_t strides[2] = {cols * 2, plane_rows * cols * 2};
    cuuint32_t box[3] = {(cuuint32_t)kBlockK, box_rows, box_planes};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

bool make_packed_map(CUtensorMap *map, const void *tiled, uint64_t bytes)
{
    auto fn = get_encode_fn();
    if (fn == nullptr) return false;
    cuuint64_t dims[2] = {256, bytes / 512};
    cuuint64_t strides[1] = {512};
    cuuint32_t box[2] = {256, kATileBytes / 512};
    cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(tiled), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool make_tensor_map_bf16_3d(CUtensorMap *map, const void *base, const uint64_t dims[3], const uint64_t strides_bytes[2],
                             const uint32_t box[3])
{
    auto fn = get_encode_fn();
    if (fn == nullptr) return false;
    cuuint64_t d[3] = {dims[0], dims[1], dims[2]};
    cuuint64_t s[2] = {strides_bytes[0], strides_bytes[1]};
    cuuint32_t b[3] = {box[0], box[1], box[2]};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), d, s, b, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

size_t gemm_tc_partial_floats(int n_sms, int max_tiles, int max_n_pad) { return (size_t)2 * (max_tiles + n_sms) * slot_floats(max_n_pad); }

size_t gemm_tc_wide_partial_floats(int n_sms, int max_rows, int d)
{
    // the layer's GEMMs only: 3d and d rows, and two weight tiles per output tile of the FFN's
    const int tiles = 2 * ((max_rows + kTileM - 1) / kTileM), qkv = (3 * d + kTileM - 1) / kTileM;
    return (size_t)((tiles > qkv ? tiles : qkv) + n_sms) * slot_floats(kLoRows);
}

GemmDesc make_gemm_desc(int n_in, const EpiParams &ep, const void *w_tiled, bool w4)
{
    GemmDesc d{};
    d.halves = ep.mode == EPI_SWIGLU ? 2 : 1;
    d.n_tiles = (ep.n_out + kTileM - 1) / kTileM;
    d.kb_per_tile = (n_in + kBlockK - 1) / kBlockK;
    d.pair_k = kMaxPairK;
    d.items_per_cta = 0;
    d.grid = 0;
    d.w_tiled = static_cast<const uint8_t *>(w_tiled);
    d.up_tile_offset = d.n_tiles;
    d.w4 = w4 ? 1 : 0;
    d.ep = ep;
    return d;
}

namespace {
// tuning aids from the environment, read once per process
struct Tuning {
    int pair_k = 0, stages_cap = 0, w4_xstages = kMaxXStages, w4_pstages = kMaxPStages, cta_pair_min = -1;
    Tuning()
    {
        if (const char *e = getenv("LLMCAD_GEMM_PAIR_K")) { const int v = atoi(e); if (v == 1 || v == 2) pair_k = v; }
        if (const char *e = getenv("LLMCAD_GEMM_STAGES")) { const int v = atoi(e); if (v >= 2) stages_cap = v; }
        if (const char *e = getenv("LLMCAD_CTA_PAIR_MIN")) cta_pair_min = atoi(e);
        if (const char *e = getenv("LLMCAD_W4_XSTAGES")) { const int v = atoi(e); if (v >= 2 && v <= kMaxXStages) w4_xstages = v; }
        if (const char *e = getenv("LLMCAD_W4_PSTAGES")) { const int v = atoi(e); if (v >= 2 && v <= kMaxPStages) w4_pstages = v; }
    }
};
const Tuning &tuning()
{
    static const Tuning t;
    return t;
}
}  // namespace

// Pairs from 65 nodes on (80 padded), and from 49 on (64 padded) in passes of models at least 4096 wide. Against one
// kernel per CTA, whole passes: 16 and 32 nodes 3-6 % slower (the two cluster barriers at either end of the kernel sit in
// every hand-over), 45 nodes 1-2 % slower at 7B and 1-2 % faster at 13B, 80 nodes 1.5-2.4 % faster, 128 nodes 7 %. At 49 and
// 64 nodes it is the width that decides (us, pairs / not, 3 or 4 layers): d 512 182.6 / 170.2 and 180.3 / 168.4, d 2048 282.8 /
// 270.5 and 282.8 / 271.6, d 3072 361.1 / 353.2 and 361.8 / 354.5, 7B 502.8 / 499.2 and 500.1 / 508.1, 13B 526.3 / 538.0 and 517.1 /
// 542.8, 30B 761.7 / 770.0 and 763.5 / 779.5. A GEMM on its own (d_model 0) takes them from 65 on: with 64 nodes 4096 x 4096 would
// take 18.0 us instead of 16.5, 1536 x 512 12.4 instead of 10.3. The MMA's N has to be a multiple of 32.
bool gemm_takes_pairs(int n_pad, bool comp, int d_model)
{
    if (n_pad > 128) return true;
    const int nb = n_pad * (comp ? 2 : 1), tuned = tuning().cta_pair_min, least = tuned >= 0 ? tuned : d_model >= 4096 ? 64 : 80;
    return least > 0 && n_pad >= least && nb % 32 == 0;
}

cudaError_t plan_gemm_tc(GemmParams &p, int n_sms)
{
    const Tuning &tune = tuning();
    // Ring items of two k-blocks (one 32 KB weight copy each) unless the activation tiles are so wide
    // (hi | lo planes of more than 64 nodes) that only two stages would fit. Measured on B200 in passes of 16 layers
    // of the 7B shape: single k-blocks cost 1.4 % at 1 and 16 nodes and 0.5 % at 32, and gain 2.3 % at 80 and 128. At 33
    // to 48 nodes three stages of two k-blocks leave 28 KB of shared memory unused, seven of one k-block fill it: 1673 ->
    // 1652 us (16 layers of the 7B shape, 45 nodes), 1482 -> 1458 (10 of 13B), d 3072 (4 layers) 339.1 -> 337.4. Narrower models
    // have too few k-blocks per CTA to gain (d 2560 level, d 2048 261.8 -> 263.4, d 1024 190.2 -> 192.1), and a GEMM on its own
    // with as many MMA columns loses (1536 x 512, 112 nodes: 10.7 -> 12.0), so both keep two. All GEMMs of a pass take the
    // same: with the large ones alone on single k-blocks d 3072 takes 341.7. The work is cut by two k-blocks either way, so
    // that the sums stay those of the INT4 kernel.
    const bool wide = p.n_pad > 128;
    const int nb = p.n_pad * (p.comp && !wide ? 2 : 1);       // MMA N
    if (nb > 256 || p.n_pad < 16 || p.n_pad % 16 || (wide && (!p.pairs || !p.comp || p.n_pad != 256))) return cudaErrorInvalidValue;
    int pair_k = nb > 128 ? 1 : kMaxPairK;
    if (tune.pair_k && !wide) pair_k = tune.pair_k;
    GemmDesc &d = p.g;
    int cut = 1;              // items by which the work is cut
    if (p.wide_model && p.comp && p.n_pad == 48 && !tune.pair_k && !p.pairs && !d.w4 && d.kb_per_tile % 2 == 0) {
        pair_k = 1;
        cut = 2;
    }
    d.pair_k = pair_k;
    // the items are split evenly over one CTA (CTA pair) per SM (two SMs), fewer when there are fewer items
    d.group = p.pairs ? 2 : 1;
    const int vtiles = d.n_tiles * d.halves;
    const long long total = (long long)(p.pairs ? (vtiles + 1) / 2 : vtiles) * pairs_per_tile(d);
    if (total < 1) return cudaErrorInvalidValue;
    long long groups = n_sms / d.group;
    if (groups > total / cut) groups = total / cut;
    const long long ipc = (total / cut + groups - 1) / groups * cut;
    d.items_per_cta = (int)ipc;
    d.grid = (int)((total + ipc - 1) / ipc) * d.group;
    return cudaSuccess;
}

cudaError_t launch_gemm_tc(const GemmMaps &maps, GemmParams &p, int n_sms, size_t partial_floats, cudaStream_t st, int *launched)
{
    if (launched) *launched = 0;
    const Tuning &tune = tuning();
    {
        const cudaError_t e = plan_gemm_tc(p, n_sms);
        if (e != cudaSuccess) return e;
    }
    GemmDesc &d = p.g;
    const bool wide_in = p.n_pad > 128;
    const int nb = p.n_pad * (p.comp && !wide_in ? 2 : 1);
    const int pair_k = d.pair_k, grid = d.grid;
    const long long ipc = d.items_per_cta;
    if ((size_t)(d.n_tiles * d.halves + grid) * slot_floats(p.n_pad) > partial_floats) return cudaErrorInvalidValue;
    // activation bytes of a k-block per CTA: all rows, or half of them in a pair (both planes when wide)
    const size_t act_bytes = (size_t)nb * kBlockK * 2 / (p.pairs && !d.w4 && !wide_in ? 2 : 1);
    const size_t stage_bytes = (size_t)pair_k * ((size_t)kATileBytes + act_bytes);
    // One CTA per SM with the whole shared memory as the ring.
    // two accumulators of MMA N columns each: two buffers or, wide, the sums of the hi and of the lo plane
    int cols = 2 * nb, pow2 = 32;
    while (pow2 < cols) pow2 <<= 1;
    p.tmem_cols = pow2;
    // the ring takes what the SM has, less the room that the finishing CTA of the previous GEMM needs beside it
    const size_t full_limit = 227 * 1024 - 1024 /*alignment slack*/ - 2048 /*static*/ - (kFinSmem + 4096);
    int stages = (int)(full_limit / stage_bytes);
    if (stages > kMaxStages) stages = kMaxStages;
    if (tune.stages_cap && tune.stages_cap < stages) stages = tune.stages_cap;   // tuning aid: cap the ring depth
    if (stages < 2) return cudaErrorInvalidConfiguration;
    size_t smem = (size_t)stages * stage_bytes + 1024;
    p.pstages = p.astages = p.acc_bufs = 0;
    if (d.w4) {
        // Three rings of items of 2 pair_k k-blocks (see the kernel). Tensor memory, all 512 columns: two accumulators if
        // two items of expanded weights (32 columns per k-block) fit beside them, else one. Shared memory: as many
        // activation items as there are expanded ones if they fit beside two packed ones, the rest packed items.
        if (d.w_tiled == nullptr) return cudaErrorInvalidValue;
        const int sk = 2 * pair_k;
        p.acc_bufs = 512 - 2 * nb >= 2 * sk * 32 ? 2 : 1;
        stages = (512 - p.acc_bufs * nb) / (32 * sk);
        if (stages > tune.w4_xstages) stages = tune.w4_xstages;
        const size_t pstage = (size_t)sk * kW4TileBytes, astage = (size_t)sk * nb * kBlockK * 2;
        int ast = (int)((full_limit - 2 * pstage) / astage);
        if (ast > stages) ast = stages;      // (the loader relies on it)
        int pst = (int)((full_limit - (size_t)ast * astage) / pstage);
        if (pst > tune.w4_pstages) pst = tune.w4_pstages;
        if (ast < 2 || pst < 2 || stages < 2) return cudaErrorInvalidConfiguration;
        p.pstages = pst;
        p.astages = ast;
        p.tmem_cols = 512;
        smem = (size_t)ast * astage + (size_t)pst * pstage + 1024;
        // as much as the bf16 kernels ask for, so that no second streaming CTA (and its tensor memory) settles beside it
        if (smem < full_limit) smem = full_limit;
    }
    p.stages = stages;
    static PerDeviceOnce attr_set;
    if (attr_set.needed()) {
        cudaError_t e = cudaSuccess;
        typedef void (*SKernel)(GemmMaps, GemmParams);
        const SKernel all[7] = {gemm_stream_kernel<1>, gemm_stream_kernel<2>, gemm_w4_kernel<1>, gemm_w4_kernel<2>,
                                gemm_pair_kernel<1, false>, gemm_pair_kernel<2, false>, gemm_pair_kernel<1, true>};
        // An SM splits its on-chip memory between shared memory and L1 when it is empty, to fit the kernel that
        // arrives; a streaming CTA of 195 KB would get a 196 KB split, and the finishing CTA of the same GEMM
        // could not settle beside it. Every kernel of the GEMM asks for the largest shared-memory split.
        for (int i = 0; i < 7 && e == cudaSuccess; ++i) {
            e = cudaFuncSetAttribute(all[i], cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024 - 2048);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(all[i], cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        }
        if (e != cudaSuccess) return e;
        attr_set.mark();
    }
    if (p.wait_limit_ns == 0) p.wait_limit_ns = kDefaultWaitLimitNs;
    {
        LaunchCfg lc(grid, d.w4 ? kW4Threads : kThreads, smem, st, p.pairs && !d.w4 ? 2 : 0);
        cudaError_t e;
#define LLMCAD_BY_K(KERNEL1, KERNEL2) \
    (pair_k == 1 ? cudaLaunchKernelEx(&lc.cfg, KERNEL1, maps, p) : cudaLaunchKernelEx(&lc.cfg, KERNEL2, maps, p))
        if (d.w4) e = LLMCAD_BY_K(gemm_w4_kernel<1>, gemm_w4_kernel<2>);
        else if (p.pairs && wide_in) e = cudaLaunchKernelEx(&lc.cfg, gemm_pair_kernel<1, true>, maps, p);
        else if (p.pairs) e = LLMCAD_BY_K((gemm_pair_kernel<1, false>), (gemm_pair_kernel<2, false>));
        else e = LLMCAD_BY_K(gemm_stream_kernel<1>, gemm_stream_kernel<2>);
#undef LLMCAD_BY_K
        if (e != cudaSuccess) return e;
        if (launched) ++*launched;
    }
    // finishing: (tile, row group) pairs x node groups of four, one warp-iteration each; G node groups and
    // KB segments per round trip so that the warps get through in one round where registers allow
    const long long units = (long long)d.n_tiles * 4 * (p.n_pad / 4);
    const int warps_per_cta = kFinThreads / 32;
    int fgrid = (int)((units + warps_per_cta - 1) / warps_per_cta);
    if (fgrid > n_sms) fgrid = n_sms;
    const long long per_warp = (units + (long long)fgrid * warps_per_cta - 1) / ((long long)fgrid * warps_per_cta);
    const int max_parts = (int)((pairs_per_tile(d) + ipc - 1) / ipc) + 1;
    const bool wide = max_parts > 4;           // many segments per tile (tiles split over many CTAs)
    const bool two = per_warp >= 2;            // several node groups per warp
    const bool four = per_warp >= 4 && max_parts <= 2;   // many of them, and one or two segments each
    typedef void (*FinKernel)(GemmParams);
    FinKernel fk = nullptr;
#define LLMCAD_PICK(MODE)                                                                                            \
    fk = wide ? (FinKernel)gemm_finish_kernel<MODE, 1, 8>                                                            \
              : (four ? (FinKernel)gemm_finish_kernel<MODE, 4, 2>                                                            \
                      : (two ? (FinKernel)gemm_finish_kernel<MODE, 2, 4> : (FinKernel)gemm_finish_kernel<MODE, 1, 4>))
    switch (d.ep.mode) {
    case EPI_QKV: LLMCAD_PICK(EPI_QKV); break;
    case EPI_RESID: LLMCAD_PICK(EPI_RESID); break;
    case EPI_SWIGLU:
        fk = wide ? (FinKernel)gemm_finish_kernel<EPI_SWIGLU, 1, 4> : (two ? (FinKernel)gemm_finish_kernel<EPI_SWIGLU, 2, 2> : (FinKernel)gemm_finish_kernel<EPI_SWIGLU, 1, 4>);
        break;
    default: LLMCAD_PICK(EPI_PLAIN); break;
    }
#undef LLMCAD_PICK
    {
        // once per finishing kernel and device (see above)
        static PerDeviceOnce fin_set[4][4];
        PerDeviceOnce &once = fin_set[d.ep.mode & 3][wide ? 0 : (four ? 3 : (two ? 1 : 2))];
        if (once.needed()) {
            const cudaError_t e = cudaFuncSetAttribute(fk, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
            if (e != cudaSuccess) return e;
            once.mark();
        }
    }
    p.f_grid = fgrid;
    LaunchCfg lf(fgrid, kFinThreads, kFinSmem, st);
    const cudaError_t e = cudaLaunchKernelEx(&lf.cfg, fk, p);
    if (e == cudaSuccess && launched) ++*launched;
    return e;
}

}  // namespace llmcad
