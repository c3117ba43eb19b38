// A bf16 pass over few nodes (decoding, small trees, the generating side) in one cooperative kernel.
//
// With few nodes a pass is the weight stream and little else, and what kept it from the rate of the memory was the
// hand-over between its kernels: five phases per layer, each ending in an all-to-all dependency, and behind each the
// HBM idle for the part of it that the next kernel's ring does not cover. Here one CTA per SM stays for the whole pass
// and its ring runs on through the phases: the producer asks for the weights (and the prefix keys and values) of all
// phases one after the other and never waits for anything but room, so that a barrier over the grid costs memory time
// only beyond what the ring holds. 7B shape, 32 layers, prefix 512, one node: 2822 -> 2551 us a pass, 5.3 TB/s. A layer is
// 77 us, of which the weights take 57 at the rate of a plain read and the attention phase 7.5.
//
//   warps 8-11    weight producers, each for every fourth slot of the ring. A CTA owns the same share of the output rows of a
//                 GEMM whatever its K, so that no sum is cut between CTAs and nothing has to be finished elsewhere: runs
//                 of rows of the packed tiles (128-byte rows, swizzled), one bulk copy per run and k-block, by a lane each.
//   warp 12       polls the grid barrier, then copies the phase's input into a ring of its own. Inputs are stored by
//                 whoever produces them as the B fragments of the MMA: [32 columns of K][node, plane][32], so that a
//                 lane's 16 bytes serve two MMAs.
//   warps 0-7     mma.sync m16n8k16: weights on the M side, (node, hi/lo plane) as the eight columns of the N side. Groups of warps take the
//                 k-blocks in turn; the sums are added in shared memory in a fixed order, and the epilogue (norm factor,
//                 rotary, K/V write, SwiGLU, residual) runs where they lie. The residual stream stays in shared memory.
//   INT4 weights  take the same plan, operands and order of sums (the passes are equal bit for bit): codes and exponents go through
//                 the ring as they are packed, by ordinary asynchronous copies, and are expanded on the way into the MMA. 7B widths,
//                 4 layers, prefix 512, one / four nodes: 305 / 329 us, with one kernel per step 312 / 314; 13B (3 layers) 322 / 344,
//                 313 / 316; d 512 112 / 119, 151 / 152. The latency of a k-block per warp bounds it, not the HBM.
//   attention     (head, key range) per CTA: prefix tiles of 32 keys come through the weight ring, scores and outputs
//                 by mma.sync with hi and lo planes as the two halves of the 16 rows, the new nodes' keys and values in
//                 fp32; the CTA that finishes a head last merges its key ranges.
//
// The code of a phase runs once per phase: one copy of everything, few variants, or instruction fetches set the pace.
// What another CTA wrote in this kernel is read past L1 (ld.cg, bulk copies). Every wait is bounded; when one runs
// out the CTA sets the status word and leaves, and so do the others.
#include "mbar.cuh"
#include "pass_stream.cuh"
#include "tree_dev.cuh"

namespace llmcad {

bool make_tensor_map_bf16_3d(CUtensorMap *map, const void *base, const uint64_t dims[3], const uint64_t strides_bytes[2], const uint32_t box[3]);

namespace {

constexpr int kWarps = 8;                       // consumers
// A copy costs its warp ~90 cycles to issue and an item ~500 more, all of it latency: one producer got 13 of the 26 bytes
// a cycle that an SM's share of the HBM is.
// INT4 items are many copies of 16 bytes per lane; there every slot of the ring up to seven has a producer of its own.
template <bool W4> constexpr int kProducers = W4 ? 7 : 4;
template <bool W4> constexpr int kThreads = 32 * (kWarps + kProducers<W4> + 1);
constexpr int kMaxSlots = 16;                   // items the ring can hold
constexpr int kMaxItemKb = 6;                   // k-blocks of an item at most
constexpr int kMaxItemKbW4 = 32;                // the same, of INT4 weights (16: 3 % slower, 8: 6 %)
constexpr int kXStages = 2;                     // of the ring of inputs
constexpr int kMt = 3;                          // 16-row tiles of a warp at most
constexpr int kHdim = 128, kKeys = 32;          // head size, keys of a prefix tile
constexpr int kKvItem = 4 * kKeys * 128;        // K and V of a tile, each as two swizzled halves of 64 columns
constexpr int kQRow = 272;                      // bytes of a query row in shared memory
constexpr int kPRow = 136;                      // floats of a partial row in shared memory
constexpr int kMaxResidUnits = 32;              // units of the O and down GEMMs per CTA: one per lane
constexpr int kMaxSms = 160;

// ---- this CTA's share of a GEMM
struct Share {
    int u0, U;                 // units
    int rows, row0, rows_run;  // rows of an item's k-block, first row of a run, rows of a run (two runs with `upper`)
};
__device__ __forceinline__ Share share_of(const StreamGemm &g)
{
    Share s;
    s.u0 = (int)((uint32_t)g.units * blockIdx.x / gridDim.x);
    s.U = (int)((uint32_t)g.units * (blockIdx.x + 1) / gridDim.x) - s.u0;
    s.row0 = g.upper ? s.u0 : 2 * s.u0;
    s.rows_run = g.upper ? s.U : 2 * s.U;
    s.rows = 2 * s.U;
    return s;
}
// part j of `parts` of a share (the lm_head)
__device__ __forceinline__ Share part_of(const Share &a, int j, int parts)
{
    Share s;
    s.u0 = a.u0 + a.U * j / parts;
    s.U = a.u0 + a.U * (j + 1) / parts - s.u0;
    s.row0 = 2 * s.u0;
    s.rows = s.rows_run = 2 * s.U;
    return s;
}
__device__ __forceinline__ int gemm_kind(int step) { return step == 0 ? SG_QKV : step == 2 ? SG_O : step == 3 ? SG_GU : SG_DOWN; }

// ---- this CTA's share of an attention phase
struct AttnShare {
    int head, split, t0, t1;   // tiles of 32 prefix keys
    int any;
};
__device__ __forceinline__ AttnShare attn_share(const StreamPass &p)
{
    AttnShare a;
    a.any = (int)blockIdx.x < p.H * p.splits;
    a.head = (int)blockIdx.x / p.splits;
    a.split = (int)blockIdx.x - a.head * p.splits;
    const int nt = (p.P + p.n_old + kKeys - 1) / kKeys;
    a.t0 = nt * a.split / p.splits;
    a.t1 = a.any ? nt * (a.split + 1) / p.splits : a.t0;
    return a;
}

struct Ctl {
    unsigned long long full[kMaxSlots], empty[kMaxSlots], xfull[kXStages], xempty[kXStages], ready, meet, gone;
    alignas(16) float x[kStreamMaxNodes][2 * kMaxResidUnits];     // residual stream of this CTA's rows
    float rs[kStreamMaxNodes];                                    // norm factors
    Share share[SG_HEAD + kStreamHeadParts];     // worked out once: integer divisions at every phase cost microseconds
    AttnShare attn;
    volatile int abort_flag;
    int last;
    MaskTable table;
};

// ---- INT4 weights (layer matrices only, see pack.cu): a k-block of a CTA's rows in the ring is, per run of rows, the codes of
// its columns 0 .. 31 and then 32 .. 63, 16 bytes a row; behind the runs their exponents, a byte a row, from a multiple of
// 16 rows on (copies move 16 bytes).
__device__ __host__ __forceinline__ int exp_chunks(int row0, int rows_run) { return ((row0 & 15) + rows_run + 15) >> 4; }
__device__ __host__ __forceinline__ int w4_kb_bytes(int row0, int rows_run, int runs) { return runs * (rows_run * 32 + exp_chunks(row0, rows_run) * 16); }
// Two codes of a word as a bf16 pair: OR 0x4300 into each half: 128 + u (u = q + 8); (128 + u) * 2^e - 136 * 2^e = q * 2^e, exact.
// The bf16 bits of 2^e are (e + 127) << 7, those of -136 * 2^e are that + 0x8388.
__device__ __forceinline__ uint32_t expand2(uint32_t word, uint32_t scale)
{
    uint32_t t, r;
    asm("lop3.b32 %0, %1, %2, %3, 0xea;" : "=r"(t) : "r"(word), "r"(0x000f000fu), "r"(0x43004300u));
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(t), "r"(scale), "r"(scale + 0x83888388u));
    return r;
}

// (volatile: they stay behind the barrier wait in front of them)
__device__ __forceinline__ uint4 lds128(uint32_t a)
{
    uint4 r;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(a));
    return r;
}
__device__ __forceinline__ uint32_t lds32v(uint32_t a)
{
    uint32_t r;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(r) : "r"(a));
    return r;
}
__device__ __forceinline__ uint32_t exp_scale(uint32_t a)
{
    int e;
    asm volatile("ld.shared.s8 %0, [%1];" : "=r"(e) : "r"(a));
    return (uint32_t)(e + 127) * 0x00800080u;
}
__device__ __forceinline__ uint32_t lds32(uint32_t a)
{
    uint32_t r;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(r) : "r"(a) : "memory");
    return r;
}
__device__ __forceinline__ void ldsm4(uint32_t a, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void ldsm4_t(uint32_t a, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack2(__nv_bfloat16 a, __nv_bfloat16 b)
{
    return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}
__device__ __forceinline__ void split2(float a, float b, uint32_t &hi, uint32_t &lo)
{
    __nv_bfloat16 ah, al, bh, bl;
    split_bf16(a, ah, al);
    split_bf16(b, bh, bl);
    hi = pack2(ah, bh);
    lo = pack2(al, bl);
}

// Wait of one thread.
__device__ __forceinline__ bool thread_wait(uint32_t bar, uint32_t parity, const Ctl &ctl, uint64_t limit)
{
    uint64_t t0 = 0;
    for (uint32_t it = 1; !mbar_try(bar, parity); ++it) {
        if ((it & 255u) == 0) {
            const uint64_t now = global_timer_ns();
            if (t0 == 0) t0 = now;
            else if (ctl.abort_flag || now - t0 > limit) return false;
        }
    }
    return true;
}
// (The loop that watches the clock is called, not inlined: a walk has four waits, a phase three walks, and what straight-line
// code costs here is its fetch.)
__device__ __noinline__ bool wait_watched(uint32_t bar, uint32_t parity, const Ctl &ctl, uint64_t limit)
{
    return mbar_wait_all(bar, parity, const_cast<volatile int *>(&ctl.abort_flag), limit);
}
__device__ __forceinline__ bool wait_all(uint32_t bar, uint32_t parity, const Ctl &ctl, uint64_t limit)
{
    return __all_sync(0xffffffffu, mbar_try(bar, parity)) || wait_watched(bar, parity, ctl, limit);
}

// ---- a place in the ring: slot and the parity of its turn
struct Place {
    int slot = 0;
    uint32_t turn = 0;
    __device__ __forceinline__ void add(int n, int slots)
    {
        slot += n;
        while (slot >= slots) { slot -= slots; turn ^= 1u; }
    }
};

// ---- weight producer: a warp that fetches the items of its slots, every kProducers-th of the ring. (A slot belongs to
// one producer, which so sees each of its turns: a barrier tells two of them apart and no more.)
template <bool W4>
struct Producer {
    const StreamPass &p;
    const CUtensorMap *map;
    Ctl &ctl;
    uint32_t ring;
    uint64_t policy;
    Place at;
    int issued = 0;
    int ph = -1, pos = 0;                      // the next item: phase and k-block or tile in it
    bool attention = false, codes = false;     // codes: an INT4 matrix
    int layer = 0, kb_all = 0, kb_item = 1, kb_bytes = 0;    // kb_all: k-blocks or tiles in all
    // what this lane copies of an item: one run of rows of one k-block, cut where a tile of 128 rows ends
    const char *src = nullptr;
    int my_k = 1 << 30, my_dst = 0, my_bytes = 0;
    // INT4: the CTA's rows, bytes from a weight tile to the next one below it and from run to run, and this lane's 16 exponents
    int row0 = 0, rows_run = 0, rows = 0, exp_dst = -1;
    uint32_t tile_bytes = 0, exp_src = 0;
    size_t upper = 0;
    const int lane = threadIdx.x & 31, rank = (int)(threadIdx.x >> 5) - kWarps, step, phases;
    __device__ Producer(const StreamPass &p_, const CUtensorMap *m, Ctl &c, uint32_t r)
        : p(p_), map(m), ctl(c), ring(r), step(W4 ? min(kProducers<W4>, p_.slots) : kProducers<W4>), phases(5 * p_.L + (p_.logits != nullptr ? p_.head_parts : 0))
    {
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    }
    __device__ void start()
    {
        if (rank >= step) {            // (a ring of fewer slots)
            ph = phases;
            return;
        }
        next_phase();
        skip(rank);
    }
    __device__ bool done() const { return ph >= phases; }
    // the next phase in which this CTA has something to fetch
    __device__ void next_phase()
    {
        do {
            if (++ph >= phases) return;
            const bool head = ph >= 5 * p.L;
            layer = ph / 5;
            const int st = ph - 5 * layer, kind = head ? SG_HEAD + ph - 5 * p.L : gemm_kind(st);
            attention = !head && st == 1;
            if (attention) {
                kb_all = ctl.attn.t1 - ctl.attn.t0;
                kb_item = 1;
                continue;
            }
            const StreamGemm &g = p.g[head ? SG_HEAD : kind];
            const Share s = ctl.share[kind];
            kb_all = s.U > 0 ? g.kb_all : 0;
            if (kb_all == 0) continue;
            kb_item = g.kb_item;
            codes = W4 && !head;
            if (W4 && codes) {
                const int runs = g.upper ? 2 : 1, chunks = exp_chunks(s.row0, s.rows_run), run = lane >= chunks ? 1 : 0;
                row0 = s.row0; rows_run = s.rows_run; rows = s.rows;
                upper = g.upper;
                tile_bytes = kb_all * kW4TileBytes;
                kb_bytes = w4_kb_bytes(row0, rows_run, runs);
                const int r = (row0 & ~15) + 16 * (lane - run * chunks);
                exp_dst = lane < runs * chunks ? rows * 32 + lane * 16 : -1;
                exp_src = (r >> 7) * tile_bytes + 4096 + (r & 127);
                src = p.base + p.w_off[kind] + p.layer_bytes * (size_t)layer;
                if (run) exp_src += (uint32_t)upper;
                continue;
            }
            kb_bytes = s.rows * 128;
            const int pieces = ((s.row0 & 127) + s.rows_run + 127) >> 7, per_k = (g.upper ? 2 : 1) * pieces;
            my_k = lane / per_k;
            const int rest = lane - my_k * per_k, run = rest >= pieces ? 1 : 0, tile = (s.row0 >> 7) + rest - run * pieces;
            const int r = max(s.row0, tile * 128);
            my_bytes = (min(s.row0 + s.rows_run, tile * 128 + 128) - r) * 128;
            my_dst = my_k * kb_bytes + (run * s.rows_run + r - s.row0) * 128;
            src = p.base + p.w_off[head ? SG_HEAD : kind] + (head ? 0 : p.layer_bytes * (size_t)layer) + (run ? g.upper : 0) +
                  (size_t)(tile * kb_all + my_k) * 16384 + (r & 127) * 128;
        } while (kb_all == 0);
        pos = 0;
    }
    __device__ void skip(int n)
    {
        at.add(n, p.slots);
        for (; n > 0 && !done(); --n) {
            pos += kb_item;
            if (pos >= kb_all) next_phase();
        }
    }
    __device__ bool free_now() const { return mbar_test_all(smem_u32(&ctl.empty[at.slot]), at.turn ^ 1u); }
    __device__ bool wait_free() const { return wait_all(smem_u32(&ctl.empty[at.slot]), at.turn ^ 1u, ctl, p.wait_limit_ns); }
    __device__ void fetch()
    {
        const uint32_t full = smem_u32(&ctl.full[at.slot]), dst = ring + at.slot * p.slot_bytes;
        const int nkb = min(kb_item, kb_all - pos);
        if (W4 && codes && !attention) {
            fetch_codes(full, dst, nkb);
            ++issued;
            skip(at.slot + step < p.slots ? step : p.slots - at.slot + rank);
            return;
        }
        // (INT4: the slot's last content may have come by ordinary copies)
        if (W4) asm volatile("fence.proxy.async;" ::: "memory");
        if (lane == 0) mbar_expect_tx(full, attention ? kKvItem : nkb * kb_bytes);
        else if (W4) mbar_arrive(full);
        __syncwarp();
        if (attention) {
            if (lane < 4)
                asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                             ::"r"(dst + lane * (kKvItem / 4)), "l"(map), "r"((lane & 1) * 64), "r"((ctl.attn.t0 + pos) * kKeys),
                             "r"((layer * 2 + (lane >> 1)) * p.H + ctl.attn.head), "r"(full)
                             : "memory");
        } else if (my_k < nkb) {
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
                         ::"r"(dst + my_dst), "l"(src + (size_t)pos * 16384), "r"(my_bytes), "r"(full), "l"(policy)
                         : "memory");
        }
        ++issued;
        skip(at.slot + step < p.slots ? step : p.slots - at.slot + rank);
    }
    // An item of an INT4 matrix: 16 bytes per lane and copy. (Bulk copies would be three per run, piece and k-block, of 48 to
    // 1300 bytes each.) Every lane arrives when its copies have landed.
    __device__ void fetch_codes(uint32_t full, const uint32_t dst0, int nkb)
    {
        auto copy = [&](uint32_t to, const char *from) {
            asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(to), "l"(from), "l"(policy) : "memory");
        };
        const char *first = src + (size_t)pos * kW4TileBytes;
        for (int x = lane; x < rows; x += 32) {
            const int run = x >= rows_run ? 1 : 0, in_run = x - run * rows_run, r = row0 + in_run;
            const char *from = first + (run ? upper : 0) + (size_t)((r >> 7) * tile_bytes + (r & 127) * 16);
            uint32_t to = dst0 + run * rows_run * 32 + in_run * 16;
            for (int k = 0; k < nkb; ++k, from += kW4TileBytes, to += kb_bytes) {
                copy(to, from);
                copy(to + rows_run * 16, from + 2048);
            }
        }
        if (exp_dst >= 0) {
            const char *from = first + exp_src;
            uint32_t to = dst0 + exp_dst;
            for (int k = 0; k < nkb; ++k, from += kW4TileBytes, to += kb_bytes) copy(to, from);
        }
        asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(full) : "memory");
    }
};

// ---- consumer state that runs on through the phases
struct Consumer {
    Place at;                             // in the ring: the phase's first item
    uint32_t xs = 0;                      // input stages taken so far
    uint32_t phase = 0, meets = 0;        // phases begun (0 is the embedding), barriers among the consumer warps passed
    bool ok = true;
};

struct Env {
    const StreamPass &p;
    Ctl &ctl;
    uint32_t ring;
    float *red;                           // reduction scratch
    float2 *cs;                           // rotary factors [node][unit] of this CTA's Q and K rows
    int n, warp, lane;
};

__device__ __forceinline__ bool wait_ready(const Env &e, Consumer &c)
{
    if (c.ok) c.ok = wait_all(smem_u32(&e.ctl.ready), c.phase & 1u, e.ctl, e.p.wait_limit_ns);
    ++c.phase;
    return c.ok;
}
// Barrier among the consumer warps. A hardware barrier has no bound: a warp whose wait ran out would leave the others in it.
__device__ __forceinline__ bool meet(const Env &e, Consumer &c)
{
    if (!c.ok) return false;
    __syncwarp();
    if (e.lane == 0) mbar_arrive(smem_u32(&e.ctl.meet));
    c.ok = wait_all(smem_u32(&e.ctl.meet), c.meets & 1u, e.ctl, e.p.wait_limit_ns);
    ++c.meets;
    return c.ok;
}
// This CTA's part of the phase is written: one arrival at the grid barrier.
__device__ __forceinline__ void arrive_grid(const Env &e, Consumer &c)
{
    if (meet(e, c) && threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(e.p.bar) : "memory");
        mbar_arrive(smem_u32(&e.ctl.gone));
    }
}

// Byte offset of (column k, node) in an input of C columns; the lo plane is 64 bytes behind.
__device__ __forceinline__ size_t frag_off(int k, int node, int C) { return ((size_t)(k >> 5) * C + 2 * node) * 64 + (k & 31) * 2; }

// The input of a norm-folded GEMM from this lane's two new values of the residual stream: gain * x as a fragment, and
// the sum of squares of the CTA's rows.
__device__ __forceinline__ void emit_resid(const Env &e, int node, bool has, int k, float v0, float v1, uint32_t gain2, int first, int C, float *ssq)
{
    float ss = 0.f;
    if (has) {
        ss = v0 * v0 + v1 * v1;
        const float g0 = __uint_as_float(gain2 << 16), g1 = __uint_as_float(gain2 & 0xffff0000u);
        uint32_t hi, lo;
        split2(v0 * g0, v1 * g1, hi, lo);
        if (node >= first) {
            char *dst = static_cast<char *>(e.p.xn) + frag_off(k, node - first, C);
            *reinterpret_cast<uint32_t *>(dst) = hi;
            *reinterpret_cast<uint32_t *>(dst + 64) = lo;
        }
    }
    for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (e.lane == 0) ssq[(size_t)node * gridDim.x + blockIdx.x] = ss;
}

// Where a lane finds its rows of the 16-row tiles of an item.
struct ATile {
    int lo[2], up[2];          // first and second row of its unit, for the even and odd 32 columns of a k-block
    int kb_bytes, mt_stride;
    int exp_lo, exp_up, exp_stride;      // INT4: their exponents
};
// A k-block's operands of a warp: M tiles of 16 rows, two times 32 columns (the second is left out where K ends in the
// middle). Lane (g, t) holds columns 8t .. 8t+7 of 32 on both sides, the first four for one MMA and the others for the
// next. What lanes of columns and rows that do not exist read (other data of the rings) ends in sums that nobody takes.
template <int M>
struct Block {
    uint4 b[2], lo[2][M], up[2][M];
    __device__ __forceinline__ void load(const ATile &at, uint32_t w, uint32_t x, int x_step, bool whole)
    {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            b[q] = lds128(x + q * x_step);
#pragma unroll
            for (int i = 0; i < M; ++i) {
                lo[q][i] = lds128(w + at.lo[q] + i * at.mt_stride);
                up[q][i] = lds128(w + at.up[q] + i * at.mt_stride);
            }
        }
        if (!whole) b[1] = make_uint4(0, 0, 0, 0);     // the weights there are zero
    }
    __device__ __forceinline__ void mma(float (&acc)[kMt][4]) const
    {
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int i = 0; i < M; ++i) mma_bf16(acc[i], lo[q][i].x, up[q][i].x, lo[q][i].y, up[q][i].y, b[q].x, b[q].y);
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int i = 0; i < M; ++i) mma_bf16(acc[i], lo[q][i].z, up[q][i].z, lo[q][i].w, up[q][i].w, b[q].z, b[q].w);
    }
};

// The same of INT4 weights: eight codes per row and lane in place of 16 bytes. The MMAs are those above, in their order, on the
// same bf16 values: a pass with INT4 weights is the pass with the dequantised ones bit for bit.
template <int M>
struct CodeBlock {
    uint4 b[2];
    uint32_t code[2][2][M], scale[2][M];        // [half][first, second row]
    __device__ __forceinline__ void load(const ATile &at, uint32_t a, uint32_t x, int x_step, bool)
    {
#pragma unroll
        for (int i = 0; i < M; ++i) {
            scale[0][i] = exp_scale(a + at.exp_lo + i * at.exp_stride);
            scale[1][i] = exp_scale(a + at.exp_up + i * at.exp_stride);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            b[q] = lds128(x + q * x_step);
#pragma unroll
            for (int i = 0; i < M; ++i) {
                code[q][0][i] = lds32v(a + at.lo[q] + i * at.mt_stride);
                code[q][1][i] = lds32v(a + at.up[q] + i * at.mt_stride);
            }
        }
    }
    template <int ROUND>
    __device__ __forceinline__ void round(float (&acc)[kMt][4]) const
    {
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int i = 0; i < M; ++i) {
                const uint32_t c0 = code[q][0][i] >> (8 * ROUND), c1 = code[q][1][i] >> (8 * ROUND), s0 = scale[0][i], s1 = scale[1][i];
                mma_bf16(acc[i], expand2(c0, s0), expand2(c1, s1), expand2(c0 >> 4, s0), expand2(c1 >> 4, s1), ROUND ? b[q].z : b[q].x, ROUND ? b[q].w : b[q].y);
            }
    }
    __device__ __forceinline__ void mma(float (&acc)[kMt][4]) const
    {
        round<0>(acc);
        round<1>(acc);
    }
};

// The main loop of a GEMM phase for a warp: k-blocks kq, kq + kg, ... of `kb_all`. False when a wait ran out.
struct Walk {
    uint32_t full, empty, ring, x_ring, xfull, xempty;                // shared-memory addresses
    int slots, slot_bytes, x_stage_bytes, kg, kb_item, kb_all, n_items, n_k32, x_kb, x_bytes_kb;
};
template <int M, typename Operands>
__device__ __forceinline__ bool gemm_walk(float (&acc)[kMt][4], const ATile at, const Walk k, int kq, Place pl, uint32_t &xs, const Ctl &ctl, uint64_t limit, int lane)
{
    int kb = kq, item = 0, in_item = kq, x_st = 0, in_x = kq;         // kb = item * kb_item + in_item = x_st * x_kb + in_x
    bool landed = false;                                              // the item has been seen to land
    // Every warp waits for every item and gives it back, in order, also where it has no part of it: a barrier tells two
    // turns of a slot apart and no more, and a warp that ran ahead or fell behind by one would mistake them.
    auto land = [&]() {
        if (!landed && !wait_all(k.full + pl.slot * 8, pl.turn, ctl, limit)) return false;
        landed = true;
        return true;
    };
    auto give_back = [&]() {
        if (!land()) return false;
        __syncwarp();
        if (lane == 0) mbar_arrive(k.empty + pl.slot * 8);
        pl.add(1, k.slots);
        ++item;
        landed = false;
        return true;
    };
    const int x_stages = (k.kb_all + k.x_kb - 1) / k.x_kb;
    auto x_wait = [&]() { return wait_all(k.xfull + (xs % kXStages) * 8, (xs / kXStages) & 1u, ctl, limit); };
    auto x_next = [&]() {
        __syncwarp();
        if (lane == 0) mbar_arrive(k.xempty + (xs % kXStages) * 8);
        ++xs;
        ++x_st;
    };
    if (!x_wait()) return false;
    Operands blk;
    while (kb < k.kb_all) {
        for (; in_item >= k.kb_item; in_item -= k.kb_item)
            if (!give_back()) return false;
        for (; in_x >= k.x_kb; in_x -= k.x_kb) {
            x_next();
            if (!x_wait()) return false;
        }
        if (!land()) return false;
        blk.load(at, k.ring + pl.slot * k.slot_bytes + in_item * at.kb_bytes, k.x_ring + (xs % kXStages) * k.x_stage_bytes + in_x * k.x_bytes_kb,
                 k.x_bytes_kb / 2, 2 * kb + 1 < k.n_k32);
        blk.mma(acc);
        kb += k.kg;
        in_item += k.kg;
        in_x += k.kg;
    }
    while (item < k.n_items)
        if (!give_back()) return false;
    while (x_st < x_stages) {
        x_next();
        if (x_st < x_stages && !x_wait()) return false;
    }
    return true;
}

// One GEMM phase.
template <bool W4>
__device__ __forceinline__ void gemm_phase(const Env &e, Consumer &c, int kind, int layer, int part)
{
    const StreamPass &p = e.p;
    const StreamGemm g = p.g[kind];          // (copies: behind every barrier a reference would be read again)
    const Share s = e.ctl.share[kind + part];
    const bool head = kind == SG_HEAD, norm = kind == SG_QKV || kind == SG_GU || head, resid = kind == SG_O || kind == SG_DOWN;
    const int n = head ? e.n - p.head_first : e.n, C = 2 * n;
    const int units_pad = (s.U + 15) / 16 * 16 + 4;
    uint32_t gain2 = 0;
    if (resid && e.lane < s.U) {
        const size_t off = kind == SG_O ? p.layer_bytes * (size_t)layer + p.ffn_norm
                           : layer + 1 < p.L ? p.layer_bytes * (size_t)(layer + 1) + p.attn_norm : p.final_norm;
        gain2 = __ldg(reinterpret_cast<const uint32_t *>(p.base + off) + s.u0 + e.lane);
    }
    const int kq = e.warp % g.kg, mq = e.warp / g.kg;
    const int gi = e.lane >> 2, t = e.lane & 3;
    // The eight units of a 16-row tile are dealt to the row groups so that two neighbours read rows whose swizzle
    // differs in its upper bit: their eight 16-byte reads then fall on different banks.
    const int pu = g.upper ? ((gi & 1) << 2) | (gi >> 1) : (gi & 4) | ((gi & 1) << 1) | ((gi >> 1) & 1);
    const int mt_all = (s.U + 7) / 8, row_l = (g.upper ? 1 : 2) * pu;
    const int mtn = mq < mt_all ? (mt_all - mq + g.mg - 1) / g.mg : 0;
    ATile at;
    const int sw = ((s.row0 + row_l) & 7) << 4, sw_up = g.upper ? sw : sw ^ 16, mt_bytes = (g.upper ? 8 : 16) * 128;
    at.kb_bytes = s.rows * 128;
    at.mt_stride = g.mg * mt_bytes;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        at.lo[h] = row_l * 128 + mq * mt_bytes + (((h * 4 + t) << 4) ^ sw);
        at.up[h] = row_l * 128 + mq * mt_bytes + (g.upper ? s.rows_run * 128 : 128) + (((h * 4 + t) << 4) ^ sw_up);
    }
    const bool codes = W4 && !head;
    if (W4 && codes) {
        const int mt_rows = g.upper ? 8 : 16, row = row_l + mq * mt_rows;
        at.kb_bytes = w4_kb_bytes(s.row0, s.rows_run, g.upper ? 2 : 1);
        at.mt_stride = g.mg * mt_rows * 16;
        at.exp_stride = g.mg * mt_rows;
        at.exp_lo = s.rows * 32 + (s.row0 & 15) + row;
        at.exp_up = at.exp_lo + (g.upper ? exp_chunks(s.row0, s.rows_run) * 16 : 1);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            at.lo[h] = (h * s.rows_run + row) * 16 + t * 4;
            at.up[h] = at.lo[h] + (g.upper ? s.rows_run * 32 : 16);
        }
    }
    if (part == 0 && !wait_ready(e, c)) return;
    if (s.U > 0) {
        // requested now, used behind the main loop: the sums of squares of a node per warp
        float sq[kMaxSms / 32];
        if (norm && e.warp < n) {
            const float *ssq = p.ssq + (size_t)((kind == SG_GU ? kStreamMaxNodes : 0) + e.warp + (head ? p.head_first : 0)) * gridDim.x;
#pragma unroll
            for (int j = 0; j < kMaxSms / 32; ++j) sq[j] = e.lane + 32 * j < (int)gridDim.x ? __ldcg(ssq + e.lane + 32 * j) : 0.f;
        }
        float acc[kMt][4];
#pragma unroll
        for (int i = 0; i < kMt; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;

        const Walk walk{smem_u32(&e.ctl.full[0]), smem_u32(&e.ctl.empty[0]), e.ring, e.ring + p.x_off + e.lane * 16, smem_u32(&e.ctl.xfull[0]),
                        smem_u32(&e.ctl.xempty[0]), p.slots, p.slot_bytes, p.x_stage_bytes, g.kg, g.kb_item, g.kb_all, g.n_items,
                        g.K / 32, g.x_kb, C * 128};
        if (W4 && codes) {
            if (mtn == 2) c.ok = gemm_walk<2, CodeBlock<2>>(acc, at, walk, kq, c.at, c.xs, e.ctl, p.wait_limit_ns, e.lane);
            else if (mtn == 3) c.ok = gemm_walk<3, CodeBlock<3>>(acc, at, walk, kq, c.at, c.xs, e.ctl, p.wait_limit_ns, e.lane);
            else c.ok = gemm_walk<1, CodeBlock<1>>(acc, at, walk, kq, c.at, c.xs, e.ctl, p.wait_limit_ns, e.lane);
        } else if (mtn == 2) c.ok = gemm_walk<2, Block<2>>(acc, at, walk, kq, c.at, c.xs, e.ctl, p.wait_limit_ns, e.lane);
        else if (mtn == 3) c.ok = gemm_walk<3, Block<3>>(acc, at, walk, kq, c.at, c.xs, e.ctl, p.wait_limit_ns, e.lane);
        else c.ok = gemm_walk<1, Block<1>>(acc, at, walk, kq, c.at, c.xs, e.ctl, p.wait_limit_ns, e.lane);      // (no tile at all: a tile of other data)
        if (!c.ok) return;
        c.at.add(g.n_items, p.slots);

        // ---- sums of the K parts: [part][node][unit] (first row, second row)
        float2 *red = reinterpret_cast<float2 *>(e.red);
#pragma unroll
        for (int i = 0; i < kMt; ++i) {
            if (i < mtn) {
                const int unit = (mq + i * g.mg) * 8 + pu;
                if (t < n) red[(kq * n + t) * units_pad + unit] = make_float2(acc[i][0] + acc[i][1], acc[i][2] + acc[i][3]);
            }
        }
        if (norm && e.warp < n) {
            float ss = 0.f;
#pragma unroll
            for (int j = 0; j < kMaxSms / 32; ++j) ss += sq[j];
            for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
            if (e.lane == 0) e.ctl.rs[e.warp] = rsqrtf(ss / (float)p.d + p.eps);
        }
        if (!meet(e, c)) return;
        // ---- epilogue: a warp takes 32 units of a node
        const int chunks = (s.U + 31) / 32;
        int node = 0, chunk = e.warp;
        for (; node < n; chunk += kWarps) {
            while (chunk >= chunks) { chunk -= chunks; ++node; }
            if (node >= n) break;
            const int unit = chunk * 32 + e.lane, ug = s.u0 + unit;
            const bool has = unit < s.U;
            float v0 = 0.f, v1 = 0.f;
            if (has)
                for (int q = 0; q < g.kg; ++q) {
                    const float2 r = red[(q * n + node) * units_pad + unit];
                    v0 += r.x;
                    v1 += r.y;
                }
            if (norm) { v0 *= e.ctl.rs[node]; v1 *= e.ctl.rs[node]; }
            if (kind == SG_QKV) {
                if (!has) continue;
                const int sec = 2 * ug < p.d ? 0 : 2 * ug < 2 * p.d ? 1 : 2, col = 2 * ug - sec * p.d;
                float o0 = v0, o1 = v1;
                if (sec < 2) {
                    const float2 f = e.cs[node * s.U + unit];
                    o0 = v0 * f.x - v1 * f.y;
                    o1 = v0 * f.y + v1 * f.x;
                }
                *reinterpret_cast<float2 *>(p.qkv + ((size_t)sec * kStreamMaxNodes + node) * p.d + col) = make_float2(o0, o1);
                const int slot = p.P + p.n_old + node;
                if (sec > 0 && LLMCAD_CHECK(slot < p.S && col < p.d, p.status)) {
                    const size_t row = ((size_t)(layer * 2 + sec - 1) * p.H + (col >> 7)) * p.S + slot;
                    *reinterpret_cast<uint32_t *>(p.kv + (row * kHdim + (col & 127)) * 2) = pack2(__float2bfloat16_rn(o0), __float2bfloat16_rn(o1));
                }
            } else if (kind == SG_GU) {
                if (!has) continue;
                __nv_bfloat16 hi, lo;
                split_bf16(v0 / (1.0f + expf(-v0)) * v1, hi, lo);
                char *dst = static_cast<char *>(p.h) + frag_off(ug, node, C);
                *reinterpret_cast<__nv_bfloat16 *>(dst) = hi;
                *reinterpret_cast<__nv_bfloat16 *>(dst + 64) = lo;
            } else if (head) {
                if (!has) continue;
                float *y = p.logits + (size_t)node * p.V + 2 * ug;
                y[0] = v0;
                if (2 * ug + 1 < p.V) y[1] = v1;
            } else {
                float2 x = make_float2(0.f, 0.f);
                if (has) {
                    float2 *xs = reinterpret_cast<float2 *>(&e.ctl.x[node][2 * unit]);
                    x = *xs;
                    x.x += v0;
                    x.y += v1;
                    *xs = x;
                }
                const int first = kind == SG_DOWN && layer + 1 == p.L ? p.head_first : 0;
                emit_resid(e, node, has, 2 * ug, x.x, x.y, gain2, first, 2 * (n - first), p.ssq + (kind == SG_O ? kStreamMaxNodes * gridDim.x : 0));
            }
        }
    }
    if (!head) arrive_grid(e, c);
    else meet(e, c);           // the scratch may be written again
}

// Merges partial attention rows: out = sum_s O_s 2^(m_s - M), l likewise, for four dims of one row; four rows' loads at a
// time are under way together.
template <typename Row>
__device__ __forceinline__ float4 merge_rows(int count, Row row, int dim, float &M, float &L)
{
    M = -INFINITY;
    L = 0.f;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < count; s0 += 4) {
        float4 v[4], ml[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int s = min(s0 + u, count - 1);
            ml[u] = row(s, kHdim);
            v[u] = row(s, dim);
        }
        float mx = M;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (s0 + u >= count) ml[u].x = -INFINITY;
            mx = fmaxf(mx, ml[u].x);
        }
        if (mx == -INFINITY) continue;                       // no key that these rows see
        const float old = exp2f(M - mx);
        M = mx;
        L *= old;
        a.x *= old; a.y *= old; a.z *= old; a.w *= old;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (ml[u].x == -INFINITY) continue;              // (its outputs were never written)
            const float w = exp2f(ml[u].x - M);
            L += ml[u].y * w;
            a.x += v[u].x * w; a.y += v[u].y * w; a.z += v[u].z * w; a.w += v[u].w * w;
        }
    }
    return a;
}

__device__ __forceinline__ void attention_phase(const Env &e, Consumer &c, int layer)
{
    const StreamPass &p = e.p;
    const AttnShare a = e.ctl.attn;
    const int n = e.n, d = p.d;
    if (!wait_ready(e, c)) return;
    if (a.any) {
        const int gi = e.lane >> 2, t = e.lane & 3;
        const float scale = 1.4426950408889634f * rsqrtf((float)kHdim);
        constexpr int kPrefixSlots = 8;
        const bool with_new = a.split == p.splits - 1;      // this CTA also takes the new nodes' keys
        // two warps to a tile, 16 keys each; the others take the next ones
        const int group = e.warp >> 1, half = e.warp & 1;
        const int node = gi;                                // this lane's row
        const float *q0 = p.qkv + (size_t)a.head * kHdim;
        auto scratch = [&](int slot, int nd) { return e.red + (slot * n + nd) * kPRow; };

        // ---- the new nodes' own keys and values, in fp32: a warp takes a node at a time. Scores: four lanes per key;
        // outputs: four dims per lane. All rows are requested before the first is used.
        if (with_new) {
            const float *k0 = q0 + (size_t)kStreamMaxNodes * d, *v0 = k0 + (size_t)kStreamMaxNodes * d;
            const int nd = kWarps - 1 - e.warp;
            if (nd < n) {
                float4 q[8], v[kStreamMaxNodes], acc = make_float4(0.f, 0.f, 0.f, 0.f);
                const int key = e.lane >> 2, qd = (e.lane & 3) * 4, tn = p.n_old + key;
#pragma unroll
                for (int i = 0; i < 8; ++i) q[i] = __ldcg(reinterpret_cast<const float4 *>(q0 + (size_t)nd * d + 16 * i + qd));
#pragma unroll
                for (int j = 0; j < kStreamMaxNodes; ++j) v[j] = j <= nd ? __ldcg(reinterpret_cast<const float4 *>(v0 + (size_t)j * d + 4 * e.lane)) : make_float4(0.f, 0.f, 0.f, 0.f);
                float dot = 0.f;
                if (key <= nd) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float4 kv = __ldcg(reinterpret_cast<const float4 *>(k0 + (size_t)key * d + 16 * i + qd));
                        dot = fmaf(q[i].x, kv.x, fmaf(q[i].y, kv.y, fmaf(q[i].z, kv.z, fmaf(q[i].w, kv.w, dot))));
                    }
                }
                dot += __shfl_xor_sync(0xffffffffu, dot, 1);
                dot += __shfl_xor_sync(0xffffffffu, dot, 2);
                const bool vis = key <= nd && ((e.ctl.table.anc[p.n_old + nd][tn >> 5] >> (tn & 31)) & 1u);
                const float sc = vis ? dot * scale : -INFINITY;
                float mx = sc;
                for (int o = 16; o > 2; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                const float pr = exp2f(sc - mx);           // (the node sees itself: mx is no -inf)
                float sum = pr;
                for (int o = 16; o > 2; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
#pragma unroll
                for (int j = 0; j < kStreamMaxNodes; ++j) {
                    const float wj = __shfl_sync(0xffffffffu, pr, j * 4);
                    if (wj == 0.f) continue;               // a row that is not seen has no say, whatever it holds
                    acc.x = fmaf(wj, v[j].x, acc.x); acc.y = fmaf(wj, v[j].y, acc.y); acc.z = fmaf(wj, v[j].z, acc.z); acc.w = fmaf(wj, v[j].w, acc.w);
                }
                float *row = scratch(kPrefixSlots, nd);
                *reinterpret_cast<float4 *>(row + 4 * e.lane) = acc;
                if (e.lane == 0) { row[kHdim] = mx; row[kHdim + 1] = sum; }
            }
        }
        // ---- prefix (and earlier tree nodes). Loops stay loops here: this runs once per layer, and what straight-line code
        // costs is its fetch.
        if (a.t1 > a.t0) {
            // queries as hi and lo planes; every warp writes them all (the same values), and waits for none
            uint8_t *qs = reinterpret_cast<uint8_t *>(e.red) + p.q_off;
            for (int nd = 0; nd < n; ++nd) {
                const float4 v = __ldcg(reinterpret_cast<const float4 *>(q0 + (size_t)nd * d + 4 * e.lane));
                uint2 hi, lo;
                split2(v.x, v.y, hi.x, lo.x);
                split2(v.z, v.w, hi.y, lo.y);
                *reinterpret_cast<uint2 *>(qs + nd * kQRow + 8 * e.lane) = hi;
                *reinterpret_cast<uint2 *>(qs + (8 + nd) * kQRow + 8 * e.lane) = lo;
            }
            __syncwarp();
            const uint32_t qa = smem_u32(qs) + gi * kQRow + 4 * t;      // (rows of nodes that do not exist: any values)
            float m = -INFINITY, l = 0.f;
            const int keys = p.P + p.n_old;
            float *row = scratch(e.warp, min(node, n - 1));
            bool any = false;
            for (int tile = a.t0; tile < a.t1; ++tile, c.at.add(1, p.slots)) {
                c.ok = wait_all(smem_u32(&e.ctl.full[c.at.slot]), c.at.turn, e.ctl, p.wait_limit_ns);
                if (!c.ok) return;
                if (((tile - a.t0) & 3) == group) {
                    const uint32_t kb = e.ring + c.at.slot * p.slot_bytes, vb = kb + kKvItem / 2;
                    auto swz = [&](int key, int chunk) { return (uint32_t)((chunk >> 3) * (kKvItem / 4) + key * 128 + (((chunk ^ key) & 7) << 4)); };
                    float sc[2][4];
#pragma unroll
                    for (int j = 0; j < 2; ++j) sc[j][0] = sc[j][1] = sc[j][2] = sc[j][3] = 0.f;
#pragma unroll 2
                    for (int ks = 0; ks < 8; ++ks) {
                        uint32_t b[4];
                        ldsm4(kb + swz(half * 16 + (e.lane & 7) + ((e.lane >> 4) << 3), ks * 2 + ((e.lane >> 3) & 1)), b);
                        const uint32_t a0 = lds32(qa + ks * 32), a1 = lds32(qa + 8 * kQRow + ks * 32), a2 = lds32(qa + ks * 32 + 16),
                                       a3 = lds32(qa + 8 * kQRow + ks * 32 + 16);
                        mma_bf16(sc[0], a0, a1, a2, a3, b[0], b[1]);
                        mma_bf16(sc[1], a0, a1, a2, a3, b[2], b[3]);
                    }
                    float s4[4], mx = -INFINITY;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        s4[j] = (sc[j >> 1][j & 1] + sc[j >> 1][2 + (j & 1)]) * scale;
                        const int key = tile * kKeys + half * 16 + (j >> 1) * 8 + 2 * t + (j & 1);
                        if (key >= p.P) {
                            const int tn = key - p.P;
                            if (key >= keys || node >= n || !((e.ctl.table.anc[p.n_old + node][tn >> 5] >> (tn & 31)) & 1u)) s4[j] = -INFINITY;
                        }
                        mx = fmaxf(mx, s4[j]);
                    }
                    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                    const float mn = fmaxf(m, mx), ref = mn == -INFINITY ? 0.f : mn;
                    const float alpha = exp2f(m - ref);
                    m = mn;
                    float sum = 0.f;
#pragma unroll
                    for (int j = 0; j < 4; ++j) { s4[j] = exp2f(s4[j] - ref); sum += s4[j]; }
                    l = l * alpha + sum;
                    uint32_t pa[4];
                    split2(s4[0], s4[1], pa[0], pa[1]);
                    split2(s4[2], s4[3], pa[2], pa[3]);
#pragma unroll 2
                    for (int dp = 0; dp < 8; ++dp) {
                        uint32_t b[4];
                        float o[2][4];
#pragma unroll
                        for (int j = 0; j < 2; ++j) o[j][0] = o[j][1] = o[j][2] = o[j][3] = 0.f;
                        ldsm4_t(vb + swz(half * 16 + (e.lane & 7) + (((e.lane >> 3) & 1) << 3), dp * 2 + (e.lane >> 4)), b);
                        mma_bf16(o[0], pa[0], pa[1], pa[2], pa[3], b[0], b[1]);
                        mma_bf16(o[1], pa[0], pa[1], pa[2], pa[3], b[2], b[3]);
                        if (node < n) {
#pragma unroll
                            for (int j = 0; j < 2; ++j) {
                                float2 *at = reinterpret_cast<float2 *>(row + (2 * dp + j) * 8 + 2 * t);
                                float2 v = make_float2(o[j][0] + o[j][2], o[j][1] + o[j][3]);
                                if (any) {
                                    const float2 old = *at;
                                    v.x += old.x * alpha;
                                    v.y += old.y * alpha;
                                }
                                *at = v;
                            }
                        }
                    }
                    any = true;
                }
                __syncwarp();
                if (e.lane == 0) mbar_arrive(smem_u32(&e.ctl.empty[c.at.slot]));
            }
            l += __shfl_xor_sync(0xffffffffu, l, 1);
            l += __shfl_xor_sync(0xffffffffu, l, 2);
            if (node < n && t == 0) { row[kHdim] = m; row[kHdim + 1] = l; }
        } else if (node < n && t == 0) {
            scratch(e.warp, node)[kHdim] = -INFINITY;
        }
        if (!meet(e, c)) return;
        const int slots = kPrefixSlots + (with_new ? 1 : 0);
        auto write_out = [&](int nd, int dim, float4 v, float L) {
            const float inv = 1.0f / L;
            uint32_t h0, l0, h1, l1;
            split2(v.x * inv, v.y * inv, h0, l0);
            split2(v.z * inv, v.w * inv, h1, l1);
            char *dst = static_cast<char *>(p.att) + frag_off(a.head * kHdim + dim, nd, 2 * n);
            *reinterpret_cast<uint2 *>(dst) = make_uint2(h0, h1);
            *reinterpret_cast<uint2 *>(dst + 64) = make_uint2(l0, l1);
        };
        float *part = p.part + (size_t)a.head * p.splits * n * kStreamPartRow;
        for (int i = threadIdx.x; i < n * (kHdim / 4); i += 32 * kWarps) {
            const int nd = i / (kHdim / 4), dim = (i % (kHdim / 4)) * 4;
            float M, L;
            const float4 v = merge_rows(slots, [&](int s, int at) { return *reinterpret_cast<const float4 *>(scratch(s, nd) + at); }, dim, M, L);
            if (p.splits == 1) { write_out(nd, dim, v, L); continue; }
            float *row = part + (a.split * n + nd) * kStreamPartRow;
            *reinterpret_cast<float4 *>(row + dim) = v;
            if (dim == 0) *reinterpret_cast<float2 *>(row + kHdim) = make_float2(M, L);
        }
        if (p.splits > 1) {
            if (!meet(e, c)) return;
            if (threadIdx.x == 0) {
                uint32_t before;
                asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(before) : "l"(p.bar + 2 + a.head) : "memory");
                e.ctl.last = before + 1 == (uint32_t)(p.splits * (layer + 1));
            }
            if (!meet(e, c)) return;
            if (e.ctl.last)
                for (int i = threadIdx.x; i < n * (kHdim / 4); i += 32 * kWarps) {
                    const int nd = i / (kHdim / 4), dim = (i % (kHdim / 4)) * 4;
                    float M, L;
                    const float4 v = merge_rows(p.splits, [&](int s, int at) { return __ldcg(reinterpret_cast<const float4 *>(part + (s * n + nd) * kStreamPartRow + at)); }, dim, M, L);
                    write_out(nd, dim, v, L);
                }
        }
    }
    arrive_grid(e, c);
}

template <bool W4>
__device__ __forceinline__ void consume(const Env &e, Consumer &c)
{
    const StreamPass &p = e.p;
    const int n = e.n;
    // ---- start: rotary factors of this CTA's Q and K rows, embedding rows of its part of the residual stream
    {
        const Share s = e.ctl.share[SG_QKV];
        for (int i = threadIdx.x; i < n * s.U; i += 32 * kWarps) {
            const int node = i / s.U, r = 2 * (s.u0 + i - node * s.U);
            if (r >= 2 * p.d) continue;
            double sn, cs;
            sincos((double)(p.P + mask_depth(e.ctl.table.anc[p.n_old + node])) * p.inv_freq[(r & 127) >> 1], &sn, &cs);
            e.cs[i] = make_float2((float)cs, (float)sn);
        }
        const Share x = e.ctl.share[SG_O];
        const bool has = e.lane < x.U;
        const int u = x.u0 + e.lane;
        const uint32_t gain2 = has ? __ldg(reinterpret_cast<const uint32_t *>(p.base + p.attn_norm) + u) : 0;
        for (int node = e.warp; node < n; node += kWarps) {
            uint32_t v = 0;
            if (has) v = __ldg(reinterpret_cast<const uint32_t *>(p.base + p.tok_embed) + (size_t)__ldg(p.tokens + p.n_old + node) * (p.d / 2) + u);
            const float v0 = __uint_as_float(v << 16), v1 = __uint_as_float(v & 0xffff0000u);
            if (has) *reinterpret_cast<float2 *>(&e.ctl.x[node][2 * e.lane]) = make_float2(v0, v1);
            emit_resid(e, node, has, 2 * u, v0, v1, gain2, 0, 2 * n, p.ssq);
        }
        arrive_grid(e, c);
    }
    for (int l = 0; l <= p.L && c.ok; ++l) {
        const int steps = l < p.L ? 5 : p.logits != nullptr ? p.head_parts : 0;
        for (int st = 0; st < steps && c.ok; ++st) {
            if (l < p.L && st == 1) attention_phase(e, c, l);
            else gemm_phase<W4>(e, c, l < p.L ? gemm_kind(st) : SG_HEAD, l, l < p.L ? 0 : st);
        }
    }
}

// One thread: polls the grid barrier, tells the CTA that the next phase may start, and fetches its input. False when a
// wait ran out.
__device__ __forceinline__ bool load_inputs(const StreamPass &p, Ctl &ctl, uint32_t x_ring)
{
    uint32_t target = 0, xs = 0;
    const int phases = 5 * p.L + (p.logits != nullptr ? p.head_parts : 0);
    for (int ph = 0, step = 0; ph < phases; ++ph) {
        const bool head = ph >= 5 * p.L;
        const int kind = head ? SG_HEAD : gemm_kind(step);
        const int n_kb = (!head && step == 1) || ctl.share[head ? SG_HEAD + ph - 5 * p.L : kind].U == 0 ? 0 : p.g[kind].kb_all, n_k32 = p.g[kind].K / 32;
        const int k32_bytes = 2 * (p.n_tree - p.n_old - (head ? p.head_first : 0)) * 64, x_kb = p.x_stage_bytes / (2 * k32_bytes);
        const char *src = static_cast<const char *>(kind == SG_O ? p.att : kind == SG_DOWN ? p.h : p.xn);
        if (++step == 5) step = 0;
        // Polls only once this CTA has arrived itself: every poll takes L1 along.
        const bool first = ph <= 5 * p.L;                     // the parts of the lm_head have the same input
        if (first && !thread_wait(smem_u32(&ctl.gone), ph & 1u, ctl, p.wait_limit_ns)) return false;
        target += first ? gridDim.x : 0;
        uint64_t t0 = 0;
        for (uint32_t it = 1; first && ld_acquire_gpu_u32(p.bar) < target; ++it) {
            if ((it & 63u) == 0) {
                const uint64_t now = global_timer_ns();
                if (t0 == 0) t0 = now;
                else if (ctl.abort_flag || now - t0 > p.wait_limit_ns) return false;
            }
        }
        if (first) mbar_arrive(smem_u32(&ctl.ready));
        asm volatile("fence.proxy.async;" ::: "memory");      // the input was written by ordinary stores
        for (int kb = 0; kb < n_kb; kb += x_kb, ++xs) {
            const int st = xs % kXStages;
            if (!thread_wait(smem_u32(&ctl.xempty[st]), ((xs / kXStages) & 1u) ^ 1u, ctl, p.wait_limit_ns)) return false;
            if (p.withhold_input) continue;
            const uint32_t full = smem_u32(&ctl.xfull[st]), bytes = (min(2 * (kb + x_kb), n_k32) - 2 * kb) * k32_bytes;
            mbar_expect_tx(full, bytes);
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(x_ring + st * p.x_stage_bytes), "l"(src + (size_t)(2 * kb) * k32_bytes), "r"(bytes), "r"(full)
                         : "memory");
        }
    }
    return true;
}

template <bool W4>
__global__ void __launch_bounds__(kThreads<W4>, 1)
stream_pass_kernel(const __grid_constant__ StreamPass p, const __grid_constant__ CUtensorMap kv_map)
{
    extern __shared__ uint8_t sm_raw[];
    __shared__ Ctl ctl;
    const uint32_t raw = smem_u32(sm_raw), base = (raw + 1023u) & ~1023u;     // swizzled tiles want 1024-byte alignment
    uint8_t *smp = sm_raw + (base - raw);
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    Producer<W4> prod(p, &kv_map, ctl, base);
    if (warp == kWarps) {
        if (lane < SG_HEAD + p.head_parts) ctl.share[lane] = lane < SG_HEAD ? share_of(p.g[lane]) : part_of(share_of(p.g[SG_HEAD]), lane - SG_HEAD, p.head_parts);
        if (lane == 31) ctl.attn = attn_share(p);
        if (lane == 0) {
            for (int s = 0; s < kMaxSlots; ++s) {
                mbar_init(smem_u32(&ctl.full[s]), W4 ? 32 : 1);
                mbar_init(smem_u32(&ctl.empty[s]), kWarps);
            }
            for (int s = 0; s < kXStages; ++s) {
                mbar_init(smem_u32(&ctl.xfull[s]), 1);
                mbar_init(smem_u32(&ctl.xempty[s]), kWarps);
            }
            mbar_init(smem_u32(&ctl.ready), 1);
            mbar_init(smem_u32(&ctl.meet), kWarps);
            mbar_init(smem_u32(&ctl.gone), 1);
            ctl.abort_flag = 0;
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async;" ::: "memory");
        }
    }
    __syncthreads();
    const bool producer = warp >= kWarps && warp < kWarps + kProducers<W4>;
    if (producer) {
        prod.start();
        while (!prod.done() && prod.free_now()) prod.fetch();
    }
    // every CTA checks the tree itself, and all agree
    const int err = mask_table(ctl.table, p.parent, p.tokens, p.n_tree, p.V);
    int stands = 0;
    if (p.keep_status) {
        stands = *reinterpret_cast<volatile int32_t *>(p.status);     // written by an earlier launch
        if (err && blockIdx.x == 0 && threadIdx.x == 0) atomicCAS(p.status, 0, err);
    } else if (blockIdx.x == 0 && threadIdx.x == 0) *p.status = err;
    __syncthreads();
    bool ok = true;
    if (err || stands) {
        // nothing to do but to let the weights land: the first turn of this producer's slots
        if (producer)
            for (int i = 0; i < prod.issued && ok; ++i) ok = wait_all(smem_u32(&ctl.full[warp - kWarps + i * prod.step]), 0, ctl, p.wait_limit_ns);
    } else if (warp < kWarps) {
        Env e{p, ctl, base, reinterpret_cast<float *>(smp + p.red_off), reinterpret_cast<float2 *>(smp + p.cs_off), p.n_tree - p.n_old, warp, lane};
        Consumer c;
        consume<W4>(e, c);
        ok = c.ok;
    } else if (producer) {
        while (!prod.done()) {
            ok = prod.wait_free();
            if (!ok) break;
            prod.fetch();
        }
    } else if (lane == 0) {
        ok = load_inputs(p, ctl, base + (uint32_t)p.x_off);
    }
    __syncwarp();
    if (W4) asm volatile("cp.async.wait_all;" ::: "memory");
    if (!ok) {
        ctl.abort_flag = 1;
        atomicCAS(p.status, 0, LLMCAD_ERR_TIMEOUT);
        // give copies that may still be in flight time to land before the shared memory goes away
        const uint64_t t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 2000000ull) __nanosleep(1000);
    }
    // the last CTA to leave puts the barrier words back to zero for the next launch
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(p.bar + 1, 1u) == gridDim.x - 1) {
            p.bar[0] = 0;
            p.bar[1] = 0;
            for (int h = 0; h < p.H; ++h) p.bar[2 + h] = 0;
        }
    }
}

}  // namespace

bool stream_pass_serves(int d, int f, int hd, int H, int V, int n_sms)
{
    // a CTA's rows of the residual stream are one unit per lane, K is whole halves of a k-block, and a phase has 16 tiles of 16
    // rows at most: kMt of them per warp once the warps share the rows
    auto per_cta = [&](long long units) { return (units + n_sms - 1) / n_sms; };
    return hd == kHdim && n_sms <= kMaxSms && H <= n_sms && d % 128 == 0 && f % 32 == 0 && per_cta(d / 2) <= kMaxResidUnits &&
           per_cta(3 * d / 2) <= 128 && per_cta(f) <= 128 && per_cta(((long long)V + 1) / 2) <= 128;
}

// Up to four nodes, (node, plane) is one tile of eight columns and a warp's loads of weights feed one MMA each; a variant with
// two tiles, for eight nodes, lost. Whole passes, us, this kernel against one kernel per step: 7B shape (32 layers, prefix
// 512) 2511 / 2811 with one node, 2620 / 2827 with four, 3241 / 2844 with eight; 13B widths (20 layers, prefix 1024) 2400 / 2516,
// 2423 / 2524, 2842 / 2535.
bool stream_pass_prefers(int n)
{
    static const int max_n = [] { const char *e = getenv("LLMCAD_STREAM_PASS_MAX_N"); return e ? atoi(e) : 4; }();   // tuning aid; 0: never
    return n <= kStreamMaxNodes && n <= max_n;
}

size_t stream_pass_floats_qkv(int d) { return (size_t)3 * kStreamMaxNodes * d; }
size_t stream_pass_floats_part(int n_sms) { return (size_t)n_sms * kStreamMaxNodes * kStreamPartRow; }

namespace {
constexpr size_t kib(size_t b) { return (b + 1023) / 1024 * 1024; }
constexpr size_t kStreamSmem = 227 * 1024 - 1024 - kib(sizeof(Ctl));      // 1024: alignment of the ring
}  // namespace

bool plan_stream_pass(StreamPass &p, int n_sms)
{
    const int n = p.n_tree - p.n_old;
    const int tiles = (p.P + p.n_old + kKeys - 1) / kKeys;
    // Key ranges of a head: as many as there are CTAs for, but no fewer than four tiles each, which a CTA's four pairs of warps
    // take side by side. The last CTA of a head merges its ranges one after the other: with a tile each (us a pass of 4
    // layers and 4 nodes, a tile / four tiles at least / one kernel per step) 1 head and 4096 keys take 214 / 135 / 155, 2 heads
    // and 2048 161 / 125 / 144, 4 heads and 512 127 / 123 / 148, 32 heads and 64 367 / 361 / 392. With eight at least, 512 keys
    // are 3 % slower.
    const int ranges = tiles > 4 ? (tiles + 3) / 4 : 1;
    p.splits = n_sms / p.H < ranges ? n_sms / p.H : ranges;
    const int units[SG_KINDS] = {3 * p.d / 2, p.d / 2, p.f, p.d / 2, (p.V + 1) / 2};
    const int K[SG_KINDS] = {p.d, p.d, p.d, p.f, p.d};
    size_t red = 0;
    // two stages of inputs, 32 k-blocks of one node each, or 16 of four nodes
    p.x_stage_bytes = n == 1 ? 8192 : 16384;
    int U[SG_KINDS], kbs[SG_KINDS];
    for (int i = 0; i < SG_KINDS; ++i) {
        U[i] = (units[i] + n_sms - 1) / n_sms;
        kbs[i] = (K[i] + 63) / 64;
    }
    // a part of the lm_head is no larger than the largest share of a layer's GEMMs
    int most = 64;
    for (int i = 0; i < SG_HEAD; ++i) most = U[i] > most ? U[i] : most;
    p.head_parts = (U[SG_HEAD] + most - 1) / most;
    if (p.head_parts > kStreamHeadParts) return false;
    U[SG_HEAD] = (U[SG_HEAD] + p.head_parts - 1) / p.head_parts;
    for (int i = 0; i < SG_KINDS; ++i) {
        StreamGemm &g = p.g[i];
        g.units = units[i];
        g.K = K[i];
        g.kb_all = kbs[i];
        const int mt = (U[i] + 7) / 8;
        auto scratch = [&]() { return (size_t)(kWarps / g.mg) * n * ((U[i] + 15) / 16 * 16 + 4) * 8; };
        // as few warps to a k-block as the accumulators and the reduction scratch allow
        for (g.mg = 1; g.mg < kWarps; g.mg *= 2)
            if ((mt + g.mg - 1) / g.mg <= kMt && scratch() <= 24 * 1024) break;
        g.kg = kWarps / g.mg;
        red = scratch() > red ? scratch() : red;
        g.x_kb = p.x_stage_bytes / (2 * (i == SG_HEAD ? n - p.head_first : n) * 128);
    }
    p.q_off = 9 * n * kPRow * (int)sizeof(float);
    const size_t att = (size_t)p.q_off + 16 * kQRow;
    red = kib(att > red ? att : red);
    const size_t cs = kib((size_t)n * ((units[SG_QKV] + n_sms - 1) / n_sms) * sizeof(float2));
    // The ring: slots of one size, the one that leaves most weights in flight on average over a layer's GEMMs. An item has
    // as many k-blocks as fit (and as there are lanes for, a copy each).
    const int ring = (int)((kStreamSmem - red - cs) / 1024 * 1024) - kXStages * p.x_stage_bytes;
    auto item_kb = [&](int i, int slot, bool codes) {
        const bool two = p.g[i].upper != 0;
        const int rows_run = (two ? 1 : 2) * U[i], runs = (two ? 2 : 1) * (((rows_run + 126) >> 7) + 1);
        int kb = slot / (codes ? w4_kb_bytes(15, rows_run, two ? 2 : 1) : U[i] * 256);
        for (int most_kb : {codes ? kMaxItemKbW4 : 32 / runs, codes ? kMaxItemKbW4 : kMaxItemKb, kbs[i]}) kb = kb < most_kb ? kb : most_kb;
        return kb;
    };
    double best = 0;
    for (int slot = kKvItem; slot <= 32 * 1024; slot += 1024) {
        int slots = ring / slot;
        if (slots > kMaxSlots) slots = kMaxSlots;
        double time = 0, bytes = 0;
        for (int i = 0; i < SG_HEAD; ++i) {
            // (also with INT4 weights a slot has room for a k-block in bf16: both take the same models)
            const int kb = item_kb(i, slot, false) == 0 ? 0 : item_kb(i, slot, p.w4 != 0);
            if (kb == 0) { time = 1e30; break; }
            const double all = (double)units[i] * kbs[i];
            bytes += all;
            time += all / ((double)slots * kb * U[i]);
        }
        if (item_kb(SG_HEAD, slot, false) == 0 || bytes / time <= best) continue;
        best = bytes / time;
        p.slot_bytes = slot;
        p.slots = slots;
    }
    if (best == 0 || p.slots < kProducers<false>) return false;
    for (int i = 0; i < SG_KINDS; ++i) {
        StreamGemm &g = p.g[i];
        g.kb_item = item_kb(i, p.slot_bytes, p.w4 && i != SG_HEAD);
        g.n_items = (g.kb_all + g.kb_item - 1) / g.kb_item;
    }
    p.x_off = ring;
    p.red_off = p.x_off + kXStages * p.x_stage_bytes;
    p.cs_off = p.red_off + (int)red;

    return true;
}

cudaError_t launch_stream_pass(const StreamPass &p, int n_sms, cudaStream_t st)
{
    CUtensorMap map;
    const uint64_t keys = (uint64_t)(p.P + p.n_old > 0 ? p.P + p.n_old : 1);
    const uint64_t dims[3] = {kHdim, keys, (uint64_t)p.L * 2 * p.H}, strides[2] = {kHdim * 2, (uint64_t)p.S * kHdim * 2};
    const uint32_t box[3] = {64, kKeys, 1};
    // rows behind the prefix read as zero
    if (!make_tensor_map_bf16_3d(&map, p.kv, dims, strides, box)) return cudaErrorInvalidValue;

    static PerDeviceOnce attr_set;
    if (attr_set.needed()) {
        for (auto k : {stream_pass_kernel<false>, stream_pass_kernel<true>}) {
            const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStreamSmem + 1024);
            if (e != cudaSuccess) return e;
        }
        attr_set.mark();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_sms);
    cfg.blockDim = dim3(p.w4 ? kThreads<true> : kThreads<false>);
    cfg.dynamicSmemBytes = kStreamSmem + 1024;
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, p.w4 ? stream_pass_kernel<true> : stream_pass_kernel<false>, p, map);
}

}  // namespace llmcad
