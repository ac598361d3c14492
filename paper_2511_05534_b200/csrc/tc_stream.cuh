// Skeleton shared by four tensor-core kernels (window scoring pass 1 and 2, matching, full-prefill flow).
//
// Each CTA is persistent (one per SM) and walks a list of items.  An item is up to two 128-row
// operand halves A_0, A_1 (loaded once per item) against a stream of operand tiles B_0 .. B_{n-1}
// of up to NB rows; every B tile is used by both halves, which halves the operand traffic per
// multiply-add, and yields one 128 x NB fp32 accumulator per half in TMEM (half h owns TMEM
// columns [NB h, NB h + NB)).
// Roles: warp 0 issues the TMA loads (the matching kernel has two more warps that gather its A halves), warp 1 issues tcgen05.mma, warps 2-17 run the kernel's
// epilogue: a quad of warps (one per 32 TMEM lanes) per (A half, column half), i.e. four epilogue
// warps per SM sub-partition, so that TMEM reads, shared-memory reads and dependent arithmetic of
// one warp are covered by the other three.  The two quads of a half split each accumulator's
// columns in two and combine per-row results through shared memory.
// Shared-memory stages (AST per A half, two for B) and the two accumulators are handed around
// with mbarriers; every wait is bounded.
//
// Accumulators are handed around in one of three ways, the kernel's choice (acc_arrivals of setup()):
//   8   by half, the two quads of the half together (matching: products 256 columns wide);
//   16  by half, all sixteen warps drain one half at a time while the other is refilled (row statistics);
//   4   by quad: the two column halves are refilled one by one, each as soon as its quad has released it, so that a quad
//       waits for 128 columns only and the four warps of a scheduler are in different phases of their work.  Second
//       scoring pass: 112 heads of 8448 tokens 181 -> 171 us, full-prefill flow of 2176 tokens 680 -> 657 us, of 512 66 -> 57;
//       the matching kernel was 8 % slower, the row statistics 2 %.
// Three shapes are instantiated: Skel<256, 1, 2> for long B streams (one A stage per half, two 64 KB B
// stages), and for problems whose items have few B columns, where the A operand is the stream, Skel<128, 2, 2>
// and Skel<256, 2, 1>: two A stages per half let the next item's rows load while this item is computed, and an item
// whose B tiles are the previous item's and still in their stages (TilePlan::reuse_b) takes them as they stand.
#pragma once
#include "common.cuh"
#include "tc_common.cuh"

namespace flowmm {
namespace tcs {

constexpr int kRows = 128;                   // rows of an A half (UMMA M)
constexpr int kItemRows = 2 * kRows;         // rows of A an item covers
constexpr int kEpiWarps = 16;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr uint32_t kAHalf = kRows * 128 * 2; // bytes of an A half: two 64-element K halves
constexpr int kExtraSlots = 4;               // ring of per-column constants: a slot is rewritten four B tiles later
constexpr uint32_t kEpiBytes = 16384;
constexpr int kStatusAlign = 6;              // FLOWMM_ERR_ALIGN

// Meeting of the CTA's threads that use named barrier `id`, `count` of them in whole warps; with a vote: whether any of them says yes.
__device__ __forceinline__ void named_barrier(int id, int count) { asm volatile("barrier.cta.sync %0, %1;" ::"r"(id), "r"(count) : "memory"); }
__device__ __forceinline__ bool meet_vote(int id, int count, bool yes) {
    uint32_t any;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "barrier.cta.red.or.pred p, %2, %3, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(any)
        : "r"((uint32_t)yes), "r"(id), "r"(count)
        : "memory");
    return any != 0;
}

// Where an item's operands come from.  All tensor maps are 4-D: (K element, c1, c2, c3).
struct TilePlan {
    int a1, a2, a3;            // box origin of A half 0
    int h1, h2;                // origin advance of half 1 along c1 / c2
    int n_halves;              // 0: nothing to compute, every role skips the item
    int b1, b2, b3;            // B box origin of tile 0
    int step1, step2;          // B origin advance per tile along c1 / c2
    int n_tiles;               // 0: every role skips the item
    int cols_total;            // valid B rows over all tiles (tile t has min(NB, cols_total - NB t))
    int cols_first = 0;        // ... for A half 0, where it needs fewer in the last tile (0: the same)
    bool reuse_b = false;      // the item's B tiles (and their constants), at most as many as there are stages, are those of the item before
    bool keep_b = false;       // ... and the next item's as well: their stages are not handed back after this item
    const float *extra;        // nullptr, or NB fp32 per-column constants per tile: tile t reads extra + NB t
    __device__ __forceinline__ bool empty() const { return n_tiles == 0 || n_halves == 0; }
};

template <int NB, int AST, int BST>
struct Skel {
    static constexpr int kCols = NB;                         // rows of a B tile (UMMA N)
    static constexpr int kBStages = BST;
    static constexpr uint32_t kBStage = NB * 128 * 2;
    static constexpr uint32_t kExtraBytes = NB * 4;          // per-column fp32 constants that travel with a B tile
    static constexpr uint32_t kSmemA = 0;                    // [stage][half]
    static constexpr uint32_t kSmemB = 2 * AST * kAHalf;
    static constexpr uint32_t kSmemExtra = kSmemB + BST * kBStage;
    static constexpr uint32_t kSmemEpi = kSmemExtra + kExtraSlots * kExtraBytes;   // epilogue scratch
    static constexpr uint32_t kSmemBar = kSmemEpi + kEpiBytes;
    static constexpr uint32_t kSmemBytes = kSmemBar + 256;
    // barrier slots
    static constexpr int kBarAFull = 0, kBarAEmpty = 2 * AST, kBarBFull = 4 * AST, kBarBEmpty = kBarBFull + BST,
                         kBarAccFull = kBarBEmpty + BST, kBarAccEmpty = kBarAccFull + 4, kBarXFull = kBarAccEmpty + 4,
                         kNumBars = kBarXFull + kExtraSlots;
    static_assert(8 * kNumBars + 8 <= 256, "barrier block too small");
    static_assert(kSmemBytes <= 232448, "shared memory budget");

    struct Ctx {
        uint32_t base, bars, tmem_base;
        volatile int *abort_flag;
        int warp, lane;
        int group, quarter;        // epilogue warps: which A half they serve, which 32 TMEM lanes they read
        int colhalf;               // ... and which half of each accumulator's columns
        bool ok;                   // false: shared memory was not 1024-byte aligned; nothing may run
        __device__ __forceinline__ uint32_t bar(int i) const { return bars + 8u * i; }
        // shared address of the per-column constants of the bt-th B tile this CTA streams.  Valid from the tile's acc_extra_wait to
        // the release of the item's tile after it, or, for an item's last tile, to its own release: until then the half may sit out
        // an item, and what the issuer goes by is the last release.
        __device__ __forceinline__ uint32_t extra(int bt) const {
            return base + kSmemExtra + (uint32_t)(bt & (kExtraSlots - 1)) * kExtraBytes;
        }
        // shared addresses of the scratch of this warp's quad / of its partner quad on the same rows
        __device__ __forceinline__ uint32_t epi_addr() const { return base + kSmemEpi + (uint32_t)(group * 2 + colhalf) * (kEpiBytes / 4); }
        __device__ __forceinline__ uint32_t partner_addr() const {
            return base + kSmemEpi + (uint32_t)(group * 2 + (colhalf ^ 1)) * (kEpiBytes / 4);
        }
        // shared address of A half h (one A stage)
        __device__ __forceinline__ uint32_t a_addr_of(int h) const { return base + kSmemA + (uint32_t)h * kAHalf; }
        // shared address of A half `group` of the n-th item this group takes part in
        __device__ __forceinline__ uint32_t a_addr(int n) const {
            return base + kSmemA + (uint32_t)((n % AST) * 2 + group) * kAHalf;
        }
    };

    // `a_readers`: epilogue warps per half that read the A stage themselves and release it with a_release().
    static __device__ __forceinline__ Ctx setup(uint8_t *smem_raw, const CUtensorMap *ma, const CUtensorMap *mb,
                                                int *status, int a_readers = 0, int acc_arrivals = 8) {
        Ctx c;
        c.base = tc::smem_u32(smem_raw);
        c.bars = c.base + kSmemBar;
        c.warp = tc::warp_number();
        c.lane = threadIdx.x & 31;
        c.group = ((c.warp - 2) >> 2) & 1;
        c.quarter = c.warp & 3;
        c.colhalf = (c.warp - 2) >> 3;
        c.tmem_base = 0;
        c.abort_flag = reinterpret_cast<volatile int *>(smem_raw + kSmemBar + 8 * kNumBars + 4);
        c.ok = (c.base & 1023u) == 0;              // the swizzled operand tiles need a 1024-byte aligned base
        if (!c.ok) {
            predecessor_done();
            if (threadIdx.x == 0) atomicCAS(status, 0, kStatusAlign);
            return c;
        }
        uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem_raw + kSmemBar + 8 * kNumBars);
        if (threadIdx.x == 0) {
            for (int i = 0; i < kNumBars; ++i) {
                int count = 1;
                if (i >= kBarAEmpty && i < kBarBFull) count = 1 + a_readers;
                if (i >= kBarAccEmpty && i < kBarXFull) count = acc_arrivals;   // one arrival per epilogue warp that reads it
                tc::mbar_init(c.bar(i), count);
            }
            *c.abort_flag = 0;
            tc::mbar_init_fence();
            tc::tma_prefetch_desc(ma);
            tc::tma_prefetch_desc(mb);
        }
        if (c.warp == 1) tc::tmem_alloc(tc::smem_u32(tmem_slot), 512);
        tc::tc_fence_before();
        __syncthreads();
        tc::tc_fence_after();
        c.tmem_base = *tmem_slot;
        predecessor_done();
        return c;
    }

    static __device__ __forceinline__ void teardown(const Ctx &c) {
        if (!c.ok) return;
        tc::tc_fence_before();
        __syncthreads();
        tc::tc_fence_after();
        if (c.warp == 1) tc::tmem_dealloc(c.tmem_base, 512);
    }

    // Call from a whole warp.  a_bytes / b_bytes: bytes one A-half / B box pair delivers (both K halves).
    // kLoadsA: false where warps of the kernel's own bring the A halves (they wait for kBarAEmpty and arrive at kBarAFull).
    template <bool kLoadsA = true, class PlanFn>
    static __device__ __forceinline__ void producer(const Ctx &c, const CUtensorMap *ma, const CUtensorMap *mb, int n_items,
                                                    uint32_t a_bytes, uint32_t b_bytes, PlanFn plan, int *status) {
        int ia[2] = {0, 0}, bt = 0;
        bool ok = true;
        for (int item = blockIdx.x; ok && item < n_items; item += gridDim.x) {
            const TilePlan p = plan(item);
            if (p.empty()) continue;
            for (int t = 0; ok && t < p.n_tiles; ++t) {
                const int sb = bt % BST;
                if (!p.reuse_b) ok = tc::mbar_wait_warp(c.bar(kBarBEmpty + sb), ((bt / BST) & 1) ^ 1, c.abort_flag, status);
                if (!ok) break;
                // The slot's readers are through with tile bt - 4: the stage just waited for was handed back after the products of tile
                // bt - 2, which each half's wait for the release of its tile before, bt - 3 or older (mma_issuer).
                if (p.extra && !p.reuse_b) {
                    const int xs = bt & (kExtraSlots - 1);
                    if (tc::elect_one()) {
                        tc::mbar_expect_tx(c.bar(kBarXFull + xs), kExtraBytes);
                        tc::bulk_load(c.base + kSmemExtra + (uint32_t)xs * kExtraBytes, p.extra + (size_t)t * NB, kExtraBytes,
                                      c.bar(kBarXFull + xs));
                    }
                    __syncwarp();
                }
                if (!p.reuse_b) {
                    const uint32_t b_dst = c.base + kSmemB + sb * kBStage;
                    if (tc::elect_one()) {
                        tc::mbar_expect_tx(c.bar(kBarBFull + sb), b_bytes);
                        tc::tma_load_4d(b_dst, mb, c.bar(kBarBFull + sb), 0, p.b1 + t * p.step1, p.b2 + t * p.step2, p.b3);
                        tc::tma_load_4d(b_dst + kBStage / 2, mb, c.bar(kBarBFull + sb), 64, p.b1 + t * p.step1, p.b2 + t * p.step2, p.b3);
                    }
                    __syncwarp();
                    ++bt;
                }
                if (kLoadsA && t == 0) {       // the item's A halves go out right after its first B tile
                    for (int h = 0; ok && h < p.n_halves; ++h) {
                        const int st = ia[h] % AST, full = kBarAFull + st * 2 + h;
                        ok = tc::mbar_wait_warp(c.bar(kBarAEmpty + st * 2 + h), ((ia[h] / AST) & 1) ^ 1, c.abort_flag, status);
                        if (!ok) break;
                        const uint32_t a_dst = c.base + kSmemA + (uint32_t)(st * 2 + h) * kAHalf;
                        if (tc::elect_one()) {
                            tc::mbar_expect_tx(c.bar(full), a_bytes);
                            tc::tma_load_4d(a_dst, ma, c.bar(full), 0, p.a1 + h * p.h1, p.a2 + h * p.h2, p.a3);
                            tc::tma_load_4d(a_dst + kAHalf / 2, ma, c.bar(full), 64, p.a1 + h * p.h1, p.a2 + h * p.h2, p.a3);
                        }
                        __syncwarp();
                        ++ia[h];
                    }
                }
            }
        }
        if (!ok) {          // winding down after a timeout: give copies already issued a moment to land
            for (int i = 0; kLoadsA && i < 2 * AST; ++i)
                for (int s = 0; s < (1 << 16) && !tc::mbar_try_wait(c.bar(kBarAFull + i), 0) && !tc::mbar_try_wait(c.bar(kBarAFull + i), 1); ++s) {}
            for (int i = 0; i < BST; ++i)
                for (int s = 0; s < (1 << 16) && !tc::mbar_try_wait(c.bar(kBarBFull + i), 0) && !tc::mbar_try_wait(c.bar(kBarBFull + i), 1); ++s) {}
        }
    }

    // Call from a whole warp.  kQuads: accumulators are handed around by quad, else by half.
    template <bool kQuads, class PlanFn>
    static __device__ __forceinline__ void mma_issuer(const Ctx &c, int n_items, PlanFn plan, int *status) {
        constexpr int kParts = kQuads ? 2 : 1, kPartCols = NB / kParts;   // accumulators of a half, their columns
        int ia[2] = {0, 0}, ta[4] = {0, 0, 0, 0}, bt = 0;
        bool ok = true;
        for (int item = blockIdx.x; ok && item < n_items; item += gridDim.x) {
            const TilePlan p = plan(item);
            if (p.empty()) continue;
            if (p.reuse_b) bt -= p.n_tiles;                              // bt: number of the B tile
            for (int t = 0; ok && t < p.n_tiles; ++t, ++bt) {
                const int sb = bt % BST;
                ok = tc::mbar_wait_warp(c.bar(kBarBFull + sb), (bt / BST) & 1, c.abort_flag, status);
                if (!ok) break;
                const int ncols = min(NB, p.cols_total - t * NB);
                const int ncols0 = p.cols_first ? min(NB, p.cols_first - t * NB) : ncols;
                const uint32_t b_base = c.base + kSmemB + sb * kBStage;
                uint32_t took = 0;                                       // accumulators with a part in this tile
                for (int h = 0; ok && h < p.n_halves; ++h) {
                    const int st = ia[h] % AST;
                    if (t == 0) ok = tc::mbar_wait_warp(c.bar(kBarAFull + st * 2 + h), (ia[h] / AST) & 1, c.abort_flag, status);
                    const uint32_t a_base = c.base + kSmemA + (uint32_t)(st * 2 + h) * kAHalf;
#pragma unroll
                    for (int ch = 0; ch < kParts; ++ch) {                // the accumulators that hold columns
                        const int q = kParts * h + ch, n = min(kPartCols, (h == 0 ? ncols0 : ncols) - ch * kPartCols);
                        if (n <= 0 || !ok) continue;
                        ok = tc::mbar_wait_warp(c.bar(kBarAccEmpty + q), (ta[q] & 1) ^ 1, c.abort_flag, status);
                        if (!ok) continue;
                        tc::tc_fence_after();
                        const uint32_t idesc = tc::idesc_bf16(kRows, (uint32_t)((n + 15) & ~15));
                        const uint32_t a_lo = tc::desc_lo(a_base), b_lo = tc::desc_lo(b_base + ch * (kPartCols * 128)), d = c.tmem_base + q * kPartCols;
                        if (tc::elect_one()) {
#pragma unroll
                            for (int ks = 0; ks < 8; ++ks)               // head_dim 128 = 8 K slices of 16
                                tc::umma_bf16(d, a_lo + (ks >> 2) * (kAHalf / 32) + (ks & 3) * 2, tc::kDescSw128Hi,
                                              b_lo + (ks >> 2) * (kBStage / 32) + (ks & 3) * 2, tc::kDescSw128Hi, idesc, ks > 0);
                            tc::umma_commit(c.bar(kBarAccFull + q));     // accumulator ready
                        }
                        __syncwarp();
                        ++ta[q];
                        took |= 1u << q;
                    }
                    if (!ok) break;
                    if (t == p.n_tiles - 1) {                            // that was the half's last use of its A stage
                        if (tc::elect_one()) tc::umma_commit(c.bar(kBarAEmpty + st * 2 + h));
                        __syncwarp();
                        ++ia[h];
                    }
                }
                if (!ok) break;
                if (p.extra) {
                    // accumulators without a part in this tile: their warps must be through with the tiles before it as well,
                    // so that the stage's release tells the producer that nobody reads the constants of those tiles any more
                    for (int q = 0; ok && q < 2 * kParts; ++q)
                        if (!(took & (1u << q))) ok = tc::mbar_wait_warp(c.bar(kBarAccEmpty + q), (ta[q] & 1) ^ 1, c.abort_flag, status);
                    if (!ok) break;
                }
                if (!p.keep_b && tc::elect_one()) tc::umma_commit(c.bar(kBarBEmpty + sb));   // B stage free once both halves' MMAs finish
                __syncwarp();
            }
        }
    }

    // Epilogue side.  `k` counts the accumulator tiles this warp's half has consumed.  (The waits are the whole warp's: votes,
    // shuffles and tensor-memory reads follow, which the warp must reach, or give up on, as one.)
    // Waits for the accumulator and then for the per-column constants of the bt-th B tile.  In this order: the products of tile bt
    // come after half 0, which has a part in every tile, has seen the constants of tile bt - 4, so that the slot's barrier is in the
    // phase of tile bt or just past it.  A half that sat out an item may come here while the barrier is two phases behind, where its
    // parity is that of the phase waited for.
    static __device__ __forceinline__ bool acc_extra_wait(const Ctx &c, int k, int bt, int *status) {
        const bool ok = tc::mbar_wait_both_warp(c.bar(kBarAccFull + c.group), k & 1, c.bar(kBarXFull + (bt & (kExtraSlots - 1))),
                                                (bt / kExtraSlots) & 1, c.abort_flag, status);
        tc::tc_fence_after();
        return ok;
    }
    // For kernels whose epilogue reads its A half from shared memory: wait until the half of the
    // n-th item this group takes part in has landed (at Ctx::a_addr(n)) / hand it back (one arrival per warp).
    static __device__ __forceinline__ bool a_wait(const Ctx &c, int n, int *status) {
        return tc::mbar_wait_warp(c.bar(kBarAFull + (n % AST) * 2 + c.group), (n / AST) & 1, c.abort_flag, status);
    }
    static __device__ __forceinline__ void a_release(const Ctx &c, int n) {
        __syncwarp();
        if (c.lane == 0) tc::mbar_arrive(c.bar(kBarAEmpty + (n % AST) * 2 + c.group));
    }
    static __device__ __forceinline__ void acc_release(const Ctx &c) {
        tc::tc_fence_before();
        __syncwarp();
        if (c.lane == 0) tc::mbar_arrive(c.bar(kBarAccEmpty + c.group));
    }
    // The same for kernels whose accumulators are handed around by quad: whether this warp's takes part in a tile of ncols
    // columns, and (then) the wait and the release; `k` counts the tiles it has taken part in.
    static __device__ __forceinline__ bool takes_part(const Ctx &c, int ncols) { return ncols > c.colhalf * (NB / 2); }
    static __device__ __forceinline__ bool quad_wait(const Ctx &c, int k, int *status) {
        const bool ok = tc::mbar_wait_warp(c.bar(kBarAccFull + 2 * c.group + c.colhalf), k & 1, c.abort_flag, status);
        tc::tc_fence_after();
        return ok;
    }
    // Waits for the accumulator and, where tiles carry per-column constants (bt >= 0; the second scoring pass forms its own), then for
    // those of the bt-th B tile, lane by lane: only for an epilogue whose lanes stay in step whatever their waits return, until
    // pair_meet has told all of them.
    static __device__ __forceinline__ bool quad_extra_wait_lanes(const Ctx &c, int k, int bt, int *status) {
        const bool ok = tc::mbar_wait(c.bar(kBarAccFull + 2 * c.group + c.colhalf), k & 1, c.abort_flag, status) &&
                        (bt < 0 || tc::mbar_wait(c.bar(kBarXFull + (bt & (kExtraSlots - 1))), (bt / kExtraSlots) & 1, c.abort_flag, status));
        tc::tc_fence_after();
        return ok;
    }
    static __device__ __forceinline__ void quad_release(const Ctx &c) {
        tc::tc_fence_before();
        __syncwarp();
        if (c.lane == 0) tc::mbar_arrive(c.bar(kBarAccEmpty + 2 * c.group + c.colhalf));
    }
    // TMEM address of columns [32*chunk, 32*chunk+32) of this warp's half for its 32 lanes.
    static __device__ __forceinline__ uint32_t acc_addr(const Ctx &c, int chunk) {
        return c.tmem_base + c.group * NB + chunk * 32 + ((uint32_t)(c.quarter * 32) << 16);
    }

    // Runs f(chunk, values) over this warp's 32-column chunks of the current accumulator: the chunks of
    // its column half, as far as they lie below n_chunks (the tile's chunk count).  done() is called once, as soon as the last
    // chunk is in registers: the accumulator is handed back before that chunk is worked on (full-prefill flow, 28 units of 28
    // heads and 2176 tokens: 690 -> 664 us).
    template <class F, class Done>
    static __device__ __forceinline__ void for_each_chunk(const Ctx &c, int n_chunks, F &&f, Done &&done) {
        constexpr int kPer = NB / 64;
        const int lo = kPer * c.colhalf, hi = min(n_chunks, lo + kPer);
        if (hi <= lo) done();
        for (int ch = lo; ch < hi; ++ch) {
            uint32_t a[32];
            tc::tmem_ld32(acc_addr(c, ch), a);
            tc::tmem_ld_wait(a);
            if (ch + 1 >= hi) done();
            f(ch, a);
        }
    }
    // The same for epilogues in which all sixteen warps drain one accumulator at a time (warp = 32 lanes x
    // a quarter of the columns, both halves in turn): explicit half index, `k` = tiles of that half so far.
    static __device__ __forceinline__ bool acc_wait_h(const Ctx &c, int h, int k, int *status) {
        const bool ok = tc::mbar_wait_warp(c.bar(kBarAccFull + h), k & 1, c.abort_flag, status);
        tc::tc_fence_after();
        return ok;
    }
    static __device__ __forceinline__ void acc_release_h(const Ctx &c, int h) {
        tc::tc_fence_before();
        __syncwarp();
        if (c.lane == 0) tc::mbar_arrive(c.bar(kBarAccEmpty + h));
    }
    // (n of them: first, first + step, ...; f(which of them, chunk, values))
    template <class F, class Done>
    static __device__ __forceinline__ void for_each_chunk_h(const Ctx &c, int h, int first, int step, int n, F &&f, Done &&done) {
        if (n <= 0) done();
#pragma unroll 1
        for (int i = 0, ch = first; i < n; ++i, ch += step) {
            uint32_t a[32];
            tc::tmem_ld32(c.tmem_base + h * NB + ch * 32 + ((uint32_t)(c.quarter * 32) << 16), a);
            tc::tmem_ld_wait(a);
            if (i + 1 >= n) done();
            f(i, ch, a);
        }
    }
    // Meeting point of the two warps that share rows, with a vote: returns whether either warp has given up on a wait, so that both leave
    // the item loop together and neither is left alone at the next meeting.
    static __device__ __forceinline__ bool pair_meet(const Ctx &c, bool gave_up) { return meet_vote(1 + c.group * 4 + c.quarter, 64, gave_up); }
};

using Big = Skel<256, 1, 2>;       // long B streams
using Small = Skel<128, 2, 2>;     // few B columns per item: the A operand is the stream
using Resident = Skel<256, 2, 1>;  // ... with a B tile of up to 256 columns that stays for many items

}  // namespace tcs
}  // namespace flowmm
