// Matching (Eq. 9, Eq. 10) and merge (Eq. 5) of the fused call in one launch, for many heads with up to 64 pivots each (bf16, head_dim
// 128): match_small_tc.cuh's matching and merge_tc.cuh's product with the slot-by-token weight matrix, 128 tokens per step, so that K is
// read from HBM once for both and the matches never leave the CTA.  Products in the order of merge_tc.cuh: both give the same bits.
//
// CTAs are persistent, an item is a (unit, KV head).  Per step of 128 tokens:
//   warp 0      the K tile into a TMA ring; per item the candidate matrix, its reciprocal norms and slots;
//   warp 18     the K tile once more (it is in L2) and the V tile into a second ring: a tile would else stay from its load to the
//               products with the weights, and three such stages would bound the pace (2.3 us a step; so 2.1);
//   warp 1      S = K_tile C^T into a TMEM accumulator; then, a step behind, out^T += X_tile^T W_tile^T for K and V (the tiles read as
//               MN-major operands);
//   warps 2-9   two teams, which take the steps by turns, a thread per token: norm from the K stage, winner among the admissible columns
//               (match_unit), the token's entry of W^T (bf16, K-major) and its share of the slot's weight sum (fixed point);
//   warps 10-17 out^T from TMEM, scaled by 1 / (1 + sum of weights), as bf16 rows, while the next item's steps fill a second set.
// The products of step s + 1 with the candidates are issued before those of step s with the weights, across items too, so that the
// teams work on one step while the tensor core takes another.
// Bound by HBM and, where steps are few, by a chain of five waits per step.  Against the two launches, which read K twice, us for the whole
// call: 1024 heads of 1200 tokens and 60 pivots 315 -> 268, of 640 and 64 148 -> 132, of 512 and 51 122 -> 106, of 400 and 40 105 -> 97, 256 of
// 640 42.9 -> 39.7, 96 of 250 21.7 -> 19.2.
#pragma once
#include "common.cuh"
#include "decode_tc.cuh"
#include "match_small_tc.cuh"
#include "merge_tc.cuh"
#include "tc_common.cuh"

namespace flowmm {
namespace mmt {

constexpr int kTile = 128;
constexpr int kTeams = 2;
constexpr int kReaderWarp = 2 + 4 * kTeams;                  // first reader warp
constexpr int kLoadWarp = kReaderWarp + 8;                   // the second ring's producer
constexpr int kThreads = 32 * kLoadWarp + 32;
constexpr int kMaxSlots = 64;                                // (two sets of out^T beside two accumulators of S in TMEM)
constexpr uint32_t kStageBytes = kTile * 128 * 2, kPanel = kStageBytes / 2;
constexpr int kStagesK = 2, kStagesX = 3;                    // of the two rings
constexpr int kBarKFull = 0, kBarKEmpty = kBarKFull + kStagesK, kBarXFull = kBarKEmpty + kStagesK, kBarXEmpty = kBarXFull + kStagesX,
              kBarCandFull = kBarXEmpty + kStagesX, kBarMetaEmpty = kBarCandFull + 2, kBarCandEmpty = kBarMetaEmpty + 2,
              kBarSFull = kBarCandEmpty + 1, kBarSFree = kBarSFull + 2, kBarWFull = kBarSFree + 2, kBarWEmpty = kBarWFull + 2,
              kBarOutFull = kBarWEmpty + 2, kBarOutEmpty = kBarOutFull + 2, kBarSumFull = kBarOutEmpty + 2,
              kBarSumEmpty = kBarSumFull + 2, kNumBars = kBarSumEmpty + 2;
constexpr uint32_t kOutCol = 256, kSetCols = 128, kVCol = 64;   // TMEM: products with the candidates below column 256; sets of out^T, V's part of a set

// Shared memory: the rings, two W buffers and the candidates, then what the threads share.
constexpr uint32_t kSmemX = kStagesK * kStageBytes, kSmemW = kSmemX + kStagesX * kStageBytes;
struct Smem { uint32_t cand, meta, stash, sums, inv, bars, total; };
__host__ __device__ inline Smem smem_plan(int B, int Ctot) {
    Smem m;
    m.cand = kSmemW + 2u * mtc::w_bytes(B);
    m.meta = m.cand + (uint32_t)Ctot * 256u;                 // of two heads by turns: float scale[Ctot], int slot[Ctot]
    m.stash = m.meta + 2u * 8u * (uint32_t)Ctot;             // per team: 8 floats per row
    m.sums = m.stash + kTeams * 4096u;                       // weight sums of two items by turns
    m.inv = m.sums + 2u * 4u * kMaxSlots;                    // reciprocal normalisers
    m.bars = m.inv + 4u * kMaxSlots;
    m.total = m.bars + 8u * kNumBars + 16u;
    return m;
}

struct Args {
    const int *cand_count, *cand_slot, *rank, *strategy;
    const float *cand_scale;
    const uint8_t *modality;
    int *match;                  // nullptr, or [UH, E] (then match_sim too)
    float *match_sim;
    void *k_out, *v_out;
    int *status;
    int Hkv, L, E, B, Ctot, n_items, merge_mode;
    Smem at;
    int64_t kos[3], vos[3];
};

__device__ __forceinline__ void reader_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

__global__ void __launch_bounds__(kThreads, 1)
match_merge_tc_kernel(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap, const __grid_constant__ CUtensorMap cand_map,
                      const Args A) {
    extern __shared__ __align__(1024) uint8_t mmt_smem[];
    const uint32_t base = tc::smem_u32(mmt_smem), bars = base + A.at.bars;
    const int warp = tc::warp_number(), lane = threadIdx.x & 31;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mmt_smem + A.at.bars + 8 * kNumBars);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(mmt_smem + A.at.bars + 8 * kNumBars + 4);
    if ((base & 1023u) != 0) {
        predecessor_done();
        if (threadIdx.x == 0) atomicCAS(A.status, 0, 6);
        return;
    }
    const int N = mtc::slots16(A.B);
    const uint32_t wsize = mtc::w_bytes(A.B), wpanel = (uint32_t)N * 128u;
    unsigned *wsum = reinterpret_cast<unsigned *>(mmt_smem + A.at.sums);                  // [2][kMaxSlots], units of 1 / kSumScale
    float *inv_s = reinterpret_cast<float *>(mmt_smem + A.at.inv);
    auto bar = [&](int i) { return bars + 8u * i; };
    if (threadIdx.x == 0) {
        for (int i = 0; i < kNumBars; ++i) {
            int count = 1;
            if (i >= kBarKEmpty && i < kBarXFull) count = 5;                              // the products and the warps that read the norm
            if (i >= kBarMetaEmpty && i < kBarCandEmpty) count = 4 * kTeams;              // every team warp, when it is done with the head
            if (i >= kBarSFree && i < kBarWFull) count = 4;
            if (i >= kBarWFull && i < kBarWEmpty) count = kTile;
            if (i >= kBarOutEmpty && i < kBarSumFull) count = 256;
            if (i >= kBarSumFull) count = 256;                                            // the teams' threads; the readers
            tc::mbar_init(bar(i), count);
        }
        *abort_flag = 0;
        tc::mbar_init_fence();
        tc::tma_prefetch_desc(&kmap);
        tc::tma_prefetch_desc(&vmap);
        tc::tma_prefetch_desc(&cand_map);
    }
    if (warp == 1) tc::tmem_alloc(tc::smem_u32(tmem_slot), 512);
    for (uint32_t o = threadIdx.x * 16; o < 2 * wsize; o += kThreads * 16) dtc::sts128u(base + kSmemW + o, make_uint4(0, 0, 0, 0));
    for (int i = threadIdx.x; i < 2 * kMaxSlots; i += kThreads) wsum[i] = 0u;
    dtc::fence_proxy_async();
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    predecessor_done();
    successor_may_start();
    const int nt = (A.L + kTile - 1) / kTile;
    // a tile of rows into a ring's stage
    auto load_tile = [&](uint32_t dst, const CUtensorMap *m, uint32_t full, int c, int h, int u) {
        if (tc::elect_one()) {
            tc::mbar_expect_tx(full, kStageBytes);
            tc::tma_load_4d(dst, m, full, 0, c * kTile, h, u);
            tc::tma_load_4d(dst + kPanel, m, full, 64, c * kTile, h, u);
        }
        __syncwarp();
    };
    // winding down after a timeout: copies already issued to n barriers get a moment to land
    auto let_land = [&](int first, int n) {
        for (int b = 0; b < n; ++b)
            for (int s = 0; s < (1 << 16) && !tc::mbar_try_wait(bar(first + b), 0) && !tc::mbar_try_wait(bar(first + b), 1); ++s) {}
    };

    if (warp == 0) {
        bool ok = true;
        int i = 0, it = 0;
        for (int uh = blockIdx.x; ok && uh < A.n_items; uh += gridDim.x, ++it) {
            const int u = uh / A.Hkv, h = uh - u * A.Hkv, hp = it & 1;
            for (int c = 0; ok && c < nt; ++c, ++i) {
                const int st = i % kStagesK;
                ok = tc::mbar_wait_warp(bar(kBarKEmpty + st), ((i / kStagesK) & 1) ^ 1, abort_flag, A.status);
                if (!ok) break;
                load_tile(base + st * kStageBytes, &kmap, bar(kBarKFull + st), c, h, u);
                if (c == 0) {                                        // the head's candidates, right behind its first tile
                    ok = tc::mbar_wait_warp(bar(kBarCandEmpty), (it & 1) ^ 1, abort_flag, A.status) &&
                         tc::mbar_wait_warp(bar(kBarMetaEmpty + hp), ((it >> 1) & 1) ^ 1, abort_flag, A.status);
                    if (!ok) break;
                    if (tc::elect_one()) {
                        const uint32_t cd = base + A.at.cand, md = base + A.at.meta + hp * 8u * (uint32_t)A.Ctot, full = bar(kBarCandFull + hp);
                        tc::mbar_expect_tx(full, 264u * (uint32_t)A.Ctot);
                        tc::tma_load_4d(cd, &cand_map, full, 0, 0, uh, 0);
                        tc::tma_load_4d(cd + (uint32_t)A.Ctot * 128u, &cand_map, full, 64, 0, uh, 0);
                        tc::bulk_load(md, A.cand_scale + (int64_t)uh * A.Ctot, 4u * (uint32_t)A.Ctot, full);
                        tc::bulk_load(md + 4u * (uint32_t)A.Ctot, A.cand_slot + (int64_t)uh * A.Ctot, 4u * (uint32_t)A.Ctot, full);
                    }
                    __syncwarp();
                }
            }
        }
        if (!ok) { let_land(kBarKFull, kStagesK); let_land(kBarCandFull, 2); }
    } else if (warp == kLoadWarp) {
        bool ok = true;
        int j = 0;                                                   // tiles so far: K's and V's of every step
        for (int uh = blockIdx.x; ok && uh < A.n_items; uh += gridDim.x) {
            const int u = uh / A.Hkv, h = uh - u * A.Hkv;
            for (int t = 0; ok && t < 2 * nt; ++t, ++j) {
                const int st = j % kStagesX;
                ok = tc::mbar_wait_warp(bar(kBarXEmpty + st), ((j / kStagesX) & 1) ^ 1, abort_flag, A.status);
                if (ok) load_tile(base + kSmemX + st * kStageBytes, t & 1 ? &vmap : &kmap, bar(kBarXFull + st), t >> 1, h, u);
            }
        }
        if (!ok) let_land(kBarXFull, kStagesX);
    } else if (warp == 1) {
        const uint32_t idesc_out = tc::idesc_bf16(128, (uint32_t)N) | (1u << 15);        // A operand MN-major
        const uint32_t lead = (kPanel >> 4) << 16;                                       // (and the stride between its panels)
        bool ok = true;
        int j = 0;                                                   // tiles of the second ring so far
        // products of step i (of item number it; its first, its last step) with its weights
        auto merge = [&](int i, int it, bool first, bool last) {
            const int set = it & 1, wb = i & 1;
            if (first) ok = ok && tc::mbar_wait_warp(bar(kBarOutEmpty + set), ((it >> 1) & 1) ^ 1, abort_flag, A.status);   // the set's item before is read out
            ok = ok && tc::mbar_wait_warp(bar(kBarWFull + wb), (i >> 1) & 1, abort_flag, A.status);
            const uint32_t w_lo = tc::desc_lo(base + kSmemW + wb * wsize), d = tmem + kOutCol + set * kSetCols;
#pragma unroll 1
            for (int t = 0; ok && t < 2; ++t, ++j) {                 // K, V
                const int st = j % kStagesX;
                ok = tc::mbar_wait_warp(bar(kBarXFull + st), (j / kStagesX) & 1, abort_flag, A.status);
                if (!ok) break;
                tc::tc_fence_after();
                const uint32_t a_lo = tc::desc_lo(base + kSmemX + st * kStageBytes) | lead, to = d + t * kVCol;
                if (tc::elect_one()) {
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        tc::umma_bf16(to, a_lo + q * 128, tc::kDescSw128Hi, w_lo + (q >> 2) * (wpanel >> 4) + (q & 3) * 2, tc::kDescSw128Hi,
                                      idesc_out, !first || q > 0);
                    tc::umma_commit(bar(kBarXEmpty + st));
                    if (t == 1) tc::umma_commit(bar(kBarWEmpty + wb));
                    if (t == 1 && last) tc::umma_commit(bar(kBarOutFull + set));
                }
                __syncwarp();
            }
        };
        int i = 0, it = 0;
        auto counts = [&](int uh) { return uh < A.n_items ? make_int2(A.cand_count[2 * uh], A.cand_count[2 * uh + 1]) : make_int2(0, 0); };
        int2 n_next = counts(blockIdx.x);                            // an item ahead
        for (int uh = blockIdx.x; ok && uh < A.n_items; uh += gridDim.x, ++it) {
            const int2 n_cand = n_next;
            n_next = counts(uh + gridDim.x);
            const int cols = n_cand.y > 0 ? ((n_cand.x + 31) & ~31) + n_cand.y : n_cand.x;   // columns up to the last candidate
            const uint32_t b_panel = (uint32_t)A.Ctot * 128u, b_lo = tc::desc_lo(base + A.at.cand), idesc = tc::idesc_bf16(kTile, (uint32_t)((cols + 15) & ~15));
            for (int c = 0; ok && c < nt; ++c, ++i) {
                const int st = i % kStagesK, set = i & 1;
                if (c == 0) ok = tc::mbar_wait_warp(bar(kBarCandFull + (it & 1)), (it >> 1) & 1, abort_flag, A.status);
                ok = ok && tc::mbar_wait_warp(bar(kBarKFull + st), (i / kStagesK) & 1, abort_flag, A.status) &&
                     tc::mbar_wait_warp(bar(kBarSFree + set), ((i >> 1) & 1) ^ 1, abort_flag, A.status);
                if (!ok) break;
                tc::tc_fence_after();
                const uint32_t a_lo = tc::desc_lo(base + st * kStageBytes);
                if (tc::elect_one()) {
                    if (cols > 0) {
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            tc::umma_bf16(tmem + mst::kUnitCols * set, a_lo + (q >> 2) * (kPanel >> 4) + (q & 3) * 2, tc::kDescSw128Hi,
                                          b_lo + (q >> 2) * (b_panel >> 4) + (q & 3) * 2, tc::kDescSw128Hi, idesc, q > 0);
                    }
                    tc::umma_commit(bar(kBarSFull + set));
                    tc::umma_commit(bar(kBarKEmpty + st));
                    if (c == nt - 1) tc::umma_commit(bar(kBarCandEmpty));
                }
                __syncwarp();
                if (c > 0) merge(i - 1, it, c == 1, false);
                else if (it > 0) merge(i - 1, it - 1, nt == 1, true);   // (the last step of the item before)
            }
        }
        if (ok && it > 0) merge(i - 1, it - 1, nt == 1, true);
    } else if (warp < kReaderWarp) {
        const int team = (warp - 2) >> 2, wq = warp & 3;
        const int row = 32 * wq + lane;                              // TMEM lane = token of the step
        const uint32_t trow = tmem + mst::kUnitCols * team + ((uint32_t)(32 * wq) << 16);
        const uint32_t wrow = base + A.at.stash + team * 4096 + row * 32;
        // the team's W buffer, and where this token's entry goes in a panel row: 64 tokens per 128-byte row, 16-byte groups swizzled by row
        const uint32_t w = base + kSmemW + team * wsize + (uint32_t)(row >> 6) * wpanel + (uint32_t)((row & 7) << 1);
        const int tok_grp = (row & 63) >> 3;
        uint32_t entry = 0;                                          // where this thread's last one is
        bool ok = true;
        // what a step needs from global memory is fetched a step of this team ahead, what an item needs an item ahead
        int mod_next = 0, rank_next = -1;
        auto fetch = [&](int uh, int c) {                            // (c may lie in an item after it)
            while (c >= nt && uh < A.n_items) { c -= nt; uh += gridDim.x; }
            const int token = c * kTile + row;
            mod_next = 0; rank_next = -1;
            if (uh < A.n_items && token < A.L) {
                mod_next = A.modality[(int64_t)(uh / A.Hkv) * A.L + token];
                rank_next = A.rank[(int64_t)uh * A.L + token];
            }
        };
        fetch(blockIdx.x, team);
        struct Head { int n_text, n_vis, strategy; };
        auto fetch_head = [&](int uh) -> Head {
            if (uh >= A.n_items) return Head{0, 0, 0};
            return Head{A.cand_count[2 * uh], A.cand_count[2 * uh + 1], A.strategy[uh / A.Hkv]};
        };
        Head head_next = fetch_head(blockIdx.x);
        int i = 0, it = 0;
        for (int uh = blockIdx.x; uh < A.n_items; uh += gridDim.x, ++it) {
            const int hp = it & 1;
            const uint32_t md = base + A.at.meta + hp * 8u * (uint32_t)A.Ctot;
            const int n_text = head_next.n_text, n_vis = head_next.n_vis;
            const bool intra = head_next.strategy == 0;
            head_next = fetch_head(uh + gridDim.x);
            // blocks of 16 columns: text group [0, tb) and visual group [vb, ve)
            const int t0 = (n_text + 31) & ~31, tb = (n_text + 15) >> 4, vb = t0 >> 4, ve = n_vis > 0 ? (t0 + n_vis + 15) >> 4 : 0;
            unsigned *sums = wsum + hp * kMaxSlots;
            // scales and slots have landed; the sums are zero again, the item before the last one having been read out
            ok = ok && tc::mbar_wait_warp(bar(kBarCandFull + hp), (it >> 1) & 1, abort_flag, A.status);
            ok = ok && tc::mbar_wait_warp(bar(kBarSumEmpty + hp), ((it >> 1) & 1) ^ 1, abort_flag, A.status);
            for (int c = 0; c < nt; ++c, ++i) {
                if ((i & 1) != team) continue;
                const int st = i % kStagesK, token = c * kTile + row;
                const bool in_range = token < A.L;
                const int my_mod = mod_next, my_rank = rank_next;
                fetch(uh, c + kTeams);
                const bool want_text = in_range && (!intra || my_mod == 0), want_vis = in_range && (!intra || my_mod != 0);
                // the token's key row sits in the K stage (128-byte rows, 16-byte units XOR-swizzled by the row index)
                ok = ok && tc::mbar_wait_warp(bar(kBarKFull + st), (i / kStagesK) & 1, abort_flag, A.status);
                const uint32_t a_row = base + st * kStageBytes + row * 128;
                float ssq = 0.f;
                if (ok) ssq = row_half_ssq(a_row, row) + row_half_ssq(a_row + kPanel, row);
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(bar(kBarKEmpty + st));
                ok = ok && tc::mbar_wait_warp(bar(kBarSFull + team), (i >> 1) & 1, abort_flag, A.status);
                tc::tc_fence_after();
                float best;
                int slot;
                mst::match_unit(trow, md, 4u * (uint32_t)A.Ctot, wrow, 0, tb, vb, ve, want_text, want_vis, A.Ctot, ok, A.status, best, slot, [&]() {
                    tc::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(bar(kBarSFree + team));     // this warp has read the accumulator
                });
                const bool member = my_rank >= 0;                    // a non-pivot: its match and weight; a pivot: its own slot, weight 1
                float weight = 1.f;
                if (member) {
                    float sim = 0.f;
                    if (slot >= 0 && ssq > 0.f) sim = best * rsqrtf(ssq);
                    if (A.match && in_range && ok && index_ok(my_rank, A.E, A.status)) {
                        A.match[(int64_t)uh * A.E + my_rank] = slot;
                        A.match_sim[(int64_t)uh * A.E + my_rank] = sim;
                    }
                    if (A.merge_mode != 1) weight = __expf(sim - 1.f);
                } else slot = -my_rank - 2;
                ok = ok && tc::mbar_wait_warp(bar(kBarWEmpty + team), ((i >> 1) & 1) ^ 1, abort_flag, A.status);
                if (ok) {
                    if (entry) dtc::sts16(entry, 0);                 // take back what this thread wrote last time
                    entry = 0;
                    if (in_range && slot >= 0 && slot < A.B) {
                        const __nv_bfloat16 wt = __float2bfloat16_rn(weight);
                        entry = w + (uint32_t)slot * 128u + (uint32_t)((tok_grp ^ (slot & 7)) << 4);
                        dtc::sts16(entry, __bfloat16_as_ushort(wt));
                        if (member) atomicAdd(sums + slot, (unsigned)(__bfloat162float(wt) * mtc::kSumScale + 0.5f));
                    }
                }
                dtc::fence_proxy_async();
                tc::mbar_arrive(bar(kBarWFull + team));
            }
            tc::mbar_arrive(bar(kBarSumFull + hp));                  // this thread's part of the item's weight sums is complete
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(bar(kBarMetaEmpty + hp)); // done with the head's scales and slots
        }
    } else {
        // readers: thread = output dim; columns = slots; the first four warps take K, the others V
        const int e = threadIdx.x - 32 * kReaderWarp, t = e >> 7;
        const uint32_t trow = tmem + kOutCol + t * kVCol + ((uint32_t)(32 * (warp & 3)) << 16);
        const int64_t stride = t ? A.vos[2] : A.kos[2];
        bool ok = true;
        int it = 0;
        for (int uh = blockIdx.x; uh < A.n_items; uh += gridDim.x, ++it) {
            const int u = uh / A.Hkv, h = uh - u * A.Hkv, set = it & 1, use = it >> 1;
            unsigned *sums = wsum + set * kMaxSlots;
            ok = ok && tc::mbar_wait_warp(bar(kBarSumFull + set), use & 1, abort_flag, A.status);
            if (ok && e < N) {
                inv_s[e] = 1.f / (1.f + (float)sums[e] * (1.f / mtc::kSumScale));
                sums[e] = 0u;
            }
            reader_sync();
            tc::mbar_arrive(bar(kBarSumEmpty + set));
            ok = ok && tc::mbar_wait_warp(bar(kBarOutFull + set), use & 1, abort_flag, A.status);
            tc::tc_fence_after();
            if (ok) {
                __nv_bfloat16 *out = static_cast<__nv_bfloat16 *>(t ? A.v_out : A.k_out) +
                                     (t ? u * A.vos[0] + h * A.vos[1] : u * A.kos[0] + h * A.kos[1]) + 32 * (warp & 3) + (lane & ~3);
#pragma unroll 1
                for (int s0 = 0; s0 < A.B; s0 += 32) {
                    uint32_t acc[32];
                    tc::tmem_ld32(trow + set * kSetCols + s0, acc);
                    tc::tmem_ld_wait(acc);
                    mtc::store_slots32(acc, inv_s, out, stride, s0, A.B, lane);
                }
            }
            tc::tc_fence_before();
            reader_sync();                                           // inv_s may be rewritten
            tc::mbar_arrive(bar(kBarOutEmpty + set));                // ... and the set reused
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == 1) tc::tmem_dealloc(tmem, 512);
}

}  // namespace mmt
}  // namespace flowmm
