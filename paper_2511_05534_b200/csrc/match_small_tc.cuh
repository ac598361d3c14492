// Matching step (Eq. 9 and Eq. 10) on the tensor cores for short candidate lists (at most 256 columns
// per head, i.e. budgets of up to 224 pivots): the whole candidate matrix of a head is one operand tile.
//
// Same preparation as match_tc.cuh (admissible pivots gathered into a dense matrix, text group first, visual group from
// the next multiple of 32, NaN scales where there is no candidate).
// The 128-token tiles of all heads form one sequence, of which every CTA (one per SM) takes an equal run, so that few long
// heads spread over all SMs.  Per head of its run: warp 0 loads the head's candidate tile, its reciprocal norms and
// slots (double-buffered by head up to 128 columns) and streams the token tiles through a TMA ring; warp 1 issues
// S = K_tile C^T (tcgen05.mma, M = 128 tokens) in units of up to 128 candidate columns, one unit per tile or two, into four
// TMEM accumulators (both run whole and elect a thread at each instruction); four teams of four warps take the units in turn: a thread owns a token, reads its key row from the A
// stage for the norm, walks the blocks of 16 columns that a token of its warp may take, text group then visual group, keeps
// the running maximum per group of 8 columns and recovers the exact column at the end.  With two units per tile the two
// teams of a tile meet in shared memory, row by row.
// Bound by the epilogue's latency (about 3000 clocks from a unit's products to its release, four units in flight).  Against
// whole heads per CTA and one accumulator per tile: 8 heads of 1471 tokens, 179 candidates 18.5 -> 10.4 us, 112 of 2176,
// 250 candidates 36 -> 32 us, 32 of 640 12.2 -> 10.8 us.
#pragma once
#include "common.cuh"
#include "match_tc.cuh"
#include "tc_common.cuh"

namespace flowmm {
namespace mst {

constexpr int kTile = 128;
constexpr int kStages = 4;
constexpr int kMaxCols = 256;
constexpr int kUnitCols = 128;                // candidate columns of an accumulator
constexpr int kTeams = 4;                     // and accumulators
constexpr int kThreads = 64 + kTeams * 128;
constexpr uint32_t kStageBytes = kTile * 128 * 2, kPanel = kStageBytes / 2;
constexpr uint32_t kBRegion = kMaxCols * 256;                      // candidate tiles (two panels of N rows each): two of up to 128 rows or one
constexpr uint32_t kSmemB = kStages * kStageBytes;
constexpr uint32_t kSmemMeta = kSmemB + kBRegion;                  // per candidate buffer: float scale[N], int slot[N]
constexpr uint32_t kSmemStash = kSmemMeta + 4096;                  // per team: 8 floats per row
constexpr uint32_t kSmemBar = kSmemStash + kTeams * 4096;
constexpr int kBarFull = 0, kBarEmpty = kStages, kBarBFull = 2 * kStages, kBarBEmpty = kBarBFull + 2,
              kBarAccFull = kBarBEmpty + 2, kBarSetFree = kBarAccFull + kTeams, kNumBars = kBarSetFree + kTeams;
constexpr uint32_t kSmemBytes = kSmemBar + 8 * kNumBars + 16;
static_assert(kSmemBytes <= 232448, "shared memory budget");

struct Args {
    const int *cand_count, *cand_slot, *rank, *strategy;
    const float *cand_scale;
    const uint8_t *modality;
    int *match;
    float *match_sim;
    int2 *tokmap;          // nullptr, or [UH, L]: the (slot, weight) table of the tensor-core merge, written here instead of by merge_map_kernel
    int *status;
    int Hkv, L, E, Ctot, n_heads, merge_mode;
    FastDiv by_nt, by_hkv; // exact division of tile numbers by the tiles of a head and of head numbers by Hkv
};

__device__ __forceinline__ void pair_sync(int pair, int wq) { asm volatile("bar.sync %0, 64;" ::"r"(1 + pair * 4 + wq) : "memory"); }

// The running winner of a thread's token in one candidate group: its similarity (still times the row's norm) and where its
// group of 8 columns is; the 8 values are in the thread's stash.
struct Winner { float best; int col; };

// The winner of a thread's token among the candidate columns of a unit: its similarity (still times the row's norm) and pivot slot
// (-1: none).  trow: TMEM address of the unit's columns for the warp's lanes; md, slot_off: the head's scales in shared memory and how
// far behind them its slots are; wrow: the thread's stash; blocks of 16 columns, numbered from the head's first column: the unit's first
// one blk0, the text group's [blk0, tb) and the visual group's [vb, ve).  Call with the whole warp; release() as soon as the
// accumulator has been read (whatever the waits returned: !ok).
template <class Release>
__device__ __forceinline__ void match_unit(uint32_t trow, uint32_t md, uint32_t slot_off, uint32_t wrow, int blk0, int tb, int vb, int ve,
                                           bool want_text, bool want_vis, int N, bool ok, int *status, float &best, int &slot,
                                           Release &&release) {
    // Candidates are laid out text group first, each group by ascending slot, so the first maximum of a group is
    // its lowest slot; the groups' winners meet by (similarity, slot), so that equal similarities go to the lower.
    auto slot_of = [&](const Winner &w) -> int {         // lowest column of the winning 8 that holds the maximum
        if (w.col < 0) return -1;
        int idx = 0;
#pragma unroll
        for (int q4 = 1; q4 >= 0; --q4) {
            const float4 v = tc::lds128(wrow + q4 * 16);
            if (v.w == w.best) idx = 4 * q4 + 3;
            if (v.z == w.best) idx = 4 * q4 + 2;
            if (v.y == w.best) idx = 4 * q4 + 1;
            if (v.x == w.best) idx = 4 * q4;
        }
        return index_ok(w.col + idx, N, status) ? __float_as_int(tc::lds32(md + slot_off + (w.col + idx) * 4)) : -1;
    };
    auto block = [&](int blk, const uint32_t *acc, bool want, Winner &w) {
        float v[16];
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) {                 // a column that is no candidate has scale NaN and never wins
            const float4 s4 = tc::lds128(md + (blk * 4 + q4) * 16);
            const float2 p01 = tc::fmul2(make_float2(__uint_as_float(acc[4 * q4]), __uint_as_float(acc[4 * q4 + 1])), make_float2(s4.x, s4.y));
            const float2 p23 = tc::fmul2(make_float2(__uint_as_float(acc[4 * q4 + 2]), __uint_as_float(acc[4 * q4 + 3])), make_float2(s4.z, s4.w));
            v[4 * q4] = p01.x; v[4 * q4 + 1] = p01.y; v[4 * q4 + 2] = p23.x; v[4 * q4 + 3] = p23.y;
        }
#pragma unroll
        for (int h8 = 0; h8 < 2; ++h8) {                 // two groups of 8 columns, in column order
            const float q8 = tc::max3(tc::max3(v[8 * h8], v[8 * h8 + 1], v[8 * h8 + 2]),
                                      tc::max3(v[8 * h8 + 3], v[8 * h8 + 4], v[8 * h8 + 5]), fmaxf(v[8 * h8 + 6], v[8 * h8 + 7]));
            if (want && q8 > w.best) {                   // strict: an earlier group keeps a tie (false for NaN)
                w.best = q8;
                w.col = blk * 16 + 8 * h8;
                tc::sts128(wrow, v[8 * h8], v[8 * h8 + 1], v[8 * h8 + 2], v[8 * h8 + 3]);
                tc::sts128(wrow + 16, v[8 * h8 + 4], v[8 * h8 + 5], v[8 * h8 + 6], v[8 * h8 + 7]);
            }
        }
    };
    auto walk = [&](int lo, int hi, bool want) -> Winner {    // blocks [lo, hi); pairs of blocks per read
        Winner w = {-INFINITY, -1};
        if (!__any_sync(0xFFFFFFFFu, want)) return w;
        int blk = lo;
#pragma unroll 1
        for (; blk + 1 < hi; blk += 2) {
            uint32_t acc[32];
            tc::tmem_ld32(trow + (blk - blk0) * 16, acc);
            tc::tmem_ld_wait(acc);
            block(blk, acc, want, w);
            block(blk + 1, acc + 16, want, w);
        }
        if (blk < hi) {
            uint32_t acc[16];
            tc::tmem_ld16(trow + (blk - blk0) * 16, acc);
            tc::tmem_ld_wait(acc);
            block(blk, acc, want, w);
        }
        return w;
    };
    best = -INFINITY;
    slot = -1;
    Winner wv = {-INFINITY, -1};
    if (ok) {
        const Winner wt = walk(blk0, tb, want_text);
        best = wt.best;
        slot = slot_of(wt);
        wv = walk(vb, ve, want_vis);
    }
    release();
    if (ok) {
        const int slot_v = slot_of(wv);
        if (match_better(wv.best, slot_v, best, slot)) { best = wv.best; slot = slot_v; }
    }
}

__global__ void __launch_bounds__(kThreads, 1)
match_small_tc_kernel(const __grid_constant__ CUtensorMap k_map, const __grid_constant__ CUtensorMap cand_map, const Args A) {
    extern __shared__ __align__(1024) uint8_t mst_smem[];
    const uint32_t base = tc::smem_u32(mst_smem), bars = base + kSmemBar;
    const int warp = tc::warp_number(), lane = threadIdx.x & 31;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(mst_smem + kSmemBar + 8 * kNumBars + 4);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mst_smem + kSmemBar + 8 * kNumBars);
    if ((base & 1023u) != 0) {
        predecessor_done();
        if (threadIdx.x == 0) atomicCAS(A.status, 0, 6);
        return;
    }
    const int nt = (A.L + kTile - 1) / kTile, N = A.Ctot;
    const int64_t n_tiles = (int64_t)A.n_heads * nt;
    const int g_lo = (int)(n_tiles * blockIdx.x / gridDim.x), g_hi = (int)(n_tiles * (blockIdx.x + 1) / gridDim.x);   // this CTA's run
    const uint32_t b_bytes = (uint32_t)N * 256u, b_panel = (uint32_t)N * 128u;
    const int units = N <= kUnitCols ? 1 : 2, n_bbuf = N <= 128 ? 2 : 1;
    const uint32_t b_stride = kBRegion / 2, m_stride = 2048, slot_off = 4u * (uint32_t)N;
    auto bar = [&](int i) { return bars + 8u * i; };
    if (threadIdx.x == 0) {
        for (int i = 0; i < kNumBars; ++i) {
            int count = 1;
            if (i >= kBarEmpty && i < kBarBFull) count = 1 + 4 * units;      // the MMAs and the warps that read the norm
            if (i >= kBarBEmpty && i < kBarAccFull) count = 1 + 4 * kTeams;  // the MMAs and every warp, when it is done with the head
            if (i >= kBarSetFree) count = 4;
            tc::mbar_init(bar(i), count);
        }
        *abort_flag = 0;
        tc::mbar_init_fence();
        tc::tma_prefetch_desc(&k_map);
        tc::tma_prefetch_desc(&cand_map);
    }
    if (warp == 1) tc::tmem_alloc(tc::smem_u32(tmem_slot), 512);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    predecessor_done();
    if (A.tokmap) successor_may_start();   // (the merge, a block per SM; the small blocks that come behind the step alone: 56 heads of 1200, 10.6 -> 12.4)

    // every role walks the heads of the run: tiles [t_lo, t_hi) of head uh, hc heads before it, tile number i of the run
    if (warp == 0) {
        bool ok = true;
        int hc = 0;
        for (int g = g_lo; ok && g < g_hi; ++hc) {
            const int uh = (int)A.by_nt.div(g), u = (int)A.by_hkv.div(uh), h = uh - u * A.Hkv, hp = hc % n_bbuf;
            ok = tc::mbar_wait_warp(bar(kBarBEmpty + hp), ((hc / n_bbuf) & 1) ^ 1, abort_flag, A.status);
            if (!ok) break;
            const uint32_t bd = base + kSmemB + hp * b_stride, md = base + kSmemMeta + hp * m_stride;
            if (tc::elect_one()) {
                tc::mbar_expect_tx(bar(kBarBFull + hp), b_bytes + 8u * (uint32_t)N);
                tc::tma_load_4d(bd, &cand_map, bar(kBarBFull + hp), 0, 0, uh, 0);
                tc::tma_load_4d(bd + b_panel, &cand_map, bar(kBarBFull + hp), 64, 0, uh, 0);
                tc::bulk_load(md, A.cand_scale + (int64_t)uh * N, 4u * (uint32_t)N, bar(kBarBFull + hp));
                tc::bulk_load(md + slot_off, A.cand_slot + (int64_t)uh * N, 4u * (uint32_t)N, bar(kBarBFull + hp));
            }
            __syncwarp();
            for (const int end = min(g_hi, (uh + 1) * nt); ok && g < end; ++g) {
                const int i = g - g_lo, t = g - uh * nt, st = i % kStages;
                ok = tc::mbar_wait_warp(bar(kBarEmpty + st), ((i / kStages) & 1) ^ 1, abort_flag, A.status);
                if (!ok) break;
                const uint32_t dst = base + st * kStageBytes;
                if (tc::elect_one()) {
                    tc::mbar_expect_tx(bar(kBarFull + st), kStageBytes);
                    tc::tma_load_4d(dst, &k_map, bar(kBarFull + st), 0, t * kTile, h, u);
                    tc::tma_load_4d(dst + kPanel, &k_map, bar(kBarFull + st), 64, t * kTile, h, u);
                }
                __syncwarp();
            }
        }
        if (!ok) {       // winding down after a timeout: give copies already issued a moment to land
            for (int b = 0; b < kStages; ++b)
                for (int s = 0; s < (1 << 16) && !tc::mbar_try_wait(bar(kBarFull + b), 0) && !tc::mbar_try_wait(bar(kBarFull + b), 1); ++s) {}
            for (int b = 0; b < 2; ++b)
                for (int s = 0; s < (1 << 16) && !tc::mbar_try_wait(bar(kBarBFull + b), 0) && !tc::mbar_try_wait(bar(kBarBFull + b), 1); ++s) {}
        }
    } else if (warp == 1) {
        bool ok = true;
        int hc = 0;
        int n_text_next = A.cand_count[2 * A.by_nt.div(g_lo)], n_vis_next = A.cand_count[2 * A.by_nt.div(g_lo) + 1];   // a head ahead
        for (int g = g_lo; ok && g < g_hi; ++hc) {
            const int uh = (int)A.by_nt.div(g), hp = hc % n_bbuf;
            const int n_text = n_text_next, n_vis = n_vis_next;
            if (uh + 1 < A.n_heads) { n_text_next = A.cand_count[2 * uh + 2]; n_vis_next = A.cand_count[2 * uh + 3]; }
            const int cols = n_vis > 0 ? ((n_text + 31) & ~31) + n_vis : n_text;         // columns up to the last candidate
            ok = tc::mbar_wait_warp(bar(kBarBFull + hp), (hc / n_bbuf) & 1, abort_flag, A.status);
            const uint32_t bd = base + kSmemB + hp * b_stride;
            for (const int end = min(g_hi, (uh + 1) * nt); ok && g < end; ++g) {
                const int i = g - g_lo, st = i % kStages;
                ok = tc::mbar_wait_warp(bar(kBarFull + st), (i / kStages) & 1, abort_flag, A.status);
                const uint32_t a = base + st * kStageBytes;
                for (int q = 0; ok && q < units; ++q) {          // unit number k goes to accumulator and team k mod 4
                    const int k = i * units + q, set = k & (kTeams - 1), n = min(kUnitCols, cols - q * kUnitCols);
                    ok = tc::mbar_wait_warp(bar(kBarSetFree + set), ((k / kTeams) & 1) ^ 1, abort_flag, A.status);
                    if (!ok) break;
                    tc::tc_fence_after();
                    const uint32_t idesc = tc::idesc_bf16(kTile, (uint32_t)((n + 15) & ~15));
                    const uint32_t a_lo = tc::desc_lo(a), b_lo = tc::desc_lo(bd + q * (kUnitCols * 128u));
                    if (tc::elect_one()) {
                        if (n > 0) {
#pragma unroll
                            for (int j = 0; j < 8; ++j)
                                tc::umma_bf16(tmem + kUnitCols * set, a_lo + (j >> 2) * (kPanel >> 4) + (j & 3) * 2, tc::kDescSw128Hi,
                                              b_lo + (j >> 2) * (b_panel >> 4) + (j & 3) * 2, tc::kDescSw128Hi, idesc, j > 0);
                        }
                        tc::umma_commit(bar(kBarAccFull + set));
                    }
                    __syncwarp();
                }
                if (ok && tc::elect_one()) tc::umma_commit(bar(kBarEmpty + st));
                __syncwarp();
            }
            if (ok && tc::elect_one()) tc::umma_commit(bar(kBarBEmpty + hp));
            __syncwarp();
        }
    } else {
        const int team = (warp - 2) >> 2, wq = warp & 3;
        const int hf = units == 2 ? team & 1 : 0;                    // which 128 columns this team works on
        const int row = 32 * wq + lane;                              // TMEM lane = token of the tile
        const uint32_t trow = tmem + kUnitCols * team + ((uint32_t)(32 * wq) << 16);
        const uint32_t wrow = base + kSmemStash + team * 4096 + row * 32;
        const uint32_t prow = base + kSmemStash + (team ^ 1) * 4096 + row * 32;      // the other unit's team
        bool ok = true;
        int hc = 0;
        // what a tile needs from global memory is fetched a tile of this team ahead, what a head needs a head ahead
        const int step = kTeams / units;                             // tiles between two of this team
        auto fetch_mod = [&](int g) -> int {
            const int uh = (int)A.by_nt.div(g), token = (g - uh * nt) * kTile + row;
            return g < g_hi && token < A.L ? A.modality[(int64_t)A.by_hkv.div(uh) * A.L + token] : 0;
        };
        auto fetch_rank = [&](int g) -> int {
            const int uh = (int)A.by_nt.div(g), token = (g - uh * nt) * kTile + row;
            return g < g_hi && token < A.L ? A.rank[(int64_t)uh * A.L + token] : -1;
        };
        int mod_next = fetch_mod(g_lo + team / units), rank_next = fetch_rank(g_lo + team / units);
        struct Head { int n_text, n_vis, strategy; };
        auto fetch_head = [&](int uh) -> Head {
            if (uh >= A.n_heads) return Head{0, 0, 0};
            return Head{A.cand_count[2 * uh], A.cand_count[2 * uh + 1], A.strategy[A.by_hkv.div(uh)]};
        };
        Head head_next = fetch_head((int)A.by_nt.div(g_lo));
        for (int g = g_lo; g < g_hi; ++hc) {
            const int uh = (int)A.by_nt.div(g), hp = hc % n_bbuf;
            const uint32_t md = base + kSmemMeta + hp * m_stride;
            const int n_text = head_next.n_text, n_vis = head_next.n_vis;
            const bool intra = head_next.strategy == 0;
            head_next = fetch_head(uh + 1);
            // blocks of 16 columns, text group [0, tb) and visual group [vb, ve), and this unit's share of them
            const int t0 = (n_text + 31) & ~31, c0 = hf * kUnitCols, blk0 = c0 >> 4;
            const int tb = min((n_text + 15) >> 4, blk0 + kUnitCols / 16);
            const int vb = max(t0 >> 4, blk0), ve = n_vis > 0 ? min((t0 + n_vis + 15) >> 4, blk0 + kUnitCols / 16) : 0;
            bool b_ready = false;
            for (const int end = min(g_hi, (uh + 1) * nt); g < end; ++g) {
                const int i = g - g_lo, t = g - uh * nt, st = i % kStages, k = i * units + hf;
                if ((k & (kTeams - 1)) != team) continue;            // (the parity of a tile's two units picks the pair of teams)
                const int token = t * kTile + row;
                const bool in_range = token < A.L;
                const int my_mod = mod_next, my_rank = rank_next;
                mod_next = fetch_mod(g + step);
                rank_next = fetch_rank(g + step);
                const bool want_text = in_range && (!intra || my_mod == 0), want_vis = in_range && (!intra || my_mod != 0);
                // the token's key row sits in the A stage (128-byte rows, 16-byte units XOR-swizzled by the row index)
                ok = ok && tc::mbar_wait_warp(bar(kBarFull + st), (i / kStages) & 1, abort_flag, A.status);
                const uint32_t a_row = base + st * kStageBytes + row * 128;
                float ssq = 0.f;
                if (ok) {
                    ssq = row_half_ssq(a_row + hf * kPanel, row);
                    if (units == 1) ssq += row_half_ssq(a_row + kPanel, row);
                }
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(bar(kBarEmpty + st));
                if (!b_ready) {                                      // scales and slots of this head have landed
                    ok = ok && tc::mbar_wait_warp(bar(kBarBFull + hp), (hc / n_bbuf) & 1, abort_flag, A.status);
                    b_ready = true;
                }
                ok = ok && tc::mbar_wait_warp(bar(kBarAccFull + team), (k / kTeams) & 1, abort_flag, A.status);
                tc::tc_fence_after();
                float best;
                int slot;
                match_unit(trow, md, slot_off, wrow, blk0, tb, vb, ve, want_text, want_vis, N, ok, A.status, best, slot, [&]() {
                    tc::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(bar(kBarSetFree + team));   // this warp has read the accumulator
                });
                if (units == 2) {
                    // the upper unit hands its result and its half of the norm to the lower one, which owns the row's output;
                    // (kept also after a wait that ran out, so that the partner warp is never left waiting)
                    if (hf == 1) tc::sts128(wrow, best, __int_as_float(slot), ssq, 0.f);
                    pair_sync(team >> 1, wq);
                    if (hf == 0) {
                        const float4 other = tc::lds128(prow);
                        if (match_better(other.x, __float_as_int(other.y), best, slot)) { best = other.x; slot = __float_as_int(other.y); }
                        ssq += other.z;
                    }
                    pair_sync(team >> 1, wq);                        // the stash may be overwritten again
                }
                if (hf == 0) {
                    if (in_range && my_rank >= 0 && ok && index_ok(my_rank, A.E, A.status)) {   // a non-pivot: report its match
                        float sim = 0.f;
                        if (slot >= 0 && ssq > 0.f) sim = best * rsqrtf(ssq);
                        A.match[(int64_t)uh * A.E + my_rank] = slot;
                        A.match_sim[(int64_t)uh * A.E + my_rank] = sim;
                        if (A.tokmap)                                // same entry as merge_map_kernel would write
                            A.tokmap[(int64_t)uh * A.L + token] = make_int2(slot, __float_as_int(A.merge_mode == 1 ? 1.f : __expf(sim - 1.f)));
                    } else if (in_range && ok && A.tokmap) {         // a pivot: its own slot with weight 1
                        A.tokmap[(int64_t)uh * A.L + token] = make_int2((-my_rank - 2) | (1 << 30), __float_as_int(1.f));
                    }
                }
            }
            // done with this head's scales and slots (a warp without a tile of the head waits for them all the same: it must
            // not arrive for a later head while the buffer still belongs to an earlier one)
            if (!b_ready) ok = ok && tc::mbar_wait_warp(bar(kBarBFull + hp), (hc / n_bbuf) & 1, abort_flag, A.status);
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(bar(kBarBEmpty + hp));
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == 1) tc::tmem_dealloc(tmem, 512);
}

}  // namespace mst
}  // namespace flowmm
