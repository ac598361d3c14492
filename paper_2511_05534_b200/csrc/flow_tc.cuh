// Full-prefill information flow (Eq. 6 and Eq. 7 over every query row) on the tensor cores, for bf16 inputs with
// head_dim 128: one launch for the whole call.
//
// An item is 256 consecutive query rows of one query head (two accumulator halves of 128) against the keys up to its last
// row.  Per row the softmax statistics are kept as in the first scoring pass, with the part of the exp-sum that falls on
// keys of the other modality beside it (a word of 32 keys is of one modality nearly always: then it costs one comparison;
// only mixed words go element by element).  At the end of an item the two column halves of a row meet in shared memory
// and a row's share cross / total is added up per warp, so nothing but four floats per half leaves the CTA.
//
// Bound by the epilogue: Hq L^2 / 2 exponentials per unit, a quarter of them as a polynomial on the FMA pipe, with four
// warps per scheduler to cover the latencies (half of the issue slots used; TMA and MMA alone take half the time).  A chunk
// becomes exponentials in place (28 x 28 heads x 2176 tokens 664 -> 641 us at the power
// cap; reading the next chunk ahead, which costs another 32 registers, gives that back).  The
// form before launched the statistics once per 128 query rows, with a join of all partial statistics after each: launches
// of a few hundred items in one to three uneven rounds, 1190 us for 28 layers of 28 heads and 2176 tokens against 595 us.
#pragma once
#include "common.cuh"
#include "score_tc.cuh"
#include "tc_stream.cuh"

namespace flowmm {

struct FlowTcArgs {
    const uint32_t *modbits;     // [U, mod_words] key modality, 32 keys per word
    float *parts;                // [8 n_rp][U * Hq]: shares of (256-row block, half, 32-row quarter)
    int *status;
    int Hq, G, Hkv, L, n_rp, n_heads, mod_words, n_items, n_rounds;
    int group_heads;             // query heads of a group of KV heads whose keys stay in L2 together
    FastDiv by_grid, by_group_items, by_group_heads, by_last_heads, by_g, by_hkv;   // exact divisions of item and head numbers
    float scale_log2;
};

struct FlowItem { int u, h, head, rp; };       // head: query head of the unit
// Item numbers run through the groups of KV heads; inside a group from the longest block of rows to the shortest.  A CTA takes
// one of every round of gridDim.x; every other round goes backwards, counted from the last one (which need not be full), so that
// no CTA gets the longest of each.  The call, us, all rounds forwards and so: 28 heads of 2176 tokens 38.9, 33.5; of 4096 93.0,
// 78.9; 112 of 900 35.5, 31.4; 64 of 1500 42.6, 38.1; 256 of 2000 171.9, 165.6; 784 of 2176 570.8, 563.4; up to one round the same.
__device__ __forceinline__ FlowItem flow_item(const FlowTcArgs &A, int item) {
    const int grid = (int)A.by_grid.d, round = (int)A.by_grid.div(item), first = round * grid;
    if ((A.n_rounds - round) % 2 == 0) item = first + grid - 1 - (item - first);
    const int grp = (int)A.by_group_items.div(item), in = item - grp * (int)A.by_group_items.d;
    const bool last = (grp + 1) * A.group_heads > A.n_heads;               // a last group of fewer heads
    const int back = (int)(last ? A.by_last_heads.div(in) : A.by_group_heads.div(in));
    const int hg = grp * A.group_heads + in - back * (int)(last ? A.by_last_heads.d : A.by_group_heads.d);
    FlowItem f;
    f.rp = A.n_rp - 1 - back;
    const int uh = (int)A.by_g.div(hg);
    f.u = (int)A.by_hkv.div(uh);
    f.h = uh - f.u * A.Hkv;
    f.head = hg - f.u * A.Hq;
    return f;
}

__global__ void __launch_bounds__(tcs::kThreads, 1)
flow_stats_tc_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map, const FlowTcArgs A) {
    using S = tcs::Big;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const S::Ctx c = S::setup(smem_raw, &q_map, &k_map, A.status, 0, 4);
    if (!c.ok) return;
    auto plan_of = [&](const FlowItem &f) {
        tcs::TilePlan p;
        const int lo = f.rp * tcs::kItemRows;
        p.a1 = lo; p.a2 = f.head; p.a3 = f.u;
        p.h1 = tcs::kRows; p.h2 = 0;
        p.n_halves = lo + tcs::kRows < A.L ? 2 : 1;
        p.b1 = 0; p.b2 = f.h; p.b3 = f.u; p.step1 = S::kCols; p.step2 = 0;
        p.cols_total = min(A.L, lo + tcs::kItemRows);
        p.cols_first = min(A.L, lo + tcs::kRows);            // the first half's rows end 128 keys earlier
        p.n_tiles = f.rp + 1;
        p.extra = nullptr;
        return p;
    };
    auto plan = [&](int item) { return plan_of(flow_item(A, item)); };
    if (c.warp == 0) {
        S::producer(c, &q_map, &k_map, A.n_items, tcs::kAHalf, S::kBStage, plan, A.status);
    } else if (c.warp == 1) {
        S::mma_issuer<true>(c, A.n_items, plan, A.status);
    } else {
        const int row = c.quarter * 32 + c.lane;                     // row of the half
        const uint32_t xch = c.epi_addr() + row * 16, pxch = c.partner_addr() + row * 16;   // hand-over slots of this row, the other column half's
        uint32_t turn = 0;                                           // two slots by turns: the next meeting keeps the upper half from one still being read
        int k = 0;
        bool ok = true;
        FlowItem f_next;
        uint32_t flip_next = 0;                                      // modality word of this warp's 32 rows
        auto fetch_next = [&](int item) {
            if (item >= A.n_items) return;
            f_next = flow_item(A, item);
            flip_next = A.modbits[(int64_t)f_next.u * A.mod_words + f_next.rp * (tcs::kItemRows / 32) + c.group * (tcs::kRows / 32) + c.quarter];
        };
        fetch_next(blockIdx.x);
        for (int item = blockIdx.x; ok && item < A.n_items; item += gridDim.x) {
            const FlowItem f = f_next;
            const tcs::TilePlan p = plan_of(f);
            const int lo = f.rp * tcs::kItemRows;
            const uint32_t *bits = A.modbits + (int64_t)f.u * A.mod_words;
            float m = kNegBig, l = 0.f, lc = 0.f;
            // all ones for a row of a visual token, whose other modality is the complement; fetched an item ahead
            const uint32_t flip = ((flip_next >> c.lane) & 1u) ? 0xFFFFFFFFu : 0u;
            fetch_next(item + gridDim.x);
            const bool active = c.group < p.n_halves;
            // this warp's rows r0 .. r0 + 31 see the keys up to themselves: chunks past r0 + 31 are left out and only the one
            // on the diagonal is masked
            const int r0 = lo + c.group * tcs::kRows + c.quarter * 32, half_end = c.group == 0 ? p.cols_first : p.cols_total;
            for (int t = 0; ok && active && t < p.n_tiles; ++t) {
                const int kb = t * S::kCols;
                if (!S::takes_part(c, min(S::kCols, half_end - kb))) continue;
                ok = S::quad_wait(c, k++, A.status);
                if (!ok) continue;
                const int ncols = min(S::kCols, min(r0 + 32, A.L) - kb);
                S::for_each_chunk(c, (ncols + 31) >> 5, [&](int ch, uint32_t (&acc)[32]) {
                    const int k0 = kb + ch * 32;
                    const uint32_t word = bits[k0 >> 5];
                    uint32_t other = word ^ flip;                        // keys of the other modality than the row's token
                    float mx, add, addc;
                    // Where a few keys can make up a share - on the diagonal and in words of both modalities - all exponentials are
                    // the exp2 unit's: with the polynomial in a quarter of them a share was off by up to 7e-7 instead of 2e-7.
                    if (k0 < r0 && (word == 0u || word == 0xFFFFFFFFu)) {
                        mx = fmaxf(max32(acc) * A.scale_log2, m);
                        exp2_32(acc, A.scale_log2, mx);
                        add = sum32(acc);
                        addc = other != 0u ? add : 0.f;
                    } else {
                        if (k0 >= r0) {                              // the chunk on the diagonal: exp2 of what is masked gives 0
                            other &= 0xFFFFFFFFu >> (31 - c.lane);
#pragma unroll
                            for (int j = 0; j < 32; ++j) acc[j] = j <= c.lane ? acc[j] : __float_as_uint(-INFINITY);
                        }
                        mx = fmaxf(max32(acc) * A.scale_log2, m);
                        exp2_32_exact(acc, A.scale_log2, mx);
                        add = sum32(acc);
                        float x[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int j = 0; j < 32; ++j) x[j & 3] += ((other >> j) & 1u) ? __uint_as_float(acc[j]) : 0.f;
                        addc = (x[0] + x[1]) + (x[2] + x[3]);
                    }
                    const float carry = tc::ex2(m - mx);
                    l = l * carry + add;
                    lc = lc * carry + addc;
                    m = mx;
                }, [&]() { S::quad_release(c); });
            }
            // The two column halves of every row meet.  (After a wait that ran out the meeting is still kept: the vote ends the
            // loop for both warps.)
            if (c.colhalf == 1) tc::sts128(xch + turn, m, l, lc, 0.f);
            ok = !S::pair_meet(c, !ok);
            if (c.colhalf == 0 && ok) {
                const float4 o = tc::lds128(pxch + turn);
                const float mx = fmaxf(m, o.x), wa = tc::ex2(m - mx), wb = tc::ex2(o.x - mx);
                const float z = l * wa + o.y * wb, zc = lc * wa + o.z * wb;
                const float share = warp_sum(active && r0 + c.lane < A.L && z > 0.f ? zc / z : 0.f);   // (a half without rows: 0)
                if (c.lane == 0)
                    A.parts[((int64_t)(f.rp * 2 + c.group) * 4 + c.quarter) * (int64_t)A.n_heads + (int64_t)f.u * A.Hq + f.head] = share;
            }
            turn ^= tcs::kRows * 16;
        }
    }
    S::teardown(c);
}

}  // namespace flowmm
