// Window scoring (Eq. 8 with the softmax of Eq. 4, and the masses of Eq. 7) in one pass over K, for
// short contexts with few proxy rows per KV head (bf16, head_dim 128).
//
// The two-pass kernels of score_tc.cuh read K twice because a column sum needs every row's final
// normaliser first.  When all logits of a head fit in half of TMEM - ceil(L / 128) tiles x (G W) columns
// <= 256 - a CTA computes S_t = K_t Q^T once per 128-key tile (tcgen05.mma, keys as M, proxy rows as N),
// keeps every tile of the head in TMEM, and a team of eight warps sweeps them three times:
//   A  per proxy row the maximum over all keys (running while the K tiles still stream),
//   B  per proxy row the sum of exponentials, in total and over the keys of the other modality (Eq. 7),
//   C  per key the sum over proxy rows of exp / row sum: the importance (group mean over the G heads); the exponentials are those of
//      sweep B, which leaves them in TMEM (1024 heads of 640 tokens 132 -> 122 us for the whole call, 32 of 640 24.7 -> 23.7).
// Lanes are keys, so the per-row reductions of A and B cross lanes (shuffles, then shared memory across
// the warps) once per head; everything else is per thread.  K is read from HBM exactly once.
// CTAs are persistent (one per SM) and take (unit, KV head) items in turn.  Warp 0 streams Q and the
// K tiles through a five-stage TMA ring and runs ahead of the arithmetic, warp 1 issues the MMAs of
// item i into TMEM half i mod 2 (both run whole and elect a thread at each instruction), and two teams of eight warps (two warps per 32 TMEM lanes, each with
// half of the proxy rows; their partial importances meet in shared memory) take the items alternately, so
// one head is swept while the next one streams in.
#pragma once
#include "common.cuh"
#include "decode_tc.cuh"
#include "tc_common.cuh"

namespace flowmm {
namespace sft {

constexpr int kTile = 128;
constexpr int kStages = 5;
constexpr int kRows = 32;                       // proxy rows per KV head (G W) this kernel is built for
constexpr int kMaxTiles = 8;                    // 8 x 32 columns = one half of TMEM
constexpr int kTeam = 256;                      // threads of a sweep team
constexpr int kThreads = 64 + 2 * kTeam;
constexpr uint32_t kStageBytes = kTile * 128 * 2, kPanel = kStageBytes / 2;
constexpr uint32_t kQBytes = kRows * 256;                          // Q operand of one head: two panels of 32 rows
constexpr uint32_t kSmemQ = kStages * kStageBytes;                 // two Q operands
constexpr uint32_t kSmemRed = kSmemQ + 2 * kQBytes;                // per team: float [3][4][kRows], int [kRows] mask limits, float [2][kRows] row maxima and 1 / row sums
constexpr uint32_t kRedBytes = 15 * kRows * 4;
constexpr uint32_t kSmemImp = kSmemRed + 2 * kRedBytes;            // per team: float [kMaxTiles][128] partial importances
constexpr uint32_t kImpBytes = kMaxTiles * kTile * 4;
constexpr uint32_t kSmemBar = kSmemImp + 2 * kImpBytes;
constexpr int kBarFull = 0, kBarEmpty = kStages, kBarQFull = 2 * kStages, kBarQEmpty = kBarQFull + 2,
              kBarSetFree = kBarQEmpty + 2 /* 256 arrivals */, kBarS = kBarSetFree + 2 /* [2][kMaxTiles] */,
              kNumBars = kBarS + 2 * kMaxTiles;
constexpr uint32_t kSmemBytes = kSmemBar + 8 * kNumBars + 16;

struct Args {
    const uint8_t *modality;    // [U, L]
    float *importance;          // [UH, L]
    float *cross_mass;          // [U, Hq]
    int *status;
    int Hq, Hkv, G, W, L, n_items;
    float scale_log2;
};

// Reduction of 16 values per lane across the 32 lanes of a warp with 16 shuffles instead of 80: every step a lane
// hands half of its values to the partner that keeps them.  On return v[0] holds the total of value
// number (lane >> 1) & 15 (in both lanes of the pair).
template <class Op>
__device__ __forceinline__ void warp_reduce16(float (&v)[16], Op op) {
#pragma unroll
    for (int n = 8, m = 16; n >= 1; n >>= 1, m >>= 1) {
        const bool upper = (threadIdx.x & m) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float send = upper ? v[i] : v[i + n], keep = upper ? v[i + n] : v[i];
            v[i] = op(keep, __shfl_xor_sync(0xFFFFFFFFu, send, m));
        }
    }
    v[0] = op(v[0], __shfl_xor_sync(0xFFFFFFFFu, v[0], 1));
}

__device__ __forceinline__ void team_sync(int team) { asm volatile("bar.sync %0, 256;" ::"r"(1 + team) : "memory"); }

__global__ void __launch_bounds__(kThreads, 1)
score_fused_tc_kernel(const __grid_constant__ CUtensorMap qmap, const __grid_constant__ CUtensorMap kmap, const Args A) {
    constexpr int GW = kRows, HC = GW / 2;
    extern __shared__ __align__(1024) uint8_t sft_smem[];
    const uint32_t base = tc::smem_u32(sft_smem), bars = base + kSmemBar;
    const int warp = tc::warp_number(), lane = threadIdx.x & 31;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(sft_smem + kSmemBar + 8 * kNumBars + 4);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(sft_smem + kSmemBar + 8 * kNumBars);
    if ((base & 1023u) != 0) {
        predecessor_done();
        if (threadIdx.x == 0) atomicCAS(A.status, 0, 6);
        return;
    }
    auto bar = [&](int i) { return bars + 8u * i; };
    if (threadIdx.x == 0) {
        for (int i = 0; i < kNumBars; ++i) tc::mbar_init(bar(i), (i == kBarSetFree || i == kBarSetFree + 1) ? kTeam : 1);
        *abort_flag = 0;
        tc::mbar_init_fence();
        tc::tma_prefetch_desc(&qmap);
        tc::tma_prefetch_desc(&kmap);
    }
    if (warp == 1) tc::tmem_alloc(tc::smem_u32(tmem_slot), 512);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    predecessor_done();
    const int nt = (A.L + kTile - 1) / kTile;

    if (warp == 0) {
        bool ok = true;
        int i = 0, it = 0;
        for (int item = blockIdx.x; ok && item < A.n_items; item += gridDim.x, ++it) {
            const int u = item / A.Hkv, h = item % A.Hkv, set = it & 1;
            ok = tc::mbar_wait_warp(bar(kBarQEmpty + set), ((it >> 1) & 1) ^ 1, abort_flag, A.status);
            if (!ok) break;
            const uint32_t qd = base + kSmemQ + set * kQBytes;
            if (tc::elect_one()) {
                tc::mbar_expect_tx(bar(kBarQFull + set), kQBytes);
                tc::tma_load_4d(qd, &qmap, bar(kBarQFull + set), 0, 0, h * A.G, u);
                tc::tma_load_4d(qd + kQBytes / 2, &qmap, bar(kBarQFull + set), 64, 0, h * A.G, u);
            }
            __syncwarp();
            for (int t = 0; ok && t < nt; ++t, ++i) {
                const int st = i % kStages;
                ok = tc::mbar_wait_warp(bar(kBarEmpty + st), ((i / kStages) & 1) ^ 1, abort_flag, A.status);
                if (!ok) break;
                const uint32_t dst = base + st * kStageBytes;
                if (tc::elect_one()) {
                    tc::mbar_expect_tx(bar(kBarFull + st), kStageBytes);
                    tc::tma_load_4d(dst, &kmap, bar(kBarFull + st), 0, t * kTile, h, u);
                    tc::tma_load_4d(dst + kPanel, &kmap, bar(kBarFull + st), 64, t * kTile, h, u);
                }
                __syncwarp();
            }
        }
        if (!ok) {       // winding down after a timeout: give copies already issued a moment to land
            for (int b = 0; b < kStages; ++b)
                for (int s = 0; s < (1 << 16) && !tc::mbar_try_wait(bar(kBarFull + b), 0) && !tc::mbar_try_wait(bar(kBarFull + b), 1); ++s) {}
            for (int b = 0; b < 2; ++b)
                for (int s = 0; s < (1 << 16) && !tc::mbar_try_wait(bar(kBarQFull + b), 0) && !tc::mbar_try_wait(bar(kBarQFull + b), 1); ++s) {}
        }
    } else if (warp == 1) {
        constexpr uint32_t idesc = tc::idesc_bf16(kTile, GW);
        bool ok = true;
        int i = 0, it = 0;
        for (int item = blockIdx.x; ok && item < A.n_items; item += gridDim.x, ++it) {
            const int set = it & 1, use = it >> 1;
            ok = tc::mbar_wait_warp(bar(kBarQFull + set), use & 1, abort_flag, A.status) &&
                 tc::mbar_wait_warp(bar(kBarSetFree + set), (use & 1) ^ 1, abort_flag, A.status);   // the half's previous head is swept
            tc::tc_fence_after();
            const uint32_t qd = base + kSmemQ + set * kQBytes;
            for (int t = 0; ok && t < nt; ++t, ++i) {
                const int st = i % kStages;
                ok = tc::mbar_wait_warp(bar(kBarFull + st), (i / kStages) & 1, abort_flag, A.status);
                if (!ok) break;
                tc::tc_fence_after();
                const uint32_t a = base + st * kStageBytes;
                const uint32_t a_lo = tc::desc_lo(a), b_lo = tc::desc_lo(qd), d = tmem + 256 * set + GW * t;
                if (tc::elect_one()) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        tc::umma_bf16(d, a_lo + (j >> 2) * (kPanel >> 4) + (j & 3) * 2, tc::kDescSw128Hi,
                                      b_lo + (j >> 2) * (kQBytes / 32) + (j & 3) * 2, tc::kDescSw128Hi, idesc, j > 0);
                    tc::umma_commit(bar(kBarEmpty + st));
                    tc::umma_commit(bar(kBarS + set * kMaxTiles + t));
                }
                __syncwarp();
            }
            if (ok && tc::elect_one()) tc::umma_commit(bar(kBarQEmpty + set));
            __syncwarp();
        }
    } else {
        // two sweep teams of eight warps: two warps per 32 TMEM lanes, each with half of the proxy rows (HC columns)
        const int team = (warp - 2) >> 3, tw = (warp - 2) & 7;
        const int e = (threadIdx.x - 64) & (kTeam - 1);
        const int wq = warp & 3, half = tw >> 2, cb = half * HC;     // cb: first proxy row of this thread
        const int row = 32 * wq + lane;                              // TMEM lane: key of a tile
        const uint32_t trow = tmem + ((uint32_t)(32 * wq) << 16) + 256 * team + cb;
        float *red = reinterpret_cast<float *>(sft_smem + kSmemRed + team * kRedBytes);    // [3][4][kRows]
        float *impx = reinterpret_cast<float *>(sft_smem + kSmemImp + team * kImpBytes);   // [nt][128]
        int *lim = reinterpret_cast<int *>(red + 12 * kRows);
        float *row_max = red + 13 * kRows, *row_inv = red + 14 * kRows;
        const int first_proxy = A.L - A.W;
        // a (key, proxy row c) pair counts if key <= lim[c] = first_proxy + c % W (which also keeps key < L)
        if (e < GW) lim[e] = first_proxy + e % A.W;
        const int n_plain = min(nt, (first_proxy + 1) / kTile);      // leading tiles in which no pair is masked
        auto load = [&](int t, uint32_t (&r)[HC]) {
            tc::tmem_ld16(trow + GW * t, r);
            tc::tmem_ld_wait(r);
        };
        bool ok = true;
        int it = team;
        uint8_t proxy_next = 0, key_next[kMaxTiles];
        auto fetch_modality = [&](int item) {                        // (independent loads: nothing waits in between)
            const uint8_t *mod = A.modality + (int64_t)(item / A.Hkv) * A.L;
            const bool on = item < A.n_items;
            proxy_next = on && lane < HC ? mod[first_proxy + (cb + lane) % A.W] : (uint8_t)0;
#pragma unroll
            for (int t = 0; t < kMaxTiles; ++t) key_next[t] = on && t * kTile + row < A.L ? mod[t * kTile + row] : (uint8_t)0;
        };
        fetch_modality(blockIdx.x + team * gridDim.x);
        for (int item = blockIdx.x + team * gridDim.x; item < A.n_items; item += 2 * gridDim.x, it += 2) {
            const int uh = item, u = item / A.Hkv, h = item % A.Hkv, use = it >> 1;
            // modalities, fetched an item ahead: `qvis` bit q: this thread's proxy row cb + q = g W + a belongs to a visual token
            // (token first_proxy + a); `vis_bits` bit t: its key of tile t is one
            const unsigned qvis = __ballot_sync(0xFFFFFFFFu, proxy_next != 0);
            unsigned vis_bits = 0;
#pragma unroll
            for (int t = 0; t < kMaxTiles; ++t) vis_bits |= key_next[t] != 0 ? 1u << t : 0u;
            fetch_modality(item + 2 * gridDim.x);
            team_sync(team);                                         // lim is written; the previous item's scratch is free

            float mx[HC];
#pragma unroll
            for (int q = 0; q < HC; ++q) mx[q] = kNegBig;
            for (int t = 0; t < nt; ++t) {                           // sweep A, under the K stream
                ok = ok && tc::mbar_wait_warp(bar(kBarS + team * kMaxTiles + t), use & 1, abort_flag, A.status);
                if (!ok) continue;
                tc::tc_fence_after();
                const int key = t * kTile + row;
                uint32_t r[HC];
                load(t, r);
                if (t < n_plain) {
#pragma unroll
                    for (int q = 0; q < HC; ++q) mx[q] = fmaxf(mx[q], __uint_as_float(r[q]));
                } else {
#pragma unroll
                    for (int q = 0; q < HC; ++q)
                        if (key <= lim[cb + q]) mx[q] = fmaxf(mx[q], __uint_as_float(r[q]));
                }
            }
            warp_reduce16(mx, [](float a, float b) { return fmaxf(a, b); });
            if (!(lane & 1)) red[wq * kRows + cb + (lane >> 1)] = mx[0];
            team_sync(team);
            if (tw == 0)                                             // the row's maximum in the log2 domain
                row_max[lane] = A.scale_log2 * fmaxf(fmaxf(red[lane], red[kRows + lane]), fmaxf(red[2 * kRows + lane], red[3 * kRows + lane]));
            team_sync(team);
            auto load_rows = [&](const float *from, float (&v)[HC]) {
#pragma unroll
                for (int q = 0; q < HC; q += 4) {
                    const float4 f = *reinterpret_cast<const float4 *>(from + cb + q);
                    v[q] = f.x; v[q + 1] = f.y; v[q + 2] = f.z; v[q + 3] = f.w;
                }
            };
            load_rows(row_max, mx);

            float lt[HC], lc[HC];                                    // sweep B: row sums, total and other-modality keys
#pragma unroll
            for (int q = 0; q < HC; ++q) { lt[q] = 0.f; lc[q] = 0.f; }
            const bool one_kind = qvis == 0u || qvis == (1u << HC) - 1u;   // this warp's proxy rows are of one modality
            for (int t = 0; t < nt; ++t) {
                const unsigned oth = ((vis_bits >> t) & 1u) ? ~qvis : qvis;   // proxy rows of the other modality than this key's
                uint32_t r[HC];
                load(t, r);
                float p[HC];                                         // (multiply-adds as packed pairs: half the issue slots)
#pragma unroll
                for (int q = 0; q < HC; q += 2) {
                    const float2 x = tc::ffma2(make_float2(__uint_as_float(r[q]), __uint_as_float(r[q + 1])), make_float2(A.scale_log2, A.scale_log2), make_float2(-mx[q], -mx[q + 1]));
                    p[q] = tc::ex2(x.x); p[q + 1] = tc::ex2(x.y);
                }
                if (t >= n_plain) {
                    const int key = t * kTile + row;
#pragma unroll
                    for (int q = 0; q < HC; ++q) p[q] = key > lim[cb + q] ? 0.f : p[q];
                }
                tc::tmem_st16(trow + GW * t, p);                     // in the logits' place, for sweep C
                if (one_kind) {
                    const float o = (oth & 1u) ? 1.f : 0.f;
#pragma unroll
                    for (int q = 0; q < HC; q += 2) {
                        const float2 p2 = make_float2(p[q], p[q + 1]);
                        const float2 t2 = tc::fadd2(make_float2(lt[q], lt[q + 1]), p2), c2 = tc::ffma2(make_float2(o, o), p2, make_float2(lc[q], lc[q + 1]));
                        lt[q] = t2.x; lt[q + 1] = t2.y; lc[q] = c2.x; lc[q + 1] = c2.y;
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < HC; ++q) { lt[q] += p[q]; lc[q] += ((oth >> q) & 1u) ? p[q] : 0.f; }
                }
            }
            tc::tmem_st_wait();
            warp_reduce16(lt, [](float a, float b) { return a + b; });
            warp_reduce16(lc, [](float a, float b) { return a + b; });
            if (!(lane & 1)) {
                red[(4 + wq) * kRows + cb + (lane >> 1)] = lt[0];
                red[(8 + wq) * kRows + cb + (lane >> 1)] = lc[0];
            }
            team_sync(team);
            if (tw == 0) {                                           // Eq. 7: a lane per proxy row, summed per query head as a tree
                const float tot = red[4 * kRows + lane] + red[5 * kRows + lane] + red[6 * kRows + lane] + red[7 * kRows + lane];
                const float cr = red[8 * kRows + lane] + red[9 * kRows + lane] + red[10 * kRows + lane] + red[11 * kRows + lane];
                row_inv[lane] = 1.f / tot;
                float share = cr / tot;
                for (int o = 1; o < A.W; o <<= 1) {                  // (W divides 32: lanes g W .. g W + W - 1 are head g's)
                    const float other = __shfl_down_sync(0xFFFFFFFFu, share, o);
                    if ((lane & (2 * o - 1)) == 0) share += other;
                }
                if (ok && lane % A.W == 0) A.cross_mass[(int64_t)u * A.Hq + h * A.G + lane / A.W] = share;
            }
            team_sync(team);
            load_rows(row_inv, lt);
            float imp[kMaxTiles];                                    // sweep C: this thread's share of every key's importance
#pragma unroll
            for (int t = 0; t < kMaxTiles; ++t) {
                imp[t] = 0.f;
                if (t < nt) {
                    uint32_t r[HC];
                    load(t, r);
                    float2 s2 = make_float2(0.f, 0.f);
#pragma unroll
                    for (int q = 0; q < HC; q += 2) s2 = tc::ffma2(make_float2(__uint_as_float(r[q]), __uint_as_float(r[q + 1])), make_float2(lt[q], lt[q + 1]), s2);
                    imp[t] = s2.x + s2.y;
                    if (half == 1) impx[t * kTile + row] = imp[t];
                }
            }
            tc::tc_fence_before();
            tc::mbar_arrive(bar(kBarSetFree + team));               // this thread has read the half for the last time
            team_sync(team);
            if (half == 0 && ok) {
                const float inv_g = 1.f / (float)A.G;
#pragma unroll
                for (int t = 0; t < kMaxTiles; ++t) {
                    const int key = t * kTile + row;
                    if (t < nt && key < A.L) A.importance[(int64_t)uh * A.L + key] = (imp[t] + impx[t * kTile + row]) * inv_g;
                }
            }
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == 1) tc::tmem_dealloc(tmem, 512);
}

}  // namespace sft
}  // namespace flowmm
