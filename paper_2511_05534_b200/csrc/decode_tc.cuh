// Decode-step attention over a KV cache (Eq. 4) on the tensor cores, for bf16 caches with head_dim 128.
//
// One CTA takes a range of up to 15 tiles of 128 keys of one (unit, KV head) and all query heads of
// the group (up to 8, zero-padded to the 16 rows of the narrow operand).  Both contractions run with the keys on the wide side, so the
// tiny query side costs nothing and every K and V row is read from HBM exactly once:
//   phase 1   S_t[key, head] = K_t Q^T        tcgen05.mma M = 128 keys, N = 16, contraction over head_dim;
//             every tile's logits stay in TMEM (16 columns per tile)
//   reduce    the exact per-head maximum over the CTA's range, from TMEM
//   phase 2   P_t = 2^(c S_t - max) into shared memory as two bf16 rows per head (the rounded weight and
//             the rounding remainder), then O[dim, row] += V_t^T P_t^T: M = 128 dims, N = 16 = 8 heads x 2,
//             contraction over the tile's keys; a head's output is the sum of its two columns.  The V tile is the same swizzled
//             shared-memory tile a K tile is, read the other way round (MN-major operand), so V needs no
//             transposition.  O never needs rescaling because the maximum is already final.
// A head with one range is normalised and written at once.  Two to eight ranges are a cluster: every CTA leaves its
// unnormalised output, maximum and sum of weights in its shared memory, and after a cluster barrier the CTAs join a share
// of the heads each.  With more ranges the CTA writes its record to global memory and decode_combine_kernel joins them, a
// block per query head.  (One layer of 4 KV heads of 218 keys, as two ranges 12.4 us when the range that finished last
// joined them, found by tickets that a memset had to clear first, 6.2 us as clusters of two, and as long as one range.)
// Roles: warp 0 streams K tiles then V tiles through a three-stage TMA ring, warp 1 issues
// the MMAs (both run whole and elect a thread at each instruction), warps 2-5 (one thread per key of a tile / per output dim) do the softmax and the output.
// Two CTAs fit an SM (256 TMEM columns, about 109 KB of shared memory each), so one streams while the
// other is between its phases.  Every wait is bounded.
#pragma once
#include "common.cuh"
#include "status_word.cuh"
#include "tc_common.cuh"

namespace flowmm {
namespace dtc {

constexpr int kTile = 128;                  // keys per tile
constexpr int kStages = 3;
constexpr int kHeads = 16;                  // N of both contractions
constexpr int kMaxHeads = 8;                // query heads per KV head this kernel serves
constexpr int kMaxRanges = 8;                // of a head that a cluster joins
constexpr int kMaxTiles = 15;               // 16 TMEM columns for O + 16 per score tile = 256
constexpr int kTmemCols = 256;
constexpr int kThreads = 192;
constexpr uint32_t kStageBytes = kTile * 128 * 2;            // both 64-element panels of a 128-row tile
constexpr uint32_t kPanel = kStageBytes / 2;
constexpr uint32_t kSmallPanel = kHeads * 128;               // 16 rows x 128 bytes
constexpr uint32_t kSmemQ = kStages * kStageBytes;           // Q operand: two panels of 16 rows
constexpr uint32_t kSmemP = kSmemQ + 2 * kSmallPanel;        // two P buffers of the same shape
constexpr uint32_t kSmemRed = kSmemP + 4 * kSmallPanel;      // float [4 warps][8 heads]
constexpr uint32_t kSmemBar = kSmemRed + 256;
constexpr int kBarFull = 0, kBarEmpty = kStages, kBarQ = 2 * kStages, kBarS = kBarQ + 1 /* one per score tile */,
              kBarPFull = kBarS + kMaxTiles, kBarPEmpty = kBarPFull + 2, kBarO = kBarPEmpty + 2, kNumBars = kBarO + 1;
constexpr uint32_t kSmemBytes = kSmemBar + 8 * kNumBars + 16;   // (+ TMEM address, abort flag, status)

struct Args {
    const __nv_bfloat16 *q;     // [U, Hq, 128] dense
    float *part;                // [UH, n_split, G, 130]: unnormalised output, maximum (log2 domain), sum of weights
    float *out;                 // [U, Hq, 128]
    int *status;                // the call's status word (status_word.cuh)
    uint32_t call;
    int Hq, Hkv, G, N, n_split, tiles_per_split;
    float scale_log2;
    int clustered;              // the ranges of a head are one cluster
};

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }
__device__ __forceinline__ void sts128u(uint32_t addr, uint4 v) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void sts16(uint32_t addr, unsigned short v) {
    asm volatile("st.shared.b16 [%0], %1;" ::"r"(addr), "h"(v) : "memory");
}
// The swizzled 128-row tile read as an MN-major operand: a 128-byte row holds 64 consecutive M
// elements of one K index, eight K indices make a 1024-byte group (the stride of the upper descriptor word), the second
// 64 M elements live `kPanel` bytes further on (the leading offset, bits 16 up of the lower word).  The 16 K indices (rows)
// of the next instruction add 2048 bytes.
constexpr uint32_t kDescMnLead = (kPanel >> 4) << 16;
constexpr uint32_t kIdescQK = tc::idesc_bf16(kTile, kHeads);
constexpr uint32_t kIdescPV = tc::idesc_bf16(128, kHeads) | (1u << 15);   // A operand MN-major

__global__ void __launch_bounds__(kThreads, 2)
decode_tc_kernel(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap, const Args A) {
    extern __shared__ __align__(1024) uint8_t dtc_smem[];
    const uint32_t base = tc::smem_u32(dtc_smem), bars = base + kSmemBar;
    const int warp = tc::warp_number(), lane = threadIdx.x & 31;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(dtc_smem + kSmemBar + 8 * kNumBars + 4);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(dtc_smem + kSmemBar + 8 * kNumBars);
    // what the waits report, until the CTA hands it to the call's status word
    int *cta_status = reinterpret_cast<int *>(dtc_smem + kSmemBar + 8 * kNumBars + 8);
    if ((base & 1023u) != 0) {                      // the swizzled tiles need a 1024-byte aligned base
        predecessor_done();
        if (threadIdx.x == 0) status_write(A.status, A.call, 6);
        return;
    }
    auto bar = [&](int i) { return bars + 8u * i; };
    if (threadIdx.x == 0) {
        for (int i = 0; i < kNumBars; ++i)
            tc::mbar_init(bar(i), (i == kBarQ || i == kBarPFull || i == kBarPFull + 1) ? 128 : 1);
        *abort_flag = 0;
        *cta_status = 0;
        tc::mbar_init_fence();
        tc::tma_prefetch_desc(&kmap);
        tc::tma_prefetch_desc(&vmap);
    }
    if (warp == 1) tc::tmem_alloc(tc::smem_u32(tmem_slot), kTmemCols);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    predecessor_done();
    if (A.n_split == 1 || A.clustered) successor_may_start();        // (not the small blocks that join many ranges)

    const int uh = blockIdx.x, u = uh / A.Hkv, h = uh % A.Hkv, split = blockIdx.y;
    const int tiles_total = (A.N + kTile - 1) / kTile;
    const int t0 = split * A.tiles_per_split, nt = min(A.tiles_per_split, tiles_total - t0);
    const int key0 = t0 * kTile;

    if (warp == 0) {
        bool ok = true;
        int st = 0, phase = 0;
        for (int i = 0; ok && i < 2 * nt; ++i) {                     // the K tiles, then the V tiles
            ok = tc::mbar_wait_warp(bar(kBarEmpty + st), phase ^ 1, abort_flag, cta_status);
            if (!ok) break;
            const CUtensorMap *m = i < nt ? &kmap : &vmap;
            const int row = key0 + (i < nt ? i : i - nt) * kTile;
            const uint32_t dst = base + st * kStageBytes;
            if (tc::elect_one()) {
                tc::mbar_expect_tx(bar(kBarFull + st), kStageBytes);
                tc::tma_load_4d(dst, m, bar(kBarFull + st), 0, row, h, u);
                tc::tma_load_4d(dst + kPanel, m, bar(kBarFull + st), 64, row, h, u);
            }
            __syncwarp();
            if (++st == kStages) { st = 0; phase ^= 1; }
        }
        if (!ok)         // winding down after a timeout: give copies already issued a moment to land
            for (int i = 0; i < kStages; ++i)
                for (int s = 0; s < (1 << 16) && !tc::mbar_try_wait(bar(kBarFull + i), 0) && !tc::mbar_try_wait(bar(kBarFull + i), 1); ++s) {}
        // the call's status word starts at zero; here, because this warp has nothing left to do (other CTAs may have reported already)
        if (blockIdx.x == 0 && blockIdx.y == 0 && tc::elect_one()) status_write(A.status, A.call, 0);
    } else if (warp == 1) {
        const uint32_t q_lo = tc::desc_lo(base + kSmemQ);
        bool ok = tc::mbar_wait_warp(bar(kBarQ), 0, abort_flag, cta_status);
        int st = 0, phase = 0;
        auto next = [&]() { if (++st == kStages) { st = 0; phase ^= 1; } };
        for (int t = 0; ok && t < nt; ++t, next()) {
            ok = tc::mbar_wait_warp(bar(kBarFull + st), phase, abort_flag, cta_status);
            if (!ok) break;
            tc::tc_fence_after();
            const uint32_t a_lo = tc::desc_lo(base + st * kStageBytes);
            if (tc::elect_one()) {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    tc::umma_bf16(tmem + kHeads + kHeads * t, a_lo + (j >> 2) * (kPanel >> 4) + (j & 3) * 2, tc::kDescSw128Hi,
                                  q_lo + (j >> 2) * (kSmallPanel >> 4) + (j & 3) * 2, tc::kDescSw128Hi, kIdescQK, j > 0);
                tc::umma_commit(bar(kBarEmpty + st));
                tc::umma_commit(bar(kBarS + t));
            }
            __syncwarp();
        }
        for (int t = 0; ok && t < nt; ++t, next()) {
            const int pb = t & 1;
            ok = tc::mbar_wait_warp(bar(kBarFull + st), phase, abort_flag, cta_status) &&
                 tc::mbar_wait_warp(bar(kBarPFull + pb), (t >> 1) & 1, abort_flag, cta_status);
            if (!ok) break;
            tc::tc_fence_after();
            const uint32_t a_lo = tc::desc_lo(base + st * kStageBytes) | kDescMnLead, p_lo = tc::desc_lo(base + kSmemP + pb * 2 * kSmallPanel);
            if (tc::elect_one()) {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    tc::umma_bf16(tmem, a_lo + j * 128, tc::kDescSw128Hi, p_lo + (j >> 2) * (kSmallPanel >> 4) + (j & 3) * 2, tc::kDescSw128Hi,
                                  kIdescPV, (t | j) != 0);
                tc::umma_commit(bar(kBarEmpty + st));
                tc::umma_commit(bar(kBarPEmpty + pb));
            }
            __syncwarp();
        }
        if (ok && tc::elect_one()) tc::umma_commit(bar(kBarO));
        __syncwarp();
    } else {
        const int e = threadIdx.x - 64;                              // 0 .. 127
        const int row = 32 * (warp & 3) + lane;                      // TMEM lane this thread reads: key of a tile / output dim
        const uint32_t trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
        const int G = A.G;
        // the Q operand (rows = heads, zero beyond G) and zeroed P buffers
        for (int c = e; c < 256; c += 128) {
            const int g = c >> 4, cc = c & 15;
            uint4 val = make_uint4(0, 0, 0, 0);
            if (g < G) val = *reinterpret_cast<const uint4 *>(A.q + ((int64_t)u * A.Hq + h * G + g) * 128 + cc * 8);
            sts128u(base + kSmemQ + (cc >> 3) * kSmallPanel + g * 128 + (((cc & 7) ^ (g & 7)) << 4), val);
        }
        for (int c = e; c < 512; c += 128) sts128u(base + kSmemP + c * 16, make_uint4(0, 0, 0, 0));
        fence_proxy_async();
        tc::mbar_arrive(bar(kBarQ));

        bool ok = true;
        float mx[kMaxHeads];
#pragma unroll
        for (int g = 0; g < kMaxHeads; ++g) mx[g] = kNegBig;
        for (int t = 0; t < nt; ++t) {                               // running maxima while the K tiles stream
            ok = ok && tc::mbar_wait_warp(bar(kBarS + t), 0, abort_flag, cta_status);
            if (!ok) continue;
            tc::tc_fence_after();
            uint32_t r[16];
            tc::tmem_ld16(trow + kHeads + kHeads * t, r);
            tc::tmem_ld_wait(r);
            if (key0 + t * kTile + row < A.N) {
#pragma unroll
                for (int g = 0; g < kMaxHeads; ++g) mx[g] = fmaxf(mx[g], __uint_as_float(r[g]));
            }
        }
        float *red = reinterpret_cast<float *>(dtc_smem + kSmemRed);
#pragma unroll
        for (int g = 0; g < kMaxHeads; ++g) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx[g] = fmaxf(mx[g], __shfl_xor_sync(0xFFFFFFFFu, mx[g], o));
            if (lane == 0) red[(warp & 3) * kMaxHeads + g] = mx[g];
        }
        epi_sync();
        float mref[kMaxHeads], l[kMaxHeads];
#pragma unroll
        for (int g = 0; g < kMaxHeads; ++g) {
            mref[g] = A.scale_log2 * fmaxf(fmaxf(red[g], red[kMaxHeads + g]), fmaxf(red[2 * kMaxHeads + g], red[3 * kMaxHeads + g]));
            l[g] = 0.f;
        }
        epi_sync();                                                  // red is reused for the sums below
        for (int t = 0; t < nt; ++t) {
            const int pb = t & 1;
            ok = ok && tc::mbar_wait_warp(bar(kBarPEmpty + pb), ((t >> 1) & 1) ^ 1, abort_flag, cta_status);
            if (!ok) continue;
            uint32_t r[16];
            tc::tmem_ld16(trow + kHeads + kHeads * t, r);
            tc::tmem_ld_wait(r);
            const bool valid = key0 + t * kTile + row < A.N;
            const uint32_t prow = base + kSmemP + pb * 2 * kSmallPanel + (row >> 6) * kSmallPanel + ((row & 7) << 1);
            const int chunk = (row & 63) >> 3;
#pragma unroll
            for (int g = 0; g < kMaxHeads; ++g) {
                if (g < G) {
                    const float p = valid ? tc::ex2(fmaf(__uint_as_float(r[g]), A.scale_log2, -mref[g])) : 0.f;
                    // bf16 head and bf16 remainder in rows g and 8 + g: their two products add up in fp32, so the
                    // weight enters the second contraction with about 16 bits of mantissa
                    const __nv_bfloat16 hi = __float2bfloat16_rn(p), lo = __float2bfloat16_rn(p - __bfloat162float(hi));
                    l[g] += p;
                    const uint32_t at = prow + g * 128 + ((chunk ^ g) << 4);
                    sts16(at, __bfloat16_as_ushort(hi));
                    sts16(at + 1024, __bfloat16_as_ushort(lo));
                }
            }
            fence_proxy_async();
            tc::mbar_arrive(bar(kBarPFull + pb));
        }
#pragma unroll
        for (int g = 0; g < kMaxHeads; ++g) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) l[g] += __shfl_xor_sync(0xFFFFFFFFu, l[g], o);
            if (lane == 0) red[(warp & 3) * kMaxHeads + g] = l[g];
        }
        epi_sync();
        ok = ok && tc::mbar_wait_warp(bar(kBarO), 0, abort_flag, cta_status);
        tc::tc_fence_after();
        uint32_t r[16] = {};
        if (ok) {
            tc::tmem_ld16(trow, r);
            tc::tmem_ld_wait(r);
        }
        float *out = A.out + ((int64_t)u * A.Hq + h * G) * 128 + row;
        if (A.n_split == 1) {                                        // the only range of its head: normalise and finish
#pragma unroll
            for (int g = 0; g < kMaxHeads; ++g)
                if (g < G && ok)
                    out[g * 128] = (__uint_as_float(r[g]) + __uint_as_float(r[kMaxHeads + g])) /
                                   (red[g] + red[kMaxHeads + g] + red[2 * kMaxHeads + g] + red[3 * kMaxHeads + g]);
        } else if (A.clustered) {                                    // record: output [8][128], then maxima, sums (the tile stages are idle by now)
            float *rec = reinterpret_cast<float *>(dtc_smem);
#pragma unroll
            for (int g = 0; g < kMaxHeads; ++g) {
                if (g < G) rec[g * 128 + row] = __uint_as_float(r[g]) + __uint_as_float(r[kMaxHeads + g]);
                if (e == g && g < G) {
                    rec[kMaxHeads * 128 + g] = mref[g];
                    rec[kMaxHeads * 128 + kMaxHeads + g] = red[g] + red[kMaxHeads + g] + red[2 * kMaxHeads + g] + red[3 * kMaxHeads + g];
                }
            }
        } else {
            float *dst = A.part + ((int64_t)uh * A.n_split + split) * G * 130;
#pragma unroll
            for (int g = 0; g < kMaxHeads; ++g) {
                if (g < G) dst[g * 130 + row] = __uint_as_float(r[g]) + __uint_as_float(r[kMaxHeads + g]);
                if (e == g && g < G) {
                    dst[g * 130 + 128] = mref[g];
                    dst[g * 130 + 129] = red[g] + red[kMaxHeads + g] + red[2 * kMaxHeads + g] + red[3 * kMaxHeads + g];
                }
            }
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == 1) tc::tmem_dealloc(tmem, kTmemCols);
    if (threadIdx.x == 0 && *abort_flag != 0) status_write(A.status, A.call, *cta_status);
    if (A.clustered) {                                               // (also after a wait that ran out: every thread of the cluster comes here)
        __syncwarp();
        cluster_sync();
        if (threadIdx.x >= 64 && *abort_flag == 0) {
            const int d = threadIdx.x - 64;
            for (int g = split; g < A.G; g += A.n_split) {           // this CTA's share of the heads, thread = output dim
                // every range's record is on its way before the first is looked at (8 heads of 844 keys, one after the other 8.1 us, so 6.6)
                float m[kMaxRanges], l[kMaxRanges], v[kMaxRanges], mx = kNegBig, o = 0.f, ls = 0.f;
#pragma unroll
                for (int sp = 0; sp < kMaxRanges; ++sp) {
                    const bool on = sp < A.n_split;
                    m[sp] = on ? ld_cluster(base + 4 * (kMaxHeads * 128 + g), sp) : kNegBig;
                    l[sp] = on ? ld_cluster(base + 4 * (kMaxHeads * 128 + kMaxHeads + g), sp) : 0.f;
                    v[sp] = on ? ld_cluster(base + 4 * (g * 128 + d), sp) : 0.f;
                }
#pragma unroll
                for (int sp = 0; sp < kMaxRanges; ++sp) mx = fmaxf(mx, m[sp]);
#pragma unroll
                for (int sp = 0; sp < kMaxRanges; ++sp) {
                    const float w = tc::ex2(m[sp] - mx);
                    o = fmaf(v[sp], w, o);
                    ls = fmaf(l[sp], w, ls);
                }
                A.out[((int64_t)u * A.Hq + h * A.G + g) * 128 + d] = o / ls;
            }
        }
        __syncwarp();
        cluster_sync();                                              // nobody's shared memory goes away while it is read
    }
}

}  // namespace dtc
}  // namespace flowmm
