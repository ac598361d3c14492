// Window scoring (Eq. 8 with the softmax of Eq. 4, and the masses of Eq. 7) in one pass over K for contexts of a few key tiles and 64 to
// 512 proxy rows per KV head (bf16, head_dim 128): the CTAs of a cluster share a head's keys, every logit of a CTA's keys stays in its
// TMEM, and only the rows' statistics are exchanged.
//
// A CTA has kt tiles of 128 keys against the head's rt tiles of 128 proxy rows, kt rt <= 4 (512 TMEM columns); S = Q_tile K_tile^T has
// the proxy rows as lanes, so that row maxima and sums are a thread's own, and only the column sums cross lanes, once per key:
//   1  per 32 keys a thread forms its row's exponentials against the maximum of those 32, writes them over the logits and keeps the sums
//      over text and visual keys;
//   2  warps, then CTAs (through distributed shared memory) join the rows' records; a row's constant is -(max + log2 sum);
//   3  exponentials x 2^(their maximum + constant), summed over a thread's rows, then over lanes by transposition and over the four warps
//      of a key: the importance.
// The two-pass kernels of score_tc.cuh form every logit and exponential twice and are two launches.  Bound by its chain of loads, products,
// sweeps and two meetings, about 9 us, so only for calls whose CTAs all run at once.  The whole call, us, by two passes and so: 4 heads of 500
// tokens, 224 rows 27.5, 24.3; of 1000 31.2, 28.9; 16 of 1471 37.2, 33.8; 8 of 700, 512 rows 35.9, 34.4.
// One head per cluster, blocks start afresh: warp 0 issues the copies, warp 1 the products, warps 2-17 do the rest (a warp has 32 lanes x
// 32 keys of every accumulator).
#pragma once
#include "common.cuh"
#include "decode_tc.cuh"
#include "score_fused_tc.cuh"
#include "score_tc.cuh"
#include "tc_common.cuh"

namespace flowmm {
namespace sct {

constexpr int kTile = 128, kMaxAcc = 4, kMaxCtas = 8;
constexpr int kEpiThreads = 512, kThreads = 64 + kEpiThreads;
constexpr uint32_t kTileBytes = kTile * 128 * 2, kPanel = kTileBytes / 2;
constexpr int kBarQ = 0, kBarK = kMaxAcc, kBarAcc = 2 * kMaxAcc, kNumBars = 3 * kMaxAcc;

// Shared memory behind the operand tiles: records of the warps and of the CTA, row constants, a table for sums by modality, partial sums.
constexpr uint32_t kRows = kMaxAcc * kTile;
constexpr uint32_t kStat = 0, kRec = kStat + 4 * kRows * 12, kConst = kRec + kRows * 16, kMasks = kConst + kRows * 4, kPart = kMasks + 256;
// At least so much that no other block with tensor memory fits beside it on an SM (decode attention's are the smallest, 109 KB): a cluster's
// blocks wait for one another, and two clusters of different streams, each with a block that waits for the tensor memory of one of the
// other's, would wait forever.
constexpr uint32_t kMinSmem = 120 * 1024;
static_assert(kMinSmem + dtc::kSmemBytes > 227 * 1024, "no room beside it");
inline __host__ uint32_t smem_bytes(int rt, int kt) {
    const uint32_t n = (uint32_t)(rt + kt) * kTileBytes + kPart + 4u * kt * kTile * 4u + 8 * kNumBars + 16;
    return n > kMinSmem ? n : kMinSmem;
}

struct Args {
    const uint8_t *modality;     // [U, L]
    float *importance;           // [UH, L]
    float *cross_part;           // [U*Hq, W] share of a proxy row's mass that falls on keys of the other modality
    int *status;
    int Hq, Hkv, G, W, L, GW;
    int rt, kt, ctas;            // tiles of proxy rows, key tiles per CTA, CTAs per head
    uint32_t q_bytes;            // that a Q box delivers
    float scale_log2;
};

__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 512;" ::: "memory"); }

__global__ void __launch_bounds__(kThreads, 1)
score_cluster_tc_kernel(const __grid_constant__ CUtensorMap qmap, const __grid_constant__ CUtensorMap kmap, const Args A) {
    extern __shared__ __align__(1024) uint8_t sct_smem[];
    const uint32_t base = tc::smem_u32(sct_smem), q_at = base, k_at = base + (uint32_t)A.rt * kTileBytes;
    const uint32_t data = k_at + (uint32_t)A.kt * kTileBytes, part_at = data + kPart, bars = part_at + 4u * A.kt * kTile * 4u;
    const int warp = tc::warp_number(), lane = threadIdx.x & 31;
    uint8_t *tail = sct_smem + (bars - base) + 8 * kNumBars;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(tail);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tail + 4);
    const bool aligned = (base & 1023u) == 0;                        // (the same for the CTAs of a cluster)
    if (!aligned) {
        predecessor_done();
        if (threadIdx.x == 0) atomicCAS(A.status, 0, 6);
        return;
    }
    auto bar = [&](int i) { return bars + 8u * i; };
    if (threadIdx.x == 0) {
        for (int i = 0; i < kNumBars; ++i) tc::mbar_init(bar(i), 1);
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
    const int uh = blockIdx.x / A.ctas, rank = blockIdx.x % A.ctas, u = uh / A.Hkv, h = uh - u * A.Hkv;
    const int nt = (A.L + kTile - 1) / kTile, tile0 = rank * A.kt, n_k = min(A.kt, nt - tile0);   // this CTA's key tiles (at least one)

    if (warp == 0) {
        if (tc::elect_one()) {
            auto load = [&](uint32_t dst, const CUtensorMap *m, uint32_t full, uint32_t bytes, int c1, int c2) {
                tc::mbar_expect_tx(full, bytes);
                tc::tma_load_4d(dst, m, full, 0, c1, c2, u);
                tc::tma_load_4d(dst + kPanel, m, full, 64, c1, c2, u);
            };
            for (int i = 0; i < max(A.rt, n_k); ++i) {
                if (i < n_k) load(k_at + i * kTileBytes, &kmap, bar(kBarK + i), kTileBytes, (tile0 + i) * kTile, h);
                if (i < A.rt) load(q_at + i * kTileBytes, &qmap, bar(kBarQ + i), A.q_bytes, 0, h * A.G + i * (kTile / A.W));
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        constexpr uint32_t idesc = tc::idesc_bf16(kTile, kTile);
        bool ok = true;
        for (int k = 0; ok && k < n_k; ++k) {
            ok = tc::mbar_wait_warp(bar(kBarK + k), 0, abort_flag, A.status);
            for (int t = 0; ok && t < A.rt; ++t) {
                if (k == 0) ok = tc::mbar_wait_warp(bar(kBarQ + t), 0, abort_flag, A.status);
                if (!ok) break;
                tc::tc_fence_after();
                const uint32_t a_lo = tc::desc_lo(q_at + t * kTileBytes), b_lo = tc::desc_lo(k_at + k * kTileBytes), d = tmem + (k * A.rt + t) * kTile;
                if (tc::elect_one()) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        tc::umma_bf16(d, a_lo + (j >> 2) * (kPanel >> 4) + (j & 3) * 2, tc::kDescSw128Hi, b_lo + (j >> 2) * (kPanel >> 4) + (j & 3) * 2,
                                      tc::kDescSw128Hi, idesc, j > 0);
                    tc::umma_commit(bar(kBarAcc + k * A.rt + t));
                }
                __syncwarp();
            }
        }
        if (!ok) {       // a wait ran out: copies already issued get a moment to land
            for (int i = 0; i < 2 * kMaxAcc; ++i) {
                const bool issued = i < kMaxAcc ? i < A.rt : i - kMaxAcc < n_k;
                for (int s = 0; issued && s < (1 << 16) && !tc::mbar_try_wait(bar(i), 0); ++s) {}
            }
        }
    }
    // (the first two warps go on to the cluster's meetings)
    const bool epi = warp >= 2;
    const int quarter = warp & 3, cg = ((warp - 2) >> 2) & 3, te = threadIdx.x - 64;   // 32 TMEM lanes; 32 keys of every tile
    const uint32_t trow = tmem + ((uint32_t)(32 * quarter) << 16) + cg * 32;
    bool ok = true;
    float mref[kMaxAcc];                                             // maximum that an accumulator's exponentials are relative to
    if (epi) {
        const uint8_t *mod = A.modality + (int64_t)u * A.L;
        uint8_t of_key[kMaxAcc];
#pragma unroll
        for (int k = 0; k < kMaxAcc; ++k) {
            const int key = (tile0 + k) * kTile + cg * 32 + lane;
            of_key[k] = k < n_k ? mod[min(key, A.L - 1)] : 0;        // (keys past the prompt count with its last token, so that they make no mix)
        }
        uint8_t of_row[kMaxAcc];
#pragma unroll
        for (int t = 0; t < kMaxAcc; ++t) of_row[t] = mod[A.L - A.W + ((t * kTile + quarter * 32 + lane) & (A.W - 1))];   // (the window is 32, 64 or 128 rows)
        if (te < 64) tc::sts32(data + kMasks + te * 4, (te >> 2) >> (te & 3) & 1 ? -1.f : 0.f);
        epi_sync();
        float all_m[kMaxAcc], all_t[kMaxAcc], all_v[kMaxAcc];        // this warp's keys, by tile of rows
#pragma unroll
        for (int t = 0; t < kMaxAcc; ++t) { all_m[t] = kNegBig; all_t[t] = all_v[t] = 0.f; mref[t] = kNegBig; }
#pragma unroll
        for (int i = 0; i < kMaxAcc; ++i) {                          // accumulator i: key tile i / rt, row tile i % rt
            const int k = A.rt == 1 ? i : A.rt == 2 ? i >> 1 : 0, t = A.rt == 1 ? 0 : A.rt == 2 ? i & 1 : i;
            if (k >= n_k || t >= A.rt) continue;
            ok = ok && tc::mbar_wait_warp(bar(kBarAcc + i), 0, abort_flag, A.status);
            const int kb = (tile0 + k) * kTile + cg * 32, r0 = t * kTile + quarter * 32;
            if (!ok || kb >= A.L || r0 >= A.GW) continue;            // (the whole warp)
            tc::tc_fence_after();
            uint32_t a[32];
            tc::tmem_ld32(trow + i * kTile, a);
            tc::tmem_ld_wait(a);
            const uint32_t vis = __ballot_sync(0xFFFFFFFFu, (k == 0 ? of_key[0] : k == 1 ? of_key[1] : k == 2 ? of_key[2] : of_key[3]) != 0);
            const uint32_t rows = __ballot_sync(0xFFFFFFFFu, (t == 0 ? of_row[0] : t == 1 ? of_row[1] : t == 2 ? of_row[2] : of_row[3]) != 0);
            const bool masked = kb + 32 > A.L - A.W + 1;
            if (masked) {
                const int last = A.L - A.W + ((r0 + lane) & (A.W - 1)) - kb;   // this row sees the chunk's keys 0 .. last
#pragma unroll
                for (int j = 0; j < 32; ++j) a[j] = j <= last ? a[j] : __float_as_uint(-INFINITY);
            }
            const float mx = fmaxf(max32(a) * A.scale_log2, kNegBig);
            // By the exp2 unit alone where few keys or rows can make up a result, and in the window's whole tile, whose keys the second of two
            // passes gives to that unit as well.
            if ((tile0 + k + 1) * kTile > A.L - A.W + 1 || (vis != 0u && vis != 0xFFFFFFFFu) || (rows != 0u && rows != 0xFFFFFFFFu)) exp2_32_exact(a, A.scale_log2, mx);
            else exp2_32(a, A.scale_log2, mx);
            tc::tmem_st32(trow + i * kTile, a);
            float on_text = 0.f, on_vis = 0.f;
            if (vis == 0u) on_text = sum32(a);
            else if (vis == 0xFFFFFFFFu) on_vis = sum32(a);
            else sums32_by(a, vis, data + kMasks, on_text, on_vis);
            mref[i] = mx;
#pragma unroll
            for (int q = 0; q < kMaxAcc; ++q)
                if (q == t) {
                    const RowStats s = join({all_m[q], all_t[q], all_v[q]}, {mx, on_text, on_vis});
                    all_m[q] = s.m; all_t[q] = s.t; all_v[q] = s.v;
                }
        }
        tc::tmem_st_wait();
#pragma unroll
        for (int t = 0; t < kMaxAcc; ++t) {
            const int r = t * kTile + quarter * 32 + lane;
            if (t >= A.rt || r >= A.GW) continue;
            const uint32_t at = data + kStat + (uint32_t)(cg * (int)kRows + r) * 12;
            tc::sts32(at, all_m[t]); tc::sts32(at + 4, all_t[t]); tc::sts32(at + 8, all_v[t]);
        }
        epi_sync();
        if (te < A.GW) {                                             // a thread per row: the four warps' records
            RowStats s = {kNegBig, 0.f, 0.f};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t at = data + kStat + (uint32_t)(c * (int)kRows + te) * 12;
                s = join(s, {tc::lds32(at), tc::lds32(at + 4), tc::lds32(at + 8)});
            }
            tc::sts128(data + kRec + te * 16, s.m, s.t, s.v, 0.f);
        }
    }
    cluster_sync();
    if (epi && te < A.GW) {                                          // ... and the CTAs', in their order
        uint4 o[kMaxCtas];
#pragma unroll
        for (int c = 0; c < kMaxCtas; ++c) o[c] = c < A.ctas ? ld_cluster_u128(data + kRec + te * 16, c) : make_uint4(__float_as_uint(kNegBig), 0u, 0u, 0u);
        RowStats s = {kNegBig, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < kMaxCtas; ++c) s = join(s, {__uint_as_float(o[c].x), __uint_as_float(o[c].y), __uint_as_float(o[c].z)});
        const float z = s.t + s.v;
        tc::sts32(data + kConst + te * 4, -(s.m + log2f(z)));
        if (rank == 0) {
            const bool vis = A.modality[(int64_t)(u + 1) * A.L - A.W + (te & (A.W - 1))] != 0;
            A.cross_part[((int64_t)u * A.Hq + h * A.G) * A.W + te] = (vis ? s.t : s.v) / z;
        }
    }
    cluster_arrive();                                                // the other CTAs' records have been read
    if (epi) {
        epi_sync();
        float f[kMaxAcc];
#pragma unroll
        for (int i = 0; i < kMaxAcc; ++i) {
            const int t = A.rt == 1 ? 0 : A.rt == 2 ? i & 1 : i, r = t * kTile + quarter * 32 + lane;
            f[i] = t < A.rt && r < A.GW ? tc::ex2(mref[i] + tc::lds32(data + kConst + r * 4)) : 0.f;
        }
#pragma unroll
        for (int k = 0; k < kMaxAcc; ++k) {
            if (k >= n_k) break;
            const int kb = (tile0 + k) * kTile + cg * 32;
            float sum[2][16];
#pragma unroll
            for (int j = 0; j < 16; ++j) sum[0][j] = sum[1][j] = 0.f;
            if (ok && kb < A.L) {
#pragma unroll
                for (int i = 0; i < kMaxAcc; ++i) {
                    const int of_k = A.rt == 1 ? i : A.rt == 2 ? i >> 1 : 0, t = A.rt == 1 ? 0 : A.rt == 2 ? i & 1 : i;
                    if (of_k != k || t >= A.rt || t * kTile + quarter * 32 >= A.GW) continue;
                    uint32_t a[32];
                    tc::tmem_ld32(trow + i * kTile, a);
                    tc::tmem_ld_wait(a);
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        sum[0][j] = fmaf(__uint_as_float(a[j]), f[i], sum[0][j]);
                        sum[1][j] = fmaf(__uint_as_float(a[16 + j]), f[i], sum[1][j]);
                    }
                }
            }
            sft::warp_reduce16(sum[0], [](float x, float y) { return x + y; });
            sft::warp_reduce16(sum[1], [](float x, float y) { return x + y; });
            if (!(lane & 1)) {
                const uint32_t at = part_at + (uint32_t)((quarter * A.kt + k) * kTile + cg * 32 + (lane >> 1)) * 4;
                tc::sts32(at, sum[0][0]);
                tc::sts32(at + 64, sum[1][0]);
            }
        }
        epi_sync();
        const int key = tile0 * kTile + te;
        if (te < n_k * kTile && key < A.L && *abort_flag == 0) {
            float x = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) x += tc::lds32(part_at + (uint32_t)(q * A.kt * kTile + te) * 4);
            A.importance[(int64_t)uh * A.L + key] = x / (float)A.G;  // group mean
        }
    }
    __syncwarp();
    cluster_wait();                                                  // nobody's records go away while they are read
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == 1) tc::tmem_dealloc(tmem, 512);
}

}  // namespace sct
}  // namespace flowmm
