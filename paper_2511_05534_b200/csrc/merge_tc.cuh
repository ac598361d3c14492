// Weighted merge (Eq. 5) + compaction on the tensor cores, for budgets of up to 240 pivots per head
// (bf16, head_dim 128).
//
// Eq. 5 is out = W X with X the head's L rows of K (or V) and W a B x L matrix with one non-zero per
// column: W[s, t] = w_t if token t is merged into slot s, 1 for the pivot itself.  With few slots that
// product is cheap on the tensor cores and turns the gather into two linear streams (K and V, each row
// read from HBM once, by TMA) with no sort of the match beforehand:
//   merge_map_kernel   scatters (slot, weight) of every token into a per-position table;
//   merge_tc_kernel    persistent CTAs, one (unit, KV head) at a time, 128 tokens per step:
//       builder threads (one per token of the step) write the step's W^T slice into shared memory as a
//       K-major bf16 operand and add the same bf16-rounded weight to its slot's sum (fixed point in
//       shared memory: integer additions commute, so the sum does not depend on their order);
//       out^T[dim, slot] += X_step^T W_step^T as tcgen05.mma with M = 128 dims, N = slots, contraction
//       over the step's tokens; the X tile is the swizzled TMA tile read as an MN-major operand, for K
//       and for V against the same W slice;
//       after the last step eight reader warps (four for K, four for V) take out^T from TMEM, scale by
//       1 / (1 + sum of weights), transpose 4 x 4 blocks between lanes and store bf16 rows, while the next head's steps
//       already run into a second set of sums and (up to 128 slots) a second set of accumulators.
// When the heads fill at most half of the SMs a CTA takes one head's K or V only, with its own copy of W.
// When SMs are left over even so, a cluster of two or four CTAs shares the steps: each leaves its part of out^T in fp32 in its
// shared memory (where W was) and they add the parts up in a fixed order through distributed shared memory, a slice of the
// slots each: calls of 8 heads of 1471 tokens 42.0 -> 39.8 us, 4 of 2176 47.4 -> 43.0, 4 of 4528 65.6 -> 52.5.
// Bound by HBM with few slots and by the products with many: a step of 128 tokens takes the tensor core 384 clocks per tensor with 64
// slots, 512 with 128, 896 with 224 (that X is read MN-major costs nothing).  With four readers storing two bytes per lane the readout took 9 000 (64 slots) to 30 000
// clocks (218) per head on top: 8 heads of 1471 tokens, 148 slots 32 -> 18 us, 112 of 2176, 218 slots 47 -> 36 us, 32 of 640,
// 64 slots 18 -> 12 us, 1024 of 640 68 -> 63 us.
// The weights enter rounded to bf16 (relative error <= 2^-9) in numerator and denominator alike, so every
// output row is still a weighted mean of its members with weights within 0.2 % of Eq. 5's; the change of
// the result is below the bf16 rounding of the output itself.
// Products of bf16 inputs are exact in fp32 and the accumulation order is the hardware's, fixed for a
// given shape, so results are bit-reproducible.  A non-finite K or V entry would reach every slot of its
// head through 0 x inf; the gather kernels confine it to its own slot.
#pragma once
#include "common.cuh"
#include "decode_tc.cuh"
#include "tc_common.cuh"

namespace flowmm {
namespace mtc {

constexpr int kTile = 128;                       // tokens per step
constexpr int kMaxSlots = 240;                   // N <= 240: two 60 KB weight slices and three tile stages fit in shared memory
constexpr int kThreads = 448;                    // TMA warp, MMA warp, four builder warps, eight reader warps
constexpr int kPivotFlag = 1 << 30;              // in the table's slot word: the token is the slot's pivot
constexpr uint32_t kStageBytes = kTile * 128 * 2, kPanel = kStageBytes / 2;
constexpr int kMaxStages = 4;
constexpr int kBarFull = 0, kBarEmpty = kMaxStages, kBarWFull = 2 * kMaxStages, kBarWEmpty = kBarWFull + 2,
              kBarOutFull = kBarWEmpty + 2, kBarSumFull = kBarOutFull + 2, kBarOutEmpty = kBarSumFull + 2,
              kNumBars = kBarOutEmpty + 2;               // sums: 128 arrivals; accumulators read out: 256
constexpr uint32_t kTailData = 2 * kMaxSlots * 4 + 256 * 4;           // weight sums of two heads, reciprocal normalisers (whole blocks of 32 are read)
constexpr float kSumScale = 65536.f;             // weights in [2^-3, 1] rounded to bf16 are whole multiples of 2^-10

struct Args {
    const int2 *tokmap;          // [UH, L] (slot | pivot flag, or -1; weight bits)
    void *k_out, *v_out;
    int *status;
    int Hkv, L, B, n_items, n_stages;
    int per_item;                // 2: an item is a head; 1: an item is a head's K (even items) or V (odd items)
    int ctas;                    // > 1 (per_item == 1): the steps of an item are shared by the CTAs of a cluster
    int64_t kos[3], vos[3];
};

__host__ __device__ inline int slots16(int B) { return (B + 15) & ~15; }
__host__ __device__ inline uint32_t w_bytes(int B) { return (uint32_t)slots16(B) * 256u; }      // two 64-token panels of N rows
__host__ __device__ inline uint32_t smem_bytes(int B, int n_stages) {
    return (uint32_t)n_stages * kStageBytes + 2 * w_bytes(B) + kTailData + 8 * kNumBars + 16;
}

__device__ __forceinline__ void reader_sync() { asm volatile("bar.sync 2, 256;" ::: "memory"); }

// 32 output columns (slots s0 ..) of this thread's row (dim) scaled, rounded and stored.  Lanes of four exchange so that each
// holds four consecutive dims of one slot: 8-byte stores, 64 contiguous bytes per slot and warp.
__device__ __forceinline__ void store_slots32(const uint32_t (&acc)[32], const float *inv, __nv_bfloat16 *out, int64_t stride, int s0, int B,
                                              int lane) {
    const int sub = lane & 3;
    __nv_bfloat16 *dst = out + (int64_t)(s0 + sub) * stride;
#pragma unroll
    for (int q = 0; q < 32; q += 4) {
        const float4 f = *reinterpret_cast<const float4 *>(inv + s0 + q);
        const __nv_bfloat162 p01 = __floats2bfloat162_rn(__uint_as_float(acc[q]) * f.x, __uint_as_float(acc[q + 1]) * f.y);
        const __nv_bfloat162 p23 = __floats2bfloat162_rn(__uint_as_float(acc[q + 2]) * f.z, __uint_as_float(acc[q + 3]) * f.w);
        const uint32_t w01 = *reinterpret_cast<const uint32_t *>(&p01), w23 = *reinterpret_cast<const uint32_t *>(&p23);
        const uint32_t r01 = __shfl_xor_sync(0xFFFFFFFFu, w01, 1), r23 = __shfl_xor_sync(0xFFFFFFFFu, w23, 1);
        // even lanes: the pair's first slot, dims (d, d + 1); odd lanes: its second slot, dims (d - 1, d)
        const uint32_t a = (lane & 1) ? __byte_perm(r01, w01, 0x7632) : __byte_perm(w01, r01, 0x5410);
        const uint32_t b = (lane & 1) ? __byte_perm(r23, w23, 0x7632) : __byte_perm(w23, r23, 0x5410);
        const uint32_t got = __shfl_xor_sync(0xFFFFFFFFu, (lane & 2) ? a : b, 2);
        if (s0 + q + sub < B)
            *reinterpret_cast<uint2 *>(dst + (int64_t)q * stride) = (lane & 2) ? make_uint2(got, b) : make_uint2(a, got);
    }
}

struct MapArgs {
    const int *retained, *evicted, *match;
    const float *match_sim;
    int2 *tokmap;
    int L, B, E, merge_mode;
};

// grid = (UH, ceil(max(E, B) / 256))
__global__ void __launch_bounds__(256) merge_map_kernel(const MapArgs A) {
    predecessor_done();
    const int uh = blockIdx.x, i = blockIdx.y * 256 + threadIdx.x;
    int2 *map = A.tokmap + (int64_t)uh * A.L;
    if (i < A.E) {
        const int tok = A.evicted[(int64_t)uh * A.E + i];
        const float w = A.merge_mode == 1 ? 1.f : __expf(A.match_sim[(int64_t)uh * A.E + i] - 1.f);
        if (tok >= 0 && tok < A.L) map[tok] = make_int2(A.match[(int64_t)uh * A.E + i], __float_as_int(w));
    }
    if (i < A.B) {
        const int tok = A.retained[(int64_t)uh * A.B + i];
        if (tok >= 0 && tok < A.L) map[tok] = make_int2(i | kPivotFlag, __float_as_int(1.f));
    }
}

__global__ void __launch_bounds__(kThreads, 1)
merge_tc_kernel(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap, const Args A) {
    extern __shared__ __align__(1024) uint8_t mtc_smem[];
    const uint32_t base = tc::smem_u32(mtc_smem);
    const int N = slots16(A.B);
    // accumulator sets in TMEM: up to 128 slots two sets (K at column 0, V at column 128 of a set), else one (V at 256)
    const int n_sets = N <= 128 ? 2 : 1;
    const uint32_t set_cols = 256u, v_col = N <= 128 ? 128u : 256u;
    const uint32_t wsize = w_bytes(A.B), wpanel = (uint32_t)N * 128u;
    const uint32_t w0 = base + (uint32_t)A.n_stages * kStageBytes;
    uint8_t *tail = mtc_smem + (size_t)A.n_stages * kStageBytes + 2 * (size_t)wsize;
    unsigned *wsum = reinterpret_cast<unsigned *>(tail);                                  // [2][kMaxSlots], units of 1 / kSumScale
    float *inv_s = reinterpret_cast<float *>(tail + 2 * kMaxSlots * 4);                   // [256]
    const uint32_t bars = tc::smem_u32(tail + kTailData);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(tail + kTailData + 8 * kNumBars);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tail + kTailData + 8 * kNumBars + 4);
    const int warp = tc::warp_number(), lane = threadIdx.x & 31;
    if ((base & 1023u) != 0) {
        predecessor_done();
        if (threadIdx.x == 0) atomicCAS(A.status, 0, 6);
        return;
    }
    auto bar = [&](int i) { return bars + 8u * i; };
    if (threadIdx.x == 0) {
        for (int i = 0; i < kNumBars; ++i)
            tc::mbar_init(bar(i), i >= kBarOutEmpty ? 256 : (i >= kBarWFull && i < kBarWFull + 2) || i >= kBarSumFull ? 128 : 1);
        *abort_flag = 0;
        tc::mbar_init_fence();
        tc::tma_prefetch_desc(&kmap);
        tc::tma_prefetch_desc(&vmap);
    }
    if (warp == 1) tc::tmem_alloc(tc::smem_u32(tmem_slot), 512);
    for (uint32_t o = threadIdx.x * 16; o < 2 * wsize; o += kThreads * 16) dtc::sts128u(w0 + o, make_uint4(0, 0, 0, 0));
    for (int i = threadIdx.x; i < 2 * kMaxSlots; i += kThreads) wsum[i] = 0u;
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    predecessor_done();
    successor_may_start();
    const int ctas = A.ctas, rank = ctas > 1 ? (int)(blockIdx.x % (unsigned)ctas) : 0;
    const int first_item = ctas > 1 ? (int)(blockIdx.x / (unsigned)ctas) : (int)blockIdx.x, item_step = ctas > 1 ? A.n_items : (int)gridDim.x;
    const int n_steps = (A.L + kTile - 1) / kTile, c_lo = n_steps * rank / ctas, n_chunk = n_steps * (rank + 1) / ctas;   // steps c_lo .. n_chunk - 1
    const int per_item = A.per_item;                             // tensors of an item; the first (only) one:
    auto first_tensor = [&](int item) { return per_item == 2 ? 0 : item & 1; };
    auto head_of = [&](int item) { return per_item == 2 ? item : item >> 1; };

    if (warp == 0) {
        bool ok = true;
        int st = 0, phase = 0;
        for (int item = first_item; ok && item < A.n_items; item += item_step) {
            const int u = head_of(item) / A.Hkv, h = head_of(item) % A.Hkv, t0 = first_tensor(item);
            for (int c = c_lo; ok && c < n_chunk; ++c)
                for (int t = 0; t < per_item; ++t) {             // per step the K tile, then the V tile
                    ok = tc::mbar_wait_warp(bar(kBarEmpty + st), phase ^ 1, abort_flag, A.status);
                    if (!ok) break;
                    const CUtensorMap *m = (per_item == 2 ? t : t0) ? &vmap : &kmap;
                    const uint32_t dst = base + st * kStageBytes;
                    if (tc::elect_one()) {
                        tc::mbar_expect_tx(bar(kBarFull + st), kStageBytes);
                        tc::tma_load_4d(dst, m, bar(kBarFull + st), 0, c * kTile, h, u);
                        tc::tma_load_4d(dst + kPanel, m, bar(kBarFull + st), 64, c * kTile, h, u);
                    }
                    __syncwarp();
                    if (++st == A.n_stages) { st = 0; phase ^= 1; }
                }
        }
        if (!ok)         // winding down after a timeout: give copies already issued a moment to land
            for (int i = 0; i < A.n_stages; ++i)
                for (int n = 0; n < (1 << 16) && !tc::mbar_try_wait(bar(kBarFull + i), 0) && !tc::mbar_try_wait(bar(kBarFull + i), 1); ++n) {}
    } else if (warp == 1) {
        const uint32_t idesc = tc::idesc_bf16(128, (uint32_t)N) | (1u << 15);           // A operand MN-major
        const uint32_t a_hi = tc::kDescSw128Hi, a_lead = (kPanel >> 4) << 16;            // (and the stride between its panels)
        bool ok = true;
        int st = 0, st_phase = 0, wb = 0, w_phase = 0, it = 0;
        for (int item = first_item; ok && item < A.n_items; item += item_step, ++it) {
            const int set = it % n_sets, use = it / n_sets;
            ok = tc::mbar_wait_warp(bar(kBarOutEmpty + set), (use & 1) ^ 1, abort_flag, A.status);   // the set's previous head is read out
            tc::tc_fence_after();
            for (int c = c_lo; ok && c < n_chunk; ++c) {
                ok = tc::mbar_wait_warp(bar(kBarWFull + wb), w_phase, abort_flag, A.status);
                const uint32_t w_lo = tc::desc_lo(w0 + wb * wsize);
                for (int t = 0; ok && t < per_item; ++t) {
                    ok = tc::mbar_wait_warp(bar(kBarFull + st), st_phase, abort_flag, A.status);
                    if (!ok) break;
                    tc::tc_fence_after();
                    const uint32_t a_lo = tc::desc_lo(base + st * kStageBytes) | a_lead, d = tmem + set * set_cols + t * v_col;
                    if (tc::elect_one()) {
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            tc::umma_bf16(d, a_lo + q * 128, a_hi, w_lo + (q >> 2) * (wpanel >> 4) + (q & 3) * 2, tc::kDescSw128Hi, idesc, c > c_lo || q > 0);
                        tc::umma_commit(bar(kBarEmpty + st));
                        if (t == per_item - 1) tc::umma_commit(bar(kBarWEmpty + wb));
                    }
                    __syncwarp();
                    if (++st == A.n_stages) { st = 0; st_phase ^= 1; }
                }
                wb ^= 1;
                w_phase ^= wb == 0;
            }
            if (ok && tc::elect_one()) tc::umma_commit(bar(kBarOutFull + set));
            __syncwarp();
        }
    } else if (warp < 6) {
        // builders: thread = token of a step
        const int e = threadIdx.x - 64;
        uint32_t wr0 = 0, wr1 = 0;                                   // where this thread's last entry of each W buffer sits
        bool ok = true;
        int j = 0, it = 0;
        // position of this thread's token inside a W panel row: 64 tokens per 128-byte row, 16-byte groups swizzled by row
        const uint32_t tok_off = (uint32_t)(e >> 6) * wpanel + (uint32_t)((e & 7) << 1);
        const int tok_grp = (e & 63) >> 3;
        const int e0 = c_lo * kTile + e;                             // this thread's first token
        int2 first = first_item < A.n_items && e0 < A.L ? A.tokmap[(int64_t)head_of(first_item) * A.L + e0] : make_int2(-1, 0);
        for (int item = first_item; item < A.n_items; item += item_step, ++it) {
            const int2 *map = A.tokmap + (int64_t)head_of(item) * A.L;
            const int set = it % n_sets, use = it / n_sets;
            unsigned *sums = wsum + set * kMaxSlots;
            // the set's sums are zero again once its previous head has been read out
            ok = ok && tc::mbar_wait(bar(kBarOutEmpty + set), (use & 1) ^ 1, abort_flag, A.status);
            int2 nxt = first;
            for (int c = c_lo; c < n_chunk; ++c, ++j) {
                const int2 cur = nxt;
                const int t_next = (c + 1) * kTile + e;
                if (c + 1 < n_chunk) nxt = t_next < A.L ? map[t_next] : make_int2(-1, 0);
                else first = item + item_step < A.n_items && e0 < A.L ? A.tokmap[(int64_t)head_of(item + item_step) * A.L + e0] : make_int2(-1, 0);
                const int wb = j & 1;
                ok = ok && tc::mbar_wait(bar(kBarWEmpty + wb), ((j >> 1) & 1) ^ 1, abort_flag, A.status);
                const uint32_t w = w0 + wb * wsize;
                const uint32_t prev = wb ? wr1 : wr0;
                uint32_t mine = 0;
                if (ok && prev) dtc::sts16(prev, 0);                 // take back what this thread wrote two steps ago
                const int slot = cur.x & ~kPivotFlag;
                if (ok && cur.x >= 0 && slot < A.B) {
                    const __nv_bfloat16 wt = __float2bfloat16_rn(__int_as_float(cur.y));
                    const uint32_t at = w + tok_off + (uint32_t)slot * 128u + (uint32_t)((tok_grp ^ (slot & 7)) << 4);
                    dtc::sts16(at, __bfloat16_as_ushort(wt));
                    mine = at;
                    if (!(cur.x & kPivotFlag)) atomicAdd(sums + slot, (unsigned)(__bfloat162float(wt) * kSumScale + 0.5f));
                }
                if (wb) wr1 = mine; else wr0 = mine;
                dtc::fence_proxy_async();
                tc::mbar_arrive(bar(kBarWFull + wb));
            }
            tc::mbar_arrive(bar(kBarSumFull + set));                 // this head's weight sums are complete
        }
    } else {
        // readers: thread = output dim; columns = slots; the first four warps take K, the others V
        const int e = threadIdx.x - 192, t = e >> 7;
        const uint32_t trow = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
        bool ok = true;
        int it = 0;
        for (int item = first_item; item < A.n_items; item += item_step, ++it) {
            const int u = head_of(item) / A.Hkv, h = head_of(item) % A.Hkv;
            const int set = it % n_sets, use = it / n_sets;
            unsigned *sums = wsum + set * kMaxSlots;
            ok = ok && tc::mbar_wait_warp(bar(kBarSumFull + set), use & 1, abort_flag, A.status);
            if (ctas > 1) {
                // this CTA's part of the product, slot by slot, over the weight slices (whose products are complete)
                ok = ok && tc::mbar_wait_warp(bar(kBarOutFull + set), use & 1, abort_flag, A.status);
                tc::tc_fence_after();
                if (ok) {
                    for (int s0 = 32 * t; s0 < N; s0 += 64) {
                        uint32_t acc[32];
                        tc::tmem_ld32(trow + set * set_cols + s0, acc);
                        tc::tmem_ld_wait(acc);
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (s0 + i < N) tc::sts32(w0 + ((uint32_t)(s0 + i) * 128u + (uint32_t)(32 * (warp & 3) + lane)) * 4u, __uint_as_float(acc[i]));
                    }
                }
                break;                                               // (one item per cluster)
            }
            for (int sl = e; ok && sl < N; sl += 256) {
                inv_s[sl] = 1.f / (1.f + (float)sums[sl] * (1.f / kSumScale));
                sums[sl] = 0u;
            }
            reader_sync();
            ok = ok && tc::mbar_wait_warp(bar(kBarOutFull + set), use & 1, abort_flag, A.status);
            tc::tc_fence_after();
            if (ok) {
                // a single tensor's slots go to the two quads in turn, 32 at a time
                const int which = per_item == 2 ? t : first_tensor(item);
                __nv_bfloat16 *out = static_cast<__nv_bfloat16 *>(which ? A.v_out : A.k_out) +
                                     (which ? u * A.vos[0] + h * A.vos[1] : u * A.kos[0] + h * A.kos[1]) + 32 * (warp & 3) + (lane & ~3);
                const int64_t stride = which ? A.vos[2] : A.kos[2];
                const uint32_t tcol = trow + set * set_cols + (per_item == 2 ? t * v_col : 0u);
#pragma unroll 1
                for (int s0 = per_item == 2 ? 0 : 32 * t; s0 < A.B; s0 += per_item == 2 ? 32 : 64) {
                    uint32_t acc[32];
                    tc::tmem_ld32(tcol + s0, acc);
                    tc::tmem_ld_wait(acc);
                    store_slots32(acc, inv_s, out, stride, s0, A.B, lane);
                }
            }
            tc::tc_fence_before();
            reader_sync();                                           // inv_s may be rewritten, the set reused
            tc::mbar_arrive(bar(kBarOutEmpty + set));
        }
    }
    if (ctas > 1) {
        // the parts of all CTAs added up in their order, a slice of the slots per CTA, a slot per warp
        cluster_sync();
        const int item = first_item, u = head_of(item) / A.Hkv, h = head_of(item) % A.Hkv, which = first_tensor(item);
        __nv_bfloat16 *out = static_cast<__nv_bfloat16 *>(which ? A.v_out : A.k_out) +
                             (which ? u * A.vos[0] + h * A.vos[1] : u * A.kos[0] + h * A.kos[1]) + 4 * lane;
        const int64_t stride = which ? A.vos[2] : A.kos[2];
        const uint32_t sums_at = tc::smem_u32(wsum);
        for (int sl = A.B * rank / ctas + warp; sl < A.B * (rank + 1) / ctas; sl += kThreads / 32) {
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            unsigned total = 0;
#pragma unroll 4
            for (int q = 0; q < ctas; ++q) {
                const uint4 v = ld_cluster_u128(w0 + (uint32_t)sl * 512u + (uint32_t)lane * 16u, q);
                total += ld_cluster_u32(sums_at + 4u * (uint32_t)sl, q);
                x.x += __uint_as_float(v.x); x.y += __uint_as_float(v.y); x.z += __uint_as_float(v.z); x.w += __uint_as_float(v.w);
            }
            const float inv = 1.f / (1.f + (float)total * (1.f / kSumScale));
            const __nv_bfloat162 lo = __floats2bfloat162_rn(x.x * inv, x.y * inv), hi = __floats2bfloat162_rn(x.z * inv, x.w * inv);
            *reinterpret_cast<uint2 *>(out + (int64_t)sl * stride) = make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
        }
        cluster_sync();                                              // nobody's part goes away while it is read
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == 1) tc::tmem_dealloc(tmem, 512);
}

}  // namespace mtc
}  // namespace flowmm
