// Tensor-core path of the matching step (Eq. 9 and Eq. 10) for bf16 keys with head_dim 128.
//
// Per (unit, KV head) the admissible pivots (importance <= tau) are gathered into a dense
// candidate matrix, text candidates first and visual candidates from the next multiple of 32.
// The similarity contraction then runs as  S[128 tokens x 256 candidates] = K_tile . C_tile^T
// (two such 128-token halves per candidate tile) on tcgen05, fp32 accumulators in TMEM, and an epilogue that scales each column
// by the candidate's reciprocal norm and keeps a running row maximum.  Raw bf16 keys feed the MMA (their products are exact in
// fp32); the norms enter in fp32 afterwards, so no precision is lost before the argmax.
// The token rows are the non-pivots alone, gathered from the caller's K by two warps of their own.  (Tiles of consecutive tokens,
// which the TMA unit can load, computed the pivots as well, only to drop them.  The whole call, us, so and now: 112 heads of 8448
// tokens with 1690 pivots 843 / 771, 112 of 640 with 423 95.2 / 87.5, 64 of 2407 with 1441 166 / 134; 128 of 33 792 with 1690
// 2860 / 2839.  Gathered copies by the TMA unit, four rows to one, are bit for bit the same and slower with few pivots: 256 rows took
// 3 us more than the two warps, which these hide behind the item before.)
// An intra-modal layer visits only the candidate group of the row tile's modality.
#pragma once
#include <type_traits>

#include "common.cuh"
#include "tc_stream.cuh"

namespace flowmm {

constexpr int kMtRows = tcs::kRows;          // tokens per accumulator half
constexpr int kMtItemRows = tcs::kItemRows;  // tokens per item (two halves)

struct MatchPrepArgs {
    const void *k;
    const float *importance;
    const uint8_t *modality;
    const int *retained, *evicted;
    __nv_bfloat16 *cand_k;       // [UH, Ctot, 128]
    float *cand_scale;           // [UH, Ctot]
    int *cand_slot;              // [UH, Ctot]
    int *cand_count;             // [UH, 2]  admissible text / visual pivots
    // what the matching kernel reads per token: the one for short candidate lists (copy_here) the rank of every token,
    int *rank;                   // [UH, L]  position in the non-pivot list, or -(s + 2) for the pivot of slot s
    // the general one, by position in the non-pivot list,
    uint8_t *evi_mod;            // [UH, E]  the token's modality
    uint8_t *tile_mod;           // [UH, n_rt] per tile of 256 positions; bit 0: holds text tokens, bit 1: visual tokens
    int Hkv, L, B, E, Ctot, n_rt;
    int *status;                 // device status word (index checks of the debug build report here)
    int copy_here;               // 1: this kernel also gathers the candidate rows; 0: match_gather_kernel does
    float tau_eff;
    int64_t ks[3];
};

// Copies the candidate key rows (256 bytes each) of positions [lo, hi) of one head's candidate
// list, 16 lanes per row, and takes each row's reciprocal norm on the way (0 for a zero row: its
// similarity to anything is 0).  lo, hi multiples of 32; every thread of the block takes part.
// cand_tok: the positions' tokens (-1: no candidate), or nullptr: found through the slots and the pivot list.
// kRows rows per lane are in flight together: a row is one dependent chain of loads.
template <int kRows>
struct MatchGather {
    const MatchPrepArgs &A;
    const __nv_bfloat16 *kb;
    int uh, sub, stride, tok[kRows];
    uint4 val[kRows];
    __device__ __forceinline__ MatchGather(const MatchPrepArgs &a, int uh_, int tid, int nthreads) : A(a), uh(uh_), sub(tid & 15), stride(nthreads >> 4) {
        const int u = uh / A.Hkv, h = uh % A.Hkv;
        kb = static_cast<const __nv_bfloat16 *>(A.k) + u * A.ks[0] + h * A.ks[1];
    }
    // Positions p0, p0 + stride, ... below hi: their rows start to come.
    __device__ __forceinline__ void start(const int *cand_tok, int p0, int hi) {
        const int *ret = A.retained + (int64_t)uh * A.B, *slot_out = A.cand_slot + (int64_t)uh * A.Ctot;
#pragma unroll
        for (int q = 0; q < kRows; ++q) {
            const int pos = p0 + q * stride;
            tok[q] = -1;
            if (pos < hi) {
                if (cand_tok) tok[q] = cand_tok[pos];
                else {
                    const int s = slot_out[pos];
                    if (s >= 0 && index_ok(s, A.B, A.status)) tok[q] = ret[s];
                }
            }
        }
#pragma unroll
        for (int q = 0; q < kRows; ++q) {
            val[q] = make_uint4(0, 0, 0, 0);
            if (tok[q] >= 0 && index_ok(tok[q], A.L, A.status))
                val[q] = *reinterpret_cast<const uint4 *>(kb + (int64_t)tok[q] * A.ks[2] + sub * 8);
        }
    }
    __device__ __forceinline__ void finish(int p0, int hi) {
        float *scale_out = A.cand_scale + (int64_t)uh * A.Ctot;
        uint4 *dst = reinterpret_cast<uint4 *>(A.cand_k + (int64_t)uh * A.Ctot * 128);
#pragma unroll
        for (int q = 0; q < kRows; ++q) {
            const int pos = p0 + q * stride;
            if (pos >= hi) break;                                           // (the same for both rows of a warp)
            dst[(int64_t)pos * 16 + sub] = val[q];
            float x[8], ssq = 0.f;
            Elem<__nv_bfloat16>::unpack(val[q], x);
#pragma unroll
            for (int e = 0; e < 8; ++e) ssq = fmaf(x[e], x[e], ssq);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) ssq += __shfl_xor_sync(0xFFFFFFFFu, ssq, o);
            if (sub == 0 && tok[q] >= 0) scale_out[pos] = ssq > 0.f ? rsqrtf(ssq) : 0.f;
        }
    }
};
template <int kRows>
__device__ __forceinline__ void match_gather_rows(const MatchPrepArgs &A, int uh, const int *cand_tok, int lo, int hi, int tid, int nthreads) {
    MatchGather<kRows> g(A, uh, tid, nthreads);
    for (int p0 = lo + (tid >> 4); p0 < hi; p0 += kRows * g.stride) {       // uniform trip count within a warp
        g.start(cand_tok, p0, hi);
        g.finish(p0, hi);
    }
}

// The candidate layout of one head from its pivot list, by a whole block (`scratch`: 33 ints of shared memory).  A thread takes kPer
// pivots in a row, whose loads are on their way together; one prefix sum numbers the candidates of both groups.  One pivot while the block
// has a thread for each, else eight: the steps one by one, 8 heads of 33 792 tokens with 1690 pivots, 235.8 -> 228.6 us, where rounds of a
// pivot per thread loaded twice and summed each time; flowmm_match of 56 heads of 1200 tokens with 120 pivots by eight 14.2, by one 12.4.
template <int kPer>
__device__ __forceinline__ void match_lay_out_candidates(const MatchPrepArgs &A, int uh, int *scratch) {
    const int tid = threadIdx.x, u = uh / A.Hkv, chunk = kPer * blockDim.x;
    const int *ret = A.retained + (int64_t)uh * A.B;
    const float *imp = A.importance + (int64_t)uh * A.L;
    const uint8_t *mod = A.modality + (int64_t)u * A.L;
    int *slot_out = A.cand_slot + (int64_t)uh * A.Ctot;
    float *scale_out = A.cand_scale + (int64_t)uh * A.Ctot;
    for (int i = tid; i < A.Ctot; i += blockDim.x) { slot_out[i] = -1; scale_out[i] = __int_as_float(0x7FC00000); }   // NaN: no candidate here
    // which of the thread's pivots are admissible text ones, which visual ones
    uint32_t text = 0, vis = 0;
    auto look = [&](int base) {
        int r[kPer];
        float v[kPer];
        uint8_t m[kPer];
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
            const int s = base + tid * kPer + e;
            r[e] = s < A.B ? ret[s] : -1;
            if (r[e] >= 0 && !index_ok(r[e], A.L, A.status)) r[e] = 0;
        }
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
            v[e] = r[e] >= 0 ? imp[r[e]] : 0.f;
            m[e] = r[e] >= 0 ? mod[r[e]] : 0;
        }
        text = vis = 0;
#pragma unroll
        for (int e = 0; e < kPer; ++e)
            if (r[e] >= 0 && v[e] <= A.tau_eff) {              // Eq. 10: pivots above tau are kept out of merging
                if (m[e] == 0) text |= 1u << e;
                else vis |= 1u << e;
            }
    };
    // the text group comes first: where it ends is needed before the visual group is written
    int n_text = 0, seen_t = 0, seen_v = 0;
    if (A.B > chunk) {
        for (int base = 0; base < A.B; base += chunk) {
            look(base);
            n_text += __popc(text);
        }
        int total;
        block_exclusive_scan(n_text, scratch, total);
        n_text = total;
    }
    for (int base = 0; base < A.B; base += chunk) {
        look(base);
        int tot;                                               // (both counts in one sum: text in the low half, a chunk's at most)
        const int both = block_exclusive_scan(__popc(text) | __popc(vis) << 16, scratch, tot);
        if (A.B <= chunk) n_text = tot & 0xFFFF;
        int pt = seen_t + (both & 0xFFFF), pv = ((n_text + 31) & ~31) + seen_v + (both >> 16);
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
            const int s = base + tid * kPer + e;
            if (text >> e & 1u) slot_out[pt++] = s;
            if (vis >> e & 1u) slot_out[pv++] = s;
        }
        seen_t += tot & 0xFFFF;
        seen_v += tot >> 16;
    }
    if (tid == 0) { A.cand_count[2 * uh] = seen_t; A.cand_count[2 * uh + 1] = seen_v; }
    __syncthreads();
    if (A.copy_here) match_gather_rows<4>(A, uh, nullptr, 0, A.Ctot, tid, blockDim.x);
}

// The preparation of flowmm_match, which is handed the index lists (inside flowmm_compress_layer and flowmm_recompress the
// selection kernel lays everything out itself).  grid = (U*Hkv, 1 + parts), block = 512: blocks y = 0 lay out a head's
// candidates, the others write what the matching kernel reads per token, a slice each.
constexpr int kPrepThreads = 512;
constexpr int kPrepSlice = 8 * kPrepThreads;                   // list entries of such a block: eight loads in flight per thread
static_assert(kPrepSlice % kMtItemRows == 0 && kPrepThreads % kMtItemRows == 0, "a slice is whole tiles, a step as well");
// kPer: pivots of a thread that lays out candidates.
template <int kPer>
__global__ void __launch_bounds__(kPrepThreads) match_prepare_kernel(const MatchPrepArgs A) {
    __shared__ int scratch[33];
    predecessor_done();
    const int uh = blockIdx.x, tid = threadIdx.x;
    if (blockIdx.y == 0) { match_lay_out_candidates<kPer>(A, uh, scratch); return; }
    const int part = blockIdx.y - 1, parts = gridDim.y - 1;
    const int *ret = A.retained + (int64_t)uh * A.B;
    const int *evi = A.evicted + (int64_t)uh * A.E;
    if (A.copy_here) {
        int *rank = A.rank + (int64_t)uh * A.L;
        for (int i0 = part * kPrepSlice; i0 < A.L; i0 += parts * kPrepSlice) {   // entries of the two lists, pivots first
            int tok[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int i = i0 + e * kPrepThreads + tid;
                tok[e] = i < A.B ? ret[i] : i < A.L ? evi[i - A.B] : -1;
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int i = i0 + e * kPrepThreads + tid;
                if (i < A.L && index_ok(tok[e], A.L, A.status)) rank[tok[e]] = i < A.B ? -(i + 2) : i - A.B;
            }
        }
        return;
    }
    const uint8_t *mod = A.modality + (int64_t)(uh / A.Hkv) * A.L;
    for (int j0 = part * kPrepSlice; j0 < A.E; j0 += parts * kPrepSlice) {
        int tok[8];
        uint8_t m[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int j = j0 + e * kPrepThreads + tid;
            tok[e] = j < A.E ? evi[j] : -1;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) m[e] = tok[e] >= 0 && index_ok(tok[e], A.L, A.status) ? mod[tok[e]] : 0;
        if (tid < 2 * kPrepSlice / kMtItemRows) scratch[tid] = 0;
        __syncthreads();
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int j = j0 + e * kPrepThreads + tid, t = (j - j0) / kMtItemRows;
            if (j < A.E) A.evi_mod[(int64_t)uh * A.E + j] = m[e] != 0;
            const bool any_t = __any_sync(0xFFFFFFFFu, j < A.E && m[e] == 0), any_v = __any_sync(0xFFFFFFFFu, j < A.E && m[e] != 0);
            if ((tid & 31) == 0) {
                if (any_t) scratch[2 * t] = 1;
                if (any_v) scratch[2 * t + 1] = 1;
            }
        }
        __syncthreads();
        const int t = j0 / kMtItemRows + tid;
        if (tid < kPrepSlice / kMtItemRows && t < A.n_rt) A.tile_mod[(int64_t)uh * A.n_rt + t] = (uint8_t)(scratch[2 * tid] | scratch[2 * tid + 1] << 1);
        __syncthreads();
    }
}

// The gather step of the preparation as a kernel of its own for long candidate lists, so that many
// CTAs share a head's rows.  grid = (U*Hkv, ceil(Ctot / 64)), block = 256.
__global__ void __launch_bounds__(256) match_gather_kernel(const MatchPrepArgs A) {
    predecessor_done();
    successor_may_start();
    const int lo = blockIdx.y * 64;
    match_gather_rows<4>(A, blockIdx.x, nullptr, lo, min(A.Ctot, lo + 64), threadIdx.x, blockDim.x);
}

struct MatchTcArgs {
    const int *cand_count, *cand_slot, *evicted, *strategy;
    const float *cand_scale;
    const uint8_t *evi_mod, *tile_mod;
    int *match;
    float *match_sim;
    int *status;
    int Hkv, L, E, Ctot, n_rt, n_items;
    const __nv_bfloat16 *k;
    int64_t k_unit, k_head;      // strides in elements
    uint32_t row_bytes;          // stride of the tokens (32 bits: more than 224 rows of 4 GB each are no GPU's)
    FastDiv by_nrt, by_hkv;      // exact division of item numbers by n_rt and of head numbers by Hkv
};

struct MatchItem {
    int u, h, uh, rt, lo, hi, n_text, t0, n_vis;
    bool intra, mixed;
    tcs::TilePlan tp;
};

// What an item's plan reads from global memory; kept apart so that a role can fetch the next item's
// values while it works on the current one.
struct MatchRaw { int uh, u, rt, n_text, n_vis, strategy, tile_mod; };

__device__ __forceinline__ MatchRaw match_raw(const MatchTcArgs &A, int item) {
    MatchRaw r = {0, 0, 0, 0, 0, 1, 0};
    if (item >= A.n_items) return r;
    r.uh = (int)A.by_nrt.div(item); r.rt = item - r.uh * A.n_rt; r.u = (int)A.by_hkv.div(r.uh);
    r.n_text = A.cand_count[2 * r.uh]; r.n_vis = A.cand_count[2 * r.uh + 1];
    r.strategy = A.strategy[r.u];
    r.tile_mod = A.tile_mod[item];
    return r;
}

// Which candidate columns a tile of 256 tokens has to visit: everything in a cross-modal layer or
// when the tile mixes modalities, otherwise only the group of the tile's modality.
template <class S>
__device__ __forceinline__ MatchItem match_plan(const MatchTcArgs &A, const MatchRaw &raw) {
    constexpr int kMtCols = S::kCols;        // candidates per column tile
    MatchItem p;
    p.uh = raw.uh; p.rt = raw.rt; p.u = raw.u; p.h = p.uh - p.u * A.Hkv;
    p.n_text = raw.n_text; p.n_vis = raw.n_vis;
    p.t0 = (p.n_text + 31) & ~31;
    p.intra = raw.strategy == 0;
    const int tm = raw.tile_mod;
    p.mixed = tm == 3;
    const int end_all = p.n_vis > 0 ? p.t0 + p.n_vis : p.n_text;
    if (!p.intra || tm == 3) { p.lo = 0; p.hi = end_all; }
    else if (tm == 1) { p.lo = 0; p.hi = p.n_text; }
    else { p.lo = p.t0; p.hi = p.t0 + p.n_vis; }
    const int cols = p.hi > p.lo ? p.hi - p.lo : 0;
    p.tp.a1 = p.rt * kMtItemRows;                                // first position in the non-pivot list
    p.tp.n_halves = p.tp.a1 + kMtRows < A.E ? 2 : 1;
    p.tp.b1 = p.lo; p.tp.b2 = p.uh; p.tp.b3 = 0;
    p.tp.step1 = kMtCols; p.tp.step2 = 0;
    p.tp.n_tiles = (cols + kMtCols - 1) / kMtCols;
    p.tp.cols_total = cols;
    p.tp.extra = A.cand_scale + (int64_t)p.uh * A.Ctot + p.lo;
    return p;
}
template <class S>
__device__ __forceinline__ MatchItem match_plan(const MatchTcArgs &A, int item) {
    return match_plan<S>(A, match_raw(A, item));
}

// The inner step of the epilogue, written out in PTX so that it stays inside what the tensor core leaves room for:
// a 128 x 256 accumulator is refilled in 1024 clocks, in which the four schedulers issue 4096 warp instructions for its
// 1024 warp-wide elements, and the tensor core's operand reads already take three quarters of the shared-memory
// bandwidth, so the epilogue must not stage anything through shared memory.
// One block of 16 accumulator columns of this thread's row: similarities = accumulators x the candidates' reciprocal
// norms (packed pairs; the norms are the block's only shared-memory reads); each similarity then carries its column in
// its four lowest mantissa bits (15 - column, so that of equal similarities the lower column is the larger number; the
// change is below 2^-19 relative, far inside the margin the decision is judged with); one maximum over the 16 tagged
// values; the block's maximum with the tag cleared is compared with the row's running maximum `best`: a block that
// beats it - strictly, so that an earlier block keeps a tie, and never with NaN (= no candidate there) - replaces it
// and `win` records where it was: 16 x block number + tag.
//   taddr   TMEM address of the block for this warp's lanes        scales   shared address of the block's 16 norms
// (A full share is read 16 columns at a time, match_blocks; where a tile ends or changes group, pairs of blocks with one read of 32.
// The width does not slow the products: sixteen warps read a column of 32 lanes in 0.15 clocks either way.)
#define FLOWMM_MB_MUL2(i, j, k, ti, tj, MASK)                                                                  \
    "mov.b64 t0, {a" #i ", a" #j "};\n\tmul.rn.f32x2 t0, t0, s" #k ";\n\tmov.b64 {a" #i ", a" #j "}, t0;\n\t"    \
    "lop3.b32 a" #i ", a" #i ", " MASK ", " #ti ", 0xEA;\n\t"                                                   \
    "lop3.b32 a" #j ", a" #j ", " MASK ", " #tj ", 0xEA;\n\t"
#define FLOWMM_MB_LDS(OFF)                                     \
    "ld.shared.v2.b64 {s0, s1}, [%3 + " #OFF "];\n\t"          \
    "ld.shared.v2.b64 {s2, s3}, [%3 + " #OFF " + 16];\n\t"     \
    "ld.shared.v2.b64 {s4, s5}, [%3 + " #OFF " + 32];\n\t"     \
    "ld.shared.v2.b64 {s6, s7}, [%3 + " #OFF " + 48];\n\t"
// 16 columns held in registers a<c0> .. a<c15>: products, tags, maximum, comparison with the running maximum;
// WIN = 16 x block number and MASK = 0xFFFFFFF0 held in a register, as asm operand references (the tag-insertion takes
// one immediate only: with the mask as a literal too, each tag would first be moved into a register)
#define FLOWMM_MB_STEP(c0, c1, c2, c3, c4, c5, c6, c7, c8, c9, c10, c11, c12, c13, c14, c15, WIN, MASK)         \
    FLOWMM_MB_MUL2(c0, c1, 0, 15, 14, MASK) FLOWMM_MB_MUL2(c2, c3, 1, 13, 12, MASK) FLOWMM_MB_MUL2(c4, c5, 2, 11, 10, MASK) \
    FLOWMM_MB_MUL2(c6, c7, 3, 9, 8, MASK) FLOWMM_MB_MUL2(c8, c9, 4, 7, 6, MASK) FLOWMM_MB_MUL2(c10, c11, 5, 5, 4, MASK)     \
    FLOWMM_MB_MUL2(c12, c13, 6, 3, 2, MASK) FLOWMM_MB_MUL2(c14, c15, 7, 1, 0, MASK)                             \
    "max.f32 m0, a" #c0 ", a" #c1 ", a" #c2 ";\n\t"                                                             \
    "max.f32 m1, a" #c3 ", a" #c4 ", a" #c5 ";\n\t"                                                             \
    "max.f32 m2, a" #c6 ", a" #c7 ", a" #c8 ";\n\t"                                                             \
    "max.f32 m3, a" #c9 ", a" #c10 ", a" #c11 ";\n\t"                                                           \
    "max.f32 m4, a" #c12 ", a" #c13 ", a" #c14 ";\n\t"                                                          \
    "max.f32 m0, m0, m1, m2;\n\t"                                                                               \
    "max.f32 m3, m3, m4, a" #c15 ";\n\t"                                                                        \
    "max.f32 q0, m0, m3;\n\t"                                                                                   \
    "and.b32 qm, q0, " MASK ";\n\t"                                                                             \
    "setp.gt.f32 p0, qm, %0;\n\t"                                                                               \
    "@p0 mov.b32 %0, qm;\n\t"                                                                                   \
    "@p0 lop3.b32 %1, q0, 15, " WIN ", 0xEA;\n\t"
#define FLOWMM_MB_HEAD                 \
    "{\n\t"                            \
    ".reg .b32 a<32>, qm;\n\t"         \
    ".reg .b64 s<8>, t0;\n\t"          \
    ".reg .f32 m<5>, q0;\n\t"          \
    ".reg .pred p0;\n\t"

// Block number kBlk (16 columns) of the warp's share of the tile.
template <int kBlk>
__device__ __forceinline__ void match_block16(uint32_t taddr, uint32_t scales, float &best, int &win) {
    asm volatile(FLOWMM_MB_HEAD
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {a0, a1, a2, a3, a4, a5, a6, a7, a8, a9, a10, a11, a12, a13, a14, a15}, [%2];\n\t"
        FLOWMM_MB_LDS(0)
        "tcgen05.wait::ld.sync.aligned;\n\t"
        FLOWMM_MB_STEP(0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, "%4", "%5")
        "}"
        : "+f"(best), "+r"(win)
        : "r"(taddr), "r"(scales), "n"(16 * kBlk), "r"(0xFFFFFFF0u)
        : "memory");
}

// Blocks kBlk and kBlk + 1 (32 columns) with one TMEM read.
template <int kBlk>
__device__ __forceinline__ void match_block32(uint32_t taddr, uint32_t scales, float &best, int &win) {
    asm volatile(FLOWMM_MB_HEAD
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {a0, a1, a2, a3, a4, a5, a6, a7, a8, a9, a10, a11, a12, a13, a14, a15, "
        "a16, a17, a18, a19, a20, a21, a22, a23, a24, a25, a26, a27, a28, a29, a30, a31}, [%2];\n\t"
        FLOWMM_MB_LDS(0)
        "tcgen05.wait::ld.sync.aligned;\n\t"
        FLOWMM_MB_STEP(0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, "%4", "%6")
        FLOWMM_MB_LDS(64)
        FLOWMM_MB_STEP(16, 17, 18, 19, 20, 21, 22, 23, 24, 25, 26, 27, 28, 29, 30, 31, "%5", "%6")
        "}"
        : "+f"(best), "+r"(win)
        : "r"(taddr), "r"(scales), "n"(16 * kBlk), "n"(16 * kBlk + 16), "r"(0xFFFFFFF0u)
        : "memory");
}

// Block number kBlk from registers that hold its accumulators already: a share's last two blocks are read together, so that the
// accumulator goes back to the tensor core before they are worked on (112 heads of 8448 tokens against 1690 pivots 1.5 % of the call).
template <int kBlk>
__device__ __forceinline__ void match_block16(const uint32_t *r, uint32_t scales, float &best, int &win) {
    asm volatile(FLOWMM_MB_HEAD
        "mov.b32 a0, %5;\n\tmov.b32 a1, %6;\n\tmov.b32 a2, %7;\n\tmov.b32 a3, %8;\n\tmov.b32 a4, %9;\n\tmov.b32 a5, %10;\n\t"
        "mov.b32 a6, %11;\n\tmov.b32 a7, %12;\n\tmov.b32 a8, %13;\n\tmov.b32 a9, %14;\n\tmov.b32 a10, %15;\n\tmov.b32 a11, %16;\n\t"
        "mov.b32 a12, %17;\n\tmov.b32 a13, %18;\n\tmov.b32 a14, %19;\n\tmov.b32 a15, %20;\n\t"
        "ld.shared.v2.b64 {s0, s1}, [%2];\n\tld.shared.v2.b64 {s2, s3}, [%2 + 16];\n\t"
        "ld.shared.v2.b64 {s4, s5}, [%2 + 32];\n\tld.shared.v2.b64 {s6, s7}, [%2 + 48];\n\t"
        FLOWMM_MB_STEP(0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, "%3", "%4")
        "}"
        : "+f"(best), "+r"(win)
        : "r"(scales), "n"(16 * kBlk), "r"(0xFFFFFFF0u), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]),
          "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
#undef FLOWMM_MB_MUL2
#undef FLOWMM_MB_LDS
#undef FLOWMM_MB_STEP
#undef FLOWMM_MB_HEAD

// Blocks kI .. kN - 1 of the warp's share.  (One TMEM read per block of 16 columns measured a little faster than
// one per 32 columns: the narrower read leaves the compiler more registers around it.)
template <int kN, int kI = 0>
__device__ __forceinline__ void match_blocks(uint32_t taddr, uint32_t scales, float &best, int &win) {
    if constexpr (kI < kN) {
        match_block16<kI>(taddr + 16 * kI, scales + 64 * kI, best, win);
        match_blocks<kN, kI + 1>(taddr, scales, best, win);
    }
}

// Of two (similarity, slot) results the larger similarity wins and equal similarities go to the lower slot
// (slot < 0: no result).
__device__ __forceinline__ bool match_better(float va, int sa, float vb, int sb) {
    return sa >= 0 && (sb < 0 || va > vb || (va == vb && sa < sb));
}

// Squared norm of 64 bf16 elements of a key row in an operand stage (one 128-byte swizzled row: 16-byte units
// XOR-ed with the row index), as packed pairs.
__device__ __forceinline__ float row_half_ssq(uint32_t row_addr, int row) {
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int un = 0; un < 8; ++un) {
        const float4 rawf = tc::lds128(row_addr + ((un ^ (row & 7)) << 4));
        const uint32_t w[4] = {__float_as_uint(rawf.x), __float_as_uint(rawf.y), __float_as_uint(rawf.z), __float_as_uint(rawf.w)};
#pragma unroll
        for (int i = 0; i < 4; ++i) {            // a bf16 is the upper half of the fp32 with the same value
            const float2 x = make_float2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xFFFF0000u));
            acc = tc::ffma2(x, x, acc);
        }
    }
    return acc.x + acc.y;
}

// Persistent kernel, one CTA per SM; item = (unit, head, tile of 256 non-pivots).
constexpr int kMtThreads = tcs::kThreads + 64;
template <class S>
__global__ void __launch_bounds__(kMtThreads, 1)
match_tc_kernel(const __grid_constant__ CUtensorMap cand_map, const MatchTcArgs A) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    constexpr int kMtCols = S::kCols;
    constexpr int kPer = kMtCols / 32;                           // blocks of 16 columns a warp takes of a full tile
    const typename S::Ctx c = S::setup(smem_raw, &cand_map, &cand_map, A.status, 8);
    if (!c.ok) return;
    auto plan = [&](int item) { return match_plan<S>(A, item).tp; };
    if (c.warp == 0) {
        S::template producer<false>(c, nullptr, &cand_map, A.n_items, 0, S::kBStage, plan, A.status);
    } else if (c.warp >= tcs::kThreads / 32) {
        // A warp per half gathers its 128 rows, two to an instruction: lanes 0-15 and 16-31 take 16 bytes each of a row, to where the
        // 128-byte swizzle puts them.  The rows' tokens are fetched an item ahead (rows past the list's end repeat its last).
        const int h = c.warp - tcs::kThreads / 32, odd = c.lane >> 4, unit = c.lane & 15;
        const uint32_t dst = c.a_addr_of(h) + (uint32_t)(unit >> 3) * (tcs::kAHalf / 2) + (uint32_t)odd * 128;
        uint32_t at[4];                                              // rows 2 i + odd, i = 0 .. 3, of a group of eight
#pragma unroll
        for (int i = 0; i < 4; ++i) at[i] = dst + (uint32_t)i * 256 + (uint32_t)(((unit & 7) ^ (2 * i + odd)) << 4);
        int tok[4] = {0, 0, 0, 0}, n = 0;
        auto fetch_tokens = [&](int item) {
            if (item >= A.n_items) return;
            const int uh = (int)A.by_nrt.div(item), j0 = (item - uh * A.n_rt) * kMtItemRows + h * kMtRows + c.lane;
            const int *evi = A.evicted + (int64_t)uh * A.E;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                tok[q] = evi[min(j0 + 32 * q, A.E - 1)];
                if (!index_ok(tok[q], A.L, A.status)) tok[q] = 0;
            }
        };
        fetch_tokens(blockIdx.x);
        bool ok = true;
        for (int item = blockIdx.x; ok && item < A.n_items; item += gridDim.x) {
            const MatchItem p = match_plan<S>(A, item);
            if (!p.tp.empty() && h < p.tp.n_halves) {
                const char *src = reinterpret_cast<const char *>(A.k + p.u * A.k_unit + p.h * A.k_head + unit * 8);
                ok = tc::mbar_wait_warp(c.bar(S::kBarAEmpty + h), (n & 1) ^ 1, c.abort_flag, A.status);
                if (!ok) break;
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const int t = __shfl_sync(0xFFFFFFFFu, tok[q], 2 * i + odd);
                        tc::copy16_async(at[i & 3] + (uint32_t)(q * 32 + (i >> 2) * 8) * 128, src + (uint64_t)((uint32_t)t) * A.row_bytes);
                    }
                fetch_tokens(item + gridDim.x);
                tc::copies_landed();
                __syncwarp();
                if (c.lane == 0) tc::mbar_arrive(c.bar(S::kBarAFull + h));
                ++n;
            } else fetch_tokens(item + gridDim.x);
        }
    } else if (c.warp == 1) {
        S::template mma_issuer<false>(c, A.n_items, plan, A.status);
    } else {
        const int lane = c.lane, row = c.quarter * 32 + lane;
        const int b0 = kPer * c.colhalf;                         // first block of this warp's share of a tile
        const uint32_t wrow = c.epi_addr() + row * 16;          // hand-over slots of this row, by turns
        const uint32_t prow = c.partner_addr() + row * 16;      // the other column half's
        uint32_t turn = 0;
        const uint32_t t_lane = c.tmem_base + c.group * kMtCols + b0 * 16 + ((uint32_t)(c.quarter * 32) << 16);
        int k = 0, bt = 0, n_mine = 0;
        bool ok = true;
        // what an item needs from global memory is fetched one item ahead: its plan values and the token's modality
        auto fetch_mod = [&](const MatchRaw &r, int item) -> int {
            const int j = r.rt * kMtItemRows + c.group * kMtRows + row;
            return item < A.n_items && j < A.E ? A.evi_mod[(int64_t)r.uh * A.E + j] : 0;
        };
        MatchRaw raw_next = match_raw(A, blockIdx.x);
        int mod_next = fetch_mod(raw_next, blockIdx.x);
        for (int item = blockIdx.x; ok && item < A.n_items; item += gridDim.x) {
            const MatchRaw raw = raw_next;
            const int my_mod = mod_next;
            raw_next = match_raw(A, item + gridDim.x);
            mod_next = fetch_mod(raw_next, item + gridDim.x);
            const MatchItem p = match_plan<S>(A, raw);
            const bool active = !p.tp.empty() && c.group < p.tp.n_halves;
            const int j = p.rt * kMtItemRows + c.group * kMtRows + row;      // position in the non-pivot list
            const bool row_masked = p.intra && p.mixed;
            const int *slots = A.cand_slot + (int64_t)p.uh * A.Ctot;
            // Running winner of this row among the warp's columns: its similarity (still times the row's norm, four
            // lowest mantissa bits cleared), the tile it came from, and in `win` the block of 16 columns inside the warp's
            // share of that tile (x 16) with 15 - column inside the block.  Candidates are laid out text group first, each group by ascending
            // slot, so within a group the first maximum is the lowest slot; where a tile visits both groups the text group's
            // winner is set aside when the first visual column comes up: in a cross-modal layer the two meet by
            // (similarity, slot), in an intra-modal one, whose tile then holds tokens of both modalities, the row's modality
            // picks one.  (Masking such a row's columns one by one took half of all epilogue time where a tenth of the tiles
            // were mixed: 28 units x 4 heads of 8448 tokens against 1690 pivots 441 us, this 330.)
            float best = -INFINITY, before = -INFINITY;
            int win = -1, best_tile = 0;
            float val_a = -INFINITY;                                 // the winner set aside
            int slot_a = -1;
            bool parked = p.intra && !row_masked;                    // (one group only)
            float ssq = 0.f;                                         // squared norm of this row's key, this warp's half of it
            auto resolve = [&]() -> int {                            // slot of the running winner
                if (win < 0) return -1;
                const int col = p.lo + best_tile * kMtCols + (b0 + (win >> 4)) * 16 + 15 - (win & 15);
                return index_ok(col, A.Ctot, A.status) ? slots[col] : -1;
            };
            auto park = [&](int t) {
                if (best > before) best_tile = t;                   // the winner may be of this tile's earlier blocks
                slot_a = resolve();
                val_a = best;
                best = -INFINITY; before = -INFINITY; win = -1;
                parked = true;
            };
            if (!active) {
                if (!p.tp.empty()) bt += p.tp.n_tiles;               // keep the B-tile count in step
            } else {
                {   // the token's key row sits in this half's A stage: each of the row's two warps reads one 64-element
                    // half of it for the norm while the first MMAs run, then hands the stage back
                    ok = S::a_wait(c, n_mine, A.status);
                    if (ok) ssq = row_half_ssq(c.a_addr(n_mine) + c.colhalf * (tcs::kAHalf / 2) + row * 128, row);
                    S::a_release(c, n_mine++);
                }
                for (int t = 0; ok && t < p.tp.n_tiles; ++t, ++k, ++bt) {
                    const int col0 = p.lo + t * kMtCols;
                    const int ncols = min(kMtCols, p.hi - col0);
                    ok = S::acc_extra_wait(c, k, bt, A.status);
                    if (!ok) break;
                    const uint32_t scale4 = c.extra(bt);             // reciprocal norms of this tile's candidates
                    const int n_blocks = (ncols + 15) >> 4;
                    const int nb = min(n_blocks - b0, kPer);     // blocks of this warp in this tile (may be <= 0)
                    // block before which the text group's winner is set aside (>= nb: not in this tile)
                    // (splitting a ragged last tile evenly between the row's two warps was measured and is no faster:
                    // the tile's arithmetic, not the longer of its two shares, is what takes the time)
                    const int pk = parked ? kPer : max(0, (p.t0 - (col0 + b0 * 16)) >> 4);
                    const uint32_t sc = scale4 + b0 * 64, tl = t_lane;
                    before = best;
                    if (nb == kPer && pk >= kPer) {
                        match_blocks<kPer - 2>(tl, sc, best, win);
                        uint32_t a[32];
                        tc::tmem_ld32(tl + 16 * (kPer - 2), a);
                        tc::tmem_ld_wait(a);
                        if (t + 1 < p.tp.n_tiles) S::acc_release(c);
                        match_block16<kPer - 2>(a, sc + 64 * (kPer - 2), best, win);
                        match_block16<kPer - 1>(a + 16, sc + 64 * (kPer - 1), best, win);
                        if (t + 1 == p.tp.n_tiles) S::acc_release(c);   // (the norms are safe until the item's last release: Ctx::extra)
                    } else {
                        // (the group boundary is a multiple of 32 columns, the warp's share starts at one: pairs of blocks)
#pragma unroll
                        for (int i = 0; i < kPer; i += 2) {
                            if (i < nb) {
                                if (i == pk) park(t);
                                const bool two = i + 1 < nb;
                                switch (i) {                     // (the block's number is a compile-time constant)
                                    case 0: if (two) match_block32<0>(tl, sc, best, win); else match_block16<0>(tl, sc, best, win); break;
                                    case 2: if (two) match_block32<2>(tl + 32, sc + 128, best, win); else match_block16<2>(tl + 32, sc + 128, best, win); break;
                                    case 4: if (two) match_block32<4>(tl + 64, sc + 256, best, win); else match_block16<4>(tl + 64, sc + 256, best, win); break;
                                    default: if (two) match_block32<6>(tl + 96, sc + 384, best, win); else match_block16<6>(tl + 96, sc + 384, best, win); break;
                                }
                            }
                        }
                        S::acc_release(c);
                    }
                    if (best > before) best_tile = t;                // the winner moved into this tile
                }
            }
            // (after a wait that ran out the results are garbage, but the two meeting points below are still
            // kept so that the partner warp is never left waiting; the first one tells both warps, and the loop
            // ends for both right after them)
            // this warp's result for the row: similarity (still times the row's norm) and pivot slot
            int slot = -1;
            if (ok && active) {
                slot = resolve();
                if (row_masked) {                                        // the group of the row's own modality counts
                    if (my_mod == 0 && parked) { best = val_a; slot = slot_a; }
                    if (my_mod != 0 && !parked) slot = -1;
                } else if (match_better(val_a, slot_a, best, slot)) { best = val_a; slot = slot_a; }
            }
            // the upper column half hands its result and its half of the norm to the lower one, which owns the row's output
            if (c.colhalf == 1) tc::sts128(wrow + turn, best, __int_as_float(slot), ssq, 0.f);
            ok = !S::pair_meet(c, !ok);                            // (both warps of a row go on, or neither)
            if (c.colhalf == 0 && ok) {
                const float4 other = tc::lds128(prow + turn);
                if (match_better(other.x, __float_as_int(other.y), best, slot)) { best = other.x; slot = __float_as_int(other.y); }
                ssq += other.z;
                if (j < A.E) {
                    float sim = 0.f;
                    if (slot >= 0 && ssq > 0.f) sim = best * rsqrtf(ssq);
                    A.match[(int64_t)p.uh * A.E + j] = slot;
                    A.match_sim[(int64_t)p.uh * A.E + j] = sim;
                }
            }
            turn ^= kMtRows * 16;                                  // (the next meeting keeps the upper half from a slot that is still being read)
        }
    }
    S::teardown(c);
}

}  // namespace flowmm
