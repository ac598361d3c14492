// Tensor-core path of the scoring step (Eq. 8 with the softmax of Eq. 4, and the masses of
// Eq. 7) for bf16 inputs, head_dim 128 and a window of 32, 64 or 128 tokens.
//
// The proxy attention needs every row's softmax normaliser before any column can be summed, so
// the keys are streamed twice:
//   pass 1  S = Q_group . K^T with the G*W proxy rows of a KV head as accumulator lanes (two
//           halves of 128 rows per item) and 256 keys per tile: each thread keeps the running
//           maximum and the exp-sums over text and over visual keys of its own row (no
//           cross-thread traffic), which also give the cross-modal mass;
//   pass 2  S^T = K . Q_group^T with keys as the lanes (two halves of 128 keys per item) and the
//           proxy rows as columns: each thread owns one key, recomputes its logits, normalises
//           them with the per-column constants of pass 1 and sums along its row, which is
//           exactly the key's importance.
// Both passes run on tcgen05 with TMA-fed operands; logits never leave TMEM / registers.
#pragma once
#include "common.cuh"
#include "tc_stream.cuh"

namespace flowmm {

struct ScoreTcArgs {
    float4 *row_part;            // [UH*GW, n_part] (max, exp-sum over text keys, exp-sum over visual keys, -) per proxy row and run that its keys are in, log2 domain
    int n_part;                  // runs a head's key tiles can be spread over
    const float4 *row_all;       // nullptr, or [UH*GW] the records of row_part joined to one per row, which pass 2 then reads
    const uint8_t *modality;     // [U, L]
    float *importance;           // [UH, L]
    float *cross_part;           // [U*Hq, W] share of a proxy row's mass that falls on keys of the other modality
    int *status;
    int Hq, Hkv, G, W, L, GW;
    int q_rows, n_qt;            // pass 1: proxy rows of an item (256, or 128: one half), tiles of so many over the G*W rows
    int n_runs1;                 // pass 1: runs that the key tiles of all heads are cut into
    FastDiv by_grid1, by_grid2, by_hkv, by_rt, by_rt2, by_tiles;   // exact divisions by the passes' grids, Hkv, n_rt, n_rt2, n_tiles1
    int n_rt;                    // 256-key tiles of a head
    int keys2, n_rt2;            // pass 2: keys of an item (256, or 128: one half), items of a head
    int a_heads, b_heads;        // query heads one A box (pass 1) / B box (pass 2) delivers
    int n_tiles1, n_items2;      // key tiles and items of all heads
    float scale_log2;
};

// max of 32 values with three-input maxima
__device__ __forceinline__ float max32(const uint32_t (&a)[32]) {
    float v[32], m12[12];
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(a[i]);
#pragma unroll
    for (int i = 0; i < 10; ++i) m12[i] = tc::max3(v[3 * i], v[3 * i + 1], v[3 * i + 2]);
    m12[10] = v[30]; m12[11] = v[31];
    const float a0 = tc::max3(m12[0], m12[1], m12[2]), a1 = tc::max3(m12[3], m12[4], m12[5]);
    const float a2 = tc::max3(m12[6], m12[7], m12[8]), a3 = tc::max3(m12[9], m12[10], m12[11]);
    return fmaxf(tc::max3(a0, a1, a2), a3);
}

__device__ __forceinline__ float2 pair_of(const uint32_t (&a)[32], int j) { return make_float2(__uint_as_float(a[j]), __uint_as_float(a[j + 1])); }
// Sum of 2^(a * scale - mx) over 32 accumulator columns; every fourth exponential on the FMA pipe, two at a time.
__device__ __forceinline__ float exp_sum32(const uint32_t (&a)[32], float scale_log2, float mx) {
    const float2 neg2 = make_float2(-mx, -mx), sc2 = make_float2(scale_log2, scale_log2);
    float2 a01 = make_float2(0.f, 0.f), a23 = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 32; j += 8) {
        const float2 x01 = tc::ffma2(pair_of(a, j), sc2, neg2), x23 = tc::ffma2(pair_of(a, j + 2), sc2, neg2);
        const float2 x45 = tc::ffma2(pair_of(a, j + 4), sc2, neg2), x67 = tc::ffma2(pair_of(a, j + 6), sc2, neg2);
        const float2 pf = tc::ex2_fma2(x67);
        a01 = tc::fadd2(a01, make_float2(tc::ex2(x01.x), tc::ex2(x01.y)));
        a23 = tc::fadd2(a23, make_float2(tc::ex2(x23.x), tc::ex2(x23.y)));
        a01 = tc::fadd2(a01, make_float2(tc::ex2(x45.x), tc::ex2(x45.y)));
        a23 = tc::fadd2(a23, pf);
    }
    return (a01.x + a01.y) + (a23.x + a23.y);
}

// The exponentials of the scoring and flow epilogues, written out in PTX so that they cost what they must and no more: 32
// accumulator columns become probabilities in place, multiply-adds as packed pairs, every fourth exponential (two of each
// eight, neighbours) on the FMA pipe instead of the exp2 unit, which sets these steps' pace.
#define FLOWMM_EX_FMA(i, j, ADD)                                                           \
    "mov.b64 x0, {%" #i ", %" #j "};\n\t"                                                  \
    "fma.rn.f32x2 x0, x0, sc, " ADD ";\n\t"                                                \
    "mov.b64 {%" #i ", %" #j "}, x0;\n\t"
#define FLOWMM_EX_E(i) "ex2.approx.ftz.f32 %" #i ", %" #i ";\n\t"
// 2^x for the pair on the FMA pipe: x clamped at -125, n = round(x) by the 1.5 * 2^23 trick, 2^f on f = x - n in [-0.5, 0.5]
// by a degree-4 polynomial (own least-squares fit at Chebyshev nodes with the constant fixed at 1: relative error 3.6e-6), n
// added to the exponent field.
#define FLOWMM_EX_POLY(i, j)                                                          \
    "max.f32 %" #i ", %" #i ", 0fC2FA0000;\n\t"                                        \
    "max.f32 %" #j ", %" #j ", 0fC2FA0000;\n\t"                                        \
    "mov.b64 x0, {%" #i ", %" #j "};\n\t"                                              \
    "add.rn.f32x2 x1, x0, kmg;\n\t"          /* t = x + 1.5 * 2^23 */                  \
    "mov.b64 {f0, f1}, x1;\n\t"                                                       \
    "sub.rn.f32x2 x1, x1, kmg;\n\t"          /* n */                                   \
    "sub.rn.f32x2 x0, x0, x1;\n\t"           /* f */                                   \
    "fma.rn.f32x2 x1, kc4, x0, kc3;\n\t"                                              \
    "fma.rn.f32x2 x1, x1, x0, kc2;\n\t"                                               \
    "fma.rn.f32x2 x1, x1, x0, kc1;\n\t"                                               \
    "fma.rn.f32x2 x1, x1, x0, kone;\n\t"                                              \
    "mov.b64 {%" #i ", %" #j "}, x1;\n\t"                                              \
    "mad.lo.s32 %" #i ", f0, 8388608, %" #i ";\n\t"                                    \
    "mad.lo.s32 %" #j ", f1, 8388608, %" #j ";\n\t"
#define FLOWMM_EX_DECL                                                                 \
    ".reg .b64 x0, x1, sc, kmg, kc1, kc2, kc3, kc4, kone;\n\t"                          \
    ".reg .b32 f0, f1;\n\t"                                                           \
    "mov.b64 kmg, 0x4B4000004B400000;\n\t"      /* 12582912.0f twice */                \
    "mov.b64 kone, 0x3F8000003F800000;\n\t"                                           \
    "mov.b64 kc1, 0x3F3170613F317061;\n\t"      /* 0.69312102 */                       \
    "mov.b64 kc2, 0x3E75FCD43E75FCD4;\n\t"      /* 0.24022228 */                       \
    "mov.b64 kc3, 0x3D650E813D650E81;\n\t"      /* 0.05592204 */                       \
    "mov.b64 kc4, 0x3C1E78073C1E7807;\n\t"      /* 0.00967217 */
#define FLOWMM_EX_ALL                                                                                                             \
    FLOWMM_EX_E(0) FLOWMM_EX_E(1) FLOWMM_EX_E(2) FLOWMM_EX_E(3) FLOWMM_EX_E(4) FLOWMM_EX_E(5) FLOWMM_EX_POLY(6, 7)                  \
    FLOWMM_EX_E(8) FLOWMM_EX_E(9) FLOWMM_EX_E(10) FLOWMM_EX_E(11) FLOWMM_EX_E(12) FLOWMM_EX_E(13) FLOWMM_EX_POLY(14, 15)            \
    FLOWMM_EX_E(16) FLOWMM_EX_E(17) FLOWMM_EX_E(18) FLOWMM_EX_E(19) FLOWMM_EX_E(20) FLOWMM_EX_E(21) FLOWMM_EX_POLY(22, 23)          \
    FLOWMM_EX_E(24) FLOWMM_EX_E(25) FLOWMM_EX_E(26) FLOWMM_EX_E(27) FLOWMM_EX_E(28) FLOWMM_EX_E(29) FLOWMM_EX_POLY(30, 31)
#define FLOWMM_EX_HW                                                                                                              \
    FLOWMM_EX_E(0) FLOWMM_EX_E(1) FLOWMM_EX_E(2) FLOWMM_EX_E(3) FLOWMM_EX_E(4) FLOWMM_EX_E(5) FLOWMM_EX_E(6) FLOWMM_EX_E(7)          \
    FLOWMM_EX_E(8) FLOWMM_EX_E(9) FLOWMM_EX_E(10) FLOWMM_EX_E(11) FLOWMM_EX_E(12) FLOWMM_EX_E(13) FLOWMM_EX_E(14) FLOWMM_EX_E(15)    \
    FLOWMM_EX_E(16) FLOWMM_EX_E(17) FLOWMM_EX_E(18) FLOWMM_EX_E(19) FLOWMM_EX_E(20) FLOWMM_EX_E(21) FLOWMM_EX_E(22) FLOWMM_EX_E(23)  \
    FLOWMM_EX_E(24) FLOWMM_EX_E(25) FLOWMM_EX_E(26) FLOWMM_EX_E(27) FLOWMM_EX_E(28) FLOWMM_EX_E(29) FLOWMM_EX_E(30) FLOWMM_EX_E(31)
#define FLOWMM_EX_REGS(a)                                                                                                          \
    "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]), "+r"(a[8]), "+r"(a[9]), "+r"(a[10]), \
        "+r"(a[11]), "+r"(a[12]), "+r"(a[13]), "+r"(a[14]), "+r"(a[15]), "+r"(a[16]), "+r"(a[17]), "+r"(a[18]), "+r"(a[19]), "+r"(a[20]), \
        "+r"(a[21]), "+r"(a[22]), "+r"(a[23]), "+r"(a[24]), "+r"(a[25]), "+r"(a[26]), "+r"(a[27]), "+r"(a[28]), "+r"(a[29]), "+r"(a[30]), \
        "+r"(a[31])

// a = 2^(a * scale - mx), in place (all 32 with the same mx).  exp2_32_exact: by the exp2 unit alone, within 2^-22 of the value.
#define FLOWMM_EX2_32(EXPS)                                                                                                       \
    asm volatile(                                                                                                                 \
        "{\n\t" FLOWMM_EX_DECL ".reg .b64 ng;\n\t"                                                                                 \
        "mov.b64 sc, {%32, %32};\n\t"                                                                                             \
        "mov.b64 ng, {%33, %33};\n\t"                                                                                             \
        FLOWMM_EX_FMA(0, 1, "ng") FLOWMM_EX_FMA(2, 3, "ng") FLOWMM_EX_FMA(4, 5, "ng") FLOWMM_EX_FMA(6, 7, "ng")                     \
        FLOWMM_EX_FMA(8, 9, "ng") FLOWMM_EX_FMA(10, 11, "ng") FLOWMM_EX_FMA(12, 13, "ng") FLOWMM_EX_FMA(14, 15, "ng")               \
        FLOWMM_EX_FMA(16, 17, "ng") FLOWMM_EX_FMA(18, 19, "ng") FLOWMM_EX_FMA(20, 21, "ng") FLOWMM_EX_FMA(22, 23, "ng")             \
        FLOWMM_EX_FMA(24, 25, "ng") FLOWMM_EX_FMA(26, 27, "ng") FLOWMM_EX_FMA(28, 29, "ng") FLOWMM_EX_FMA(30, 31, "ng")             \
        EXPS "}"                                                                                                                  \
        : FLOWMM_EX_REGS(a)                                                                                                       \
        : "f"(scale_log2), "f"(-mx))
__device__ __forceinline__ void exp2_32(uint32_t (&a)[32], float scale_log2, float mx) { FLOWMM_EX2_32(FLOWMM_EX_ALL); }
__device__ __forceinline__ void exp2_32_exact(uint32_t (&a)[32], float scale_log2, float mx) { FLOWMM_EX2_32(FLOWMM_EX_HW); }
#undef FLOWMM_EX2_32
__device__ __forceinline__ float sum32(const uint32_t (&a)[32]) {
    float2 s0 = pair_of(a, 0), s1 = pair_of(a, 2);
#pragma unroll
    for (int j = 4; j < 32; j += 4) {
        s0 = tc::fadd2(s0, pair_of(a, j));
        s1 = tc::fadd2(s1, pair_of(a, j + 2));
    }
    s0 = tc::fadd2(s0, s1);
    return s0.x + s0.y;
}
// The sums over a chunk's text keys and over its visual keys (bit set in `vis`), each a sum of its own: as the difference of all and the
// others a small one would lose its digits.  `masks`: shared address of sixteen float4, entry n the bits of n as 0.f / -1.f: two
// multiply-adds with the mask, where tests per key would cost three instructions each.
__device__ __forceinline__ void sums32_by(const uint32_t (&a)[32], uint32_t vis, uint32_t masks, float &on_text, float &on_vis) {
    float2 t01 = make_float2(0.f, 0.f), t23 = t01, v01 = t01, v23 = t01;
#pragma unroll
    for (int j = 0; j < 32; j += 4) {
        const float4 v = tc::lds128(masks + (vis >> j & 15u) * 16);
        const float2 x01 = pair_of(a, j), x23 = pair_of(a, j + 2), m01 = make_float2(v.x, v.y), m23 = make_float2(v.z, v.w);
        t01 = tc::fadd2(t01, tc::ffma2(x01, m01, x01)); t23 = tc::fadd2(t23, tc::ffma2(x23, m23, x23));   // (x or 0)
        v01 = tc::ffma2(x01, m01, v01); v23 = tc::ffma2(x23, m23, v23);
    }
    on_text = (t01.x + t01.y) + (t23.x + t23.y);
    on_vis = -((v01.x + v01.y) + (v23.x + v23.y));
}

// Run `r` of n: tiles [run_start(r), run_start(r + 1)) of the n_tiles of all heads; and the run that holds tile x.
__device__ __forceinline__ int run_start(int n_tiles, int n, int r) { return (int)((int64_t)n_tiles * r / n); }
__device__ __forceinline__ int run_of(const ScoreTcArgs &A, int x) {
    const uint64_t v = ((uint64_t)x + 1) * (uint32_t)A.n_runs1 - 1;
    return v >> 32 ? (int)(v / (uint32_t)A.n_tiles1) : (int)A.by_tiles.div((uint32_t)v);
}
__device__ __forceinline__ int runs_of_head(const ScoreTcArgs &A, int uh) { return run_of(A, (uh + 1) * A.n_rt - 1) - run_of(A, uh * A.n_rt) + 1; }

// A proxy row's statistics over some keys: running maximum, exp-sums over the text and over the visual keys.
struct RowStats { float m, t, v; };
__device__ __forceinline__ RowStats join(const RowStats &a, const RowStats &b) {
    RowStats r;
    r.m = fmaxf(a.m, b.m);
    const float wa = tc::ex2(a.m - r.m), wb = tc::ex2(b.m - r.m);
    r.t = a.t * wa + b.t * wb;
    r.v = a.v * wa + b.v * wb;
    return r;
}

// ---------------------------------------------------------------------------------------------
// Pass 1.  The 256-key tiles of all heads, one head's behind the other's, are cut into equal runs; a CTA takes a run for one tile
// of 256 proxy rows, or of 128 (CTAs next to each other share a run, whose keys the second of them finds in L2).  item = a run's part of one
// head.  Whole heads or equal chunks of them as items left SMs idle in the last round.  The whole call, us, so and now: 112 heads of
// 2176 tokens, 224 rows 116.1 / 111.9; of 8448, 448 rows 867 / 851; 112 caches of 640 rows 97.9 / 95.6; 80 heads of 7906, 512
// rows 419 / 394; 128 of 33 792 2947 / 2904.
// The exp-sums are kept by modality of the key: what pass 2 had to split off its probabilities, per query head and with a sum
// over the warp for each, costs nothing here where a warp's 64 keys of a tile are of one modality and seen by every row, as
// nearly always (images are runs of tokens): one of the two sums grows, and they change places when the modality does.  128
// heads of 33 792 tokens, 512 rows each, at the power cap: this pass 605 -> 640 us, pass 2 790 -> 620, the call 3095 -> 2930.
// (With a choice by modality at every chunk this pass took 690: that code is for the other tiles.)
// The four warps that share a row join their statistics in shared memory at the end of an item.
// A wait that runs out changes no warp's way through the items (what follows is garbage, in bounds, and reported), so that no
// warp is left alone at a meeting.
template <class S>
__global__ void __launch_bounds__(tcs::kThreads, 1)
score_stats_tc_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                      const ScoreTcArgs A) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const typename S::Ctx c = S::setup(smem_raw, &q_map, &k_map, A.status, 0, 16);
    if (!c.ok) return;
    const int run = (int)blockIdx.x / A.n_qt, qt = (int)blockIdx.x - run * A.n_qt;
    const int t_lo = run_start(A.n_tiles1, A.n_runs1, run), t_hi = run_start(A.n_tiles1, A.n_runs1, run + 1);
    const int uh_lo = (int)A.by_rt.div(t_lo), n_loop = ((int)A.by_rt.div(t_hi - 1) - uh_lo + 1) * gridDim.x;   // the roles count items blockIdx.x, blockIdx.x + gridDim.x, ...
    auto plan = [&](int item) {
        tcs::TilePlan p;
        const int uh = uh_lo + (int)A.by_grid1.div(item), u = (int)A.by_hkv.div(uh), h = uh - u * A.Hkv, head0 = uh * A.n_rt;
        const int t0 = max(t_lo, head0) - head0, t1 = min(t_hi, head0 + A.n_rt) - head0;
        p.a1 = 0; p.a2 = h * A.G + qt * (A.q_rows / A.W); p.a3 = u;
        p.h1 = 0; p.h2 = tcs::kRows / A.W;
        p.n_halves = A.q_rows > tcs::kRows && qt * A.q_rows + tcs::kRows < A.GW ? 2 : 1;
        p.b1 = t0 * S::kCols; p.b2 = h; p.b3 = u; p.step1 = S::kCols; p.step2 = 0;
        p.cols_total = min(A.L, t1 * S::kCols) - p.b1;
        p.n_tiles = t1 - t0;
        p.extra = nullptr;
        return p;
    };
    const uint32_t a_bytes = (uint32_t)A.a_heads * A.W * 256u;
    if (c.warp == 0) {
        S::producer(c, &q_map, &k_map, blockIdx.x + n_loop, a_bytes, S::kBStage, plan, A.status);
    } else if (c.warp == 1) {
        S::template mma_issuer<false>(c, blockIdx.x + n_loop, plan, A.status);
    } else {
        // all sixteen warps drain one accumulator at a time: a warp owns 32 lanes x a quarter of the columns of
        // BOTH halves, so the tensor core refills one half while the other is being read
        static_assert(S::kCols == 256, "two words of 32 keys per warp and tile");
        constexpr uint32_t kMeetWarp = 32 * 12, kMeetBytes = 4 * 6 * kMeetWarp;    // (max, text, visual) of a warp's rows; a turn's
        static_assert(2 * kMeetBytes + 256 <= tcs::kExtraSlots * S::kExtraBytes + tcs::kEpiBytes, "scratch of the meetings");
        const int row_in_half = c.quarter * 32 + c.lane, colq = (c.warp - 2) >> 2;
        const uint32_t meet = c.base + S::kSmemExtra + (uint32_t)c.quarter * 6 * kMeetWarp + (uint32_t)c.lane * 12;
        const uint32_t masks = c.base + S::kSmemExtra + 2 * kMeetBytes;
        const int te = threadIdx.x - 64;
        if (te < 64) tc::sts32(masks + te * 4, (te >> 2) >> (te & 3) & 1 ? -1.f : 0.f);
        tcs::named_barrier(5, 32 * tcs::kEpiWarps);
        int kh[2] = {0, 0};
        uint32_t turn = 0;
        bool ok = true;
        // modalities of this warp's 64 keys of a tile, a tile ahead (keys past the prompt count with its last token, so that they
        // make no chunk mixed)
        const uint8_t *mod = A.modality;
        uint8_t mod0 = 0, mod1 = 0;
        // A warp's two chunks of a tile are neighbours, or, where a head ends inside the tile, every fourth, so that the four warps of a
        // row share what there is (112 heads of 2176 tokens and of 640: the whole call 111.2 -> 110.7 and 78.8 -> 77.9 us).
        auto fetch_mod = [&](int kb) {
            const bool full = kb + S::kCols <= A.L;
            const int key = kb + (full ? colq * 64 : colq * 32) + c.lane;
            mod0 = mod[min(key, A.L - 1)];
            mod1 = mod[min(key + (full ? 32 : 128), A.L - 1)];
        };
        auto first_mod = [&](int item) {
            if (item >= (int)blockIdx.x + n_loop) return;
            const tcs::TilePlan p = plan(item);
            mod = A.modality + (int64_t)p.b3 * A.L;
            fetch_mod(p.b1);
        };
        first_mod(blockIdx.x);
        // runs of a head before this CTA's: none, unless it begins inside the head
        int part = run - run_of(A, uh_lo * A.n_rt), uh = uh_lo;
        for (int item = blockIdx.x; item < (int)blockIdx.x + n_loop; item += gridDim.x, ++uh, part = 0) {
            const tcs::TilePlan p = plan(item);
            RowStats st[2] = {{kNegBig, 0.f, 0.f}, {kNegBig, 0.f, 0.f}};
            bool swapped = false;                                        // st[].t belongs to the visual keys and st[].v to the text keys
            for (int t = 0; t < p.n_tiles; ++t) {
                const int kb = p.b1 + t * S::kCols;
                const int ncols = min(S::kCols, p.cols_total - t * S::kCols);
                const uint32_t vis0 = __ballot_sync(0xFFFFFFFFu, mod0 != 0), vis1 = __ballot_sync(0xFFFFFFFFu, mod1 != 0);
                fetch_mod(kb + S::kCols);                                // (past the item's last tile: of no use)
                // the common tile: every row sees all of its keys, and this warp's are of one modality
                const bool plain = kb + S::kCols <= A.L - A.W + 1 && vis0 == vis1 && (vis0 == 0u || vis0 == 0xFFFFFFFFu);
                if (plain && (vis0 != 0u) != swapped) {
                    swapped = !swapped;
#pragma unroll
                    for (int h = 0; h < 2; ++h) { const float x = st[h].t; st[h].t = st[h].v; st[h].v = x; }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (h >= p.n_halves) continue;
                    if (ok) ok = S::acc_wait_h(c, h, kh[h], A.status);
                    ++kh[h];
                    const int r0 = qt * A.q_rows + h * tcs::kRows;
                    auto release = [&]() { if (ok) S::acc_release_h(c, h); };
                    if (r0 + c.quarter * 32 >= A.GW) release();
                    else if (plain) {
                        S::for_each_chunk_h(c, h, 2 * colq, 1, 2, [&](int, int, uint32_t (&acc)[32]) {
                            const float mx = fmaxf(max32(acc) * A.scale_log2, st[h].m);
                            const float all = exp_sum32(acc, A.scale_log2, mx), carry = tc::ex2(st[h].m - mx);
                            st[h].t = st[h].t * carry + all;
                            st[h].v *= carry;
                            st[h].m = mx;
                        }, release);
                    } else {
                        const int pa = A.L - A.W + ((r0 + row_in_half) & (A.W - 1));   // last key this proxy row may see (the window is 32, 64 or 128 rows)
                        const bool full = ncols == S::kCols;
                        S::for_each_chunk_h(c, h, full ? 2 * colq : colq, full ? 1 : 4, full ? 2 : (((ncols + 31) >> 5) - colq + 3) >> 2,
                                            [&](int i, int ch, uint32_t (&acc)[32]) {
                            const int last = pa - (kb + ch * 32);        // this row sees the chunk's keys 0 .. last
                            uint32_t vis = i ? vis1 : vis0;
                            asm volatile("" : "+r"(vis));                // (or what the sum below needs of it is formed for the plain tiles as well)
                            float mx;
                            if (kb + ch * 32 + 32 > A.L - A.W + 1) {
#pragma unroll
                                for (int j = 0; j < 32; ++j) acc[j] = j <= last ? acc[j] : __float_as_uint(-INFINITY);
                                mx = fmaxf(max32(acc) * A.scale_log2, st[h].m);
                                exp2_32_exact(acc, A.scale_log2, mx);           // (0 where masked; the polynomial would leave 2^-125)
                            } else {
                                mx = fmaxf(max32(acc) * A.scale_log2, st[h].m);
                                exp2_32(acc, A.scale_log2, mx);
                            }
                            const float carry = tc::ex2(st[h].m - mx);
                            float on_text = 0.f, on_vis = 0.f;
                            if (vis == 0u) on_text = sum32(acc);
                            else if (vis == 0xFFFFFFFFu) on_vis = sum32(acc);
                            else sums32_by(acc, vis, masks, on_text, on_vis);
                            st[h].t = st[h].t * carry + (swapped ? on_vis : on_text);
                            st[h].v = st[h].v * carry + (swapped ? on_text : on_vis);
                            st[h].m = mx;
                        }, release);
                    }
                }
            }
            if (swapped)
#pragma unroll
                for (int h = 0; h < 2; ++h) { const float x = st[h].t; st[h].t = st[h].v; st[h].v = x; }
            first_mod(item + gridDim.x);
            // the four warps of a row join their quarters of the columns: warp 0 the first half's rows, warp 1 the second's
            // (two sets of slots by turns: the next meeting keeps writers from slots that are still being read)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (colq != h) {
                    const uint32_t at = meet + turn + (uint32_t)(h * 3 + ((colq - h - 1) & 3)) * kMeetWarp;
                    tc::sts32(at, st[h].m); tc::sts32(at + 4, st[h].t); tc::sts32(at + 8, st[h].v);
                }
            ok = !__any_sync(0xFFFFFFFFu, tcs::meet_vote(1 + c.quarter, 128, !ok));   // (the vote: for the compiler, which then knows the warp to be of one mind)
            const int r = qt * A.q_rows + colq * tcs::kRows + row_in_half;
            if (colq < p.n_halves && r < A.GW) {
                RowStats s = colq == 0 ? st[0] : st[1];
#pragma unroll
                for (int w = 0; w < 3; ++w) {
                    const uint32_t at = meet + turn + (uint32_t)(colq * 3 + w) * kMeetWarp;
                    const RowStats o = {tc::lds32(at), tc::lds32(at + 4), tc::lds32(at + 8)};
                    s = join(s, o);
                }
                A.row_part[((int64_t)uh * A.GW + r) * A.n_part + part] = make_float4(s.m, s.t, s.v, 0.f);
            }
            turn ^= kMeetBytes;
        }
    }
    S::teardown(c);
}

// Packs the modality map: word w of a unit holds keys 32 w .. 32 w + 31 (bit set = visual; keys past the prompt: 0).
__global__ void pack_modality_kernel(const uint8_t *modality, int L, int n_words, uint32_t *bits) {
    const int u = blockIdx.x, w = blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    predecessor_done();
    if (w >= n_words) return;
    const int key = 32 * w + lane;
    const uint32_t word = __ballot_sync(0xFFFFFFFFu, key < L && modality[(int64_t)u * L + key] != 0);
    if (lane == 0) bits[(int64_t)u * n_words + w] = word;
}

// Joins the records of a row to one, where pass 2 would have to read many of them for each of its heads: kLanes lanes share a row
// and read its records together.
template <int kLanes>
__global__ void score_combine_kernel(const ScoreTcArgs A, int n_rows, float4 *row_all) {
    predecessor_done();
    const int i = blockIdx.x * (blockDim.x / kLanes) + threadIdx.x / kLanes, sub = threadIdx.x % kLanes;
    const bool on = i < n_rows;
    const int n = runs_of_head(A, on ? i / A.GW : 0);
    const float4 *part = A.row_part + (int64_t)i * A.n_part;
    float mx = kNegBig, t = 0.f, v = 0.f;
    if (on) {
#pragma unroll 4
        for (int c = sub; c < n; c += kLanes) mx = fmaxf(mx, part[c].x);
    }
#pragma unroll
    for (int o = kLanes / 2; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
    if (on) {
#pragma unroll 4
        for (int c = sub; c < n; c += kLanes) {
            const float4 p = part[c];
            const float w = exp2f(p.x - mx);
            t += p.y * w; v += p.z * w;
        }
    }
#pragma unroll
    for (int o = kLanes / 2; o > 0; o >>= 1) {
        t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
        v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    }
    if (sub == 0 && on) row_all[i] = make_float4(mx, t, v, 0.f);
}

// The common case of pass 2's inner step: 32 accumulator columns of this thread's key (32 proxy rows of one query head),
// probability = 2^(logit * scale + row constant), with the row constants read as packed pairs from shared memory; their sum is
// added to the packed pair `sum`.  No causal mask: chunks that need it take the general path.
//   a  the chunk's accumulators     negc  shared address of its 32 row constants
// (three phases, so that no exponential's result is needed before the last one has been issued: logits in place,
// exponentials in place, then a tree of packed additions)
#define FLOWMM_CS_X(q, i0, i1, i2, i3)                                                      \
    "ld.shared.v2.b64 {n0, n1}, [%33 + " #q " * 16];\n\t"                                   \
    FLOWMM_EX_FMA(i0, i1, "n0") FLOWMM_EX_FMA(i2, i3, "n1")
#define FLOWMM_CS_P(k, i0, i1) "mov.b64 p" #k ", {%" #i0 ", %" #i1 "};\n\t"
#define FLOWMM_CS_A(d, x, y) "add.rn.f32x2 p" #d ", p" #x ", p" #y ";\n\t"
#define FLOWMM_CS(EXPS)                                                                                                            \
    asm volatile(                                                                                                                 \
        "{\n\t" FLOWMM_EX_DECL ".reg .b64 n0, n1, p<16>;\n\t"                                                                      \
        "mov.b64 sc, {%34, %34};\n\t"                                                                                             \
        FLOWMM_CS_X(0, 0, 1, 2, 3) FLOWMM_CS_X(1, 4, 5, 6, 7) FLOWMM_CS_X(2, 8, 9, 10, 11) FLOWMM_CS_X(3, 12, 13, 14, 15)           \
        FLOWMM_CS_X(4, 16, 17, 18, 19) FLOWMM_CS_X(5, 20, 21, 22, 23) FLOWMM_CS_X(6, 24, 25, 26, 27) FLOWMM_CS_X(7, 28, 29, 30, 31) \
        EXPS                                                                                                                      \
        FLOWMM_CS_P(0, 0, 1) FLOWMM_CS_P(1, 2, 3) FLOWMM_CS_P(2, 4, 5) FLOWMM_CS_P(3, 6, 7) FLOWMM_CS_P(4, 8, 9)                    \
        FLOWMM_CS_P(5, 10, 11) FLOWMM_CS_P(6, 12, 13) FLOWMM_CS_P(7, 14, 15) FLOWMM_CS_P(8, 16, 17) FLOWMM_CS_P(9, 18, 19)          \
        FLOWMM_CS_P(10, 20, 21) FLOWMM_CS_P(11, 22, 23) FLOWMM_CS_P(12, 24, 25) FLOWMM_CS_P(13, 26, 27) FLOWMM_CS_P(14, 28, 29)     \
        FLOWMM_CS_P(15, 30, 31)                                                                                                   \
        FLOWMM_CS_A(0, 0, 1) FLOWMM_CS_A(2, 2, 3) FLOWMM_CS_A(4, 4, 5) FLOWMM_CS_A(6, 6, 7) FLOWMM_CS_A(8, 8, 9)                    \
        FLOWMM_CS_A(10, 10, 11) FLOWMM_CS_A(12, 12, 13) FLOWMM_CS_A(14, 14, 15)                                                   \
        FLOWMM_CS_A(0, 0, 2) FLOWMM_CS_A(4, 4, 6) FLOWMM_CS_A(8, 8, 10) FLOWMM_CS_A(12, 12, 14)                                   \
        FLOWMM_CS_A(0, 0, 4) FLOWMM_CS_A(8, 8, 12)                                                                                \
        FLOWMM_CS_A(0, 0, 8)                                                                                                      \
        "add.rn.f32x2 %32, %32, p0;\n\t"                                                                                          \
        "}"                                                                                                                       \
        : FLOWMM_EX_REGS(a), "+l"(sum)                                                                                            \
        : "r"(negc), "f"(scale_log2)                                                                                              \
        : "memory")
__device__ __forceinline__ void colsum_chunk32(uint32_t (&a)[32], uint32_t negc, float scale_log2, uint64_t &sum) { FLOWMM_CS(FLOWMM_EX_ALL); }
// (all exponentials by the exp2 unit)
__device__ __forceinline__ void colsum_chunk32_exact(uint32_t (&a)[32], uint32_t negc, float scale_log2, uint64_t &sum) { FLOWMM_CS(FLOWMM_EX_HW); }
#undef FLOWMM_CS
#undef FLOWMM_CS_X
#undef FLOWMM_CS_P
#undef FLOWMM_CS_A
#undef FLOWMM_EX_FMA
#undef FLOWMM_EX_E
#undef FLOWMM_EX_POLY
#undef FLOWMM_EX_DECL
#undef FLOWMM_EX_ALL
#undef FLOWMM_EX_HW
#undef FLOWMM_EX_REGS

// ---------------------------------------------------------------------------------------------
// Pass 2.  item = (unit*head, tile of 256 keys, or of 128, on which all sixteen epilogue warps work, where items are few); the B stream is the head group's proxy rows.  A CTA takes a run of
// consecutive items, so that proxy rows that fit the B stages (up to 512) are loaded once per head, not once per item.
// Row constants -(max + log2 sum) - exp2(logit + constant) is the softmax probability - are formed from pass 1's statistics by
// the epilogue warps when the run comes to another head; the CTA with a head's first tile also writes its rows' cross-modal shares.
// Bound by the epilogue (four warps per scheduler, the exp2 unit at 0.69 of its rate, 0.56 before the masses went to pass 1): a
// chunk is read while the one before it is worked on, an accumulator is handed back as soon as its last chunk is in registers,
// and no vote or shuffle stands between: 197 -> 152 instructions per chunk of 32 columns.  (Three or four words a thread of
// what belongs to the item are spilled around the chunks; unrolling two chunks instead of four leaves one, and is 1 % slower.)
template <class S, bool kSplit>
__global__ void __launch_bounds__(tcs::kThreads, 1)
score_colsum_tc_kernel(const __grid_constant__ CUtensorMap k_map, const __grid_constant__ CUtensorMap q_map,
                       const ScoreTcArgs A) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    // kSplit (A.keys2 == 128): one half per item, whose columns the two groups of warps share
    typename S::Ctx c = S::setup(smem_raw, &k_map, &q_map, A.status, 0, kSplit ? 8 : 4);
    if (!c.ok) return;
    const int share = kSplit ? c.group : 0, part_of = c.group * 2 + c.colhalf;   // which of a column half's chunks; which of a key's partial sums
    if (kSplit) c.group = 0;
    const int g_lo = (int)((int64_t)A.n_items2 * blockIdx.x / gridDim.x), g_hi = (int)((int64_t)A.n_items2 * (blockIdx.x + 1) / gridDim.x);
    const int n_loop = (g_hi - g_lo) * gridDim.x;                   // the roles count items blockIdx.x, blockIdx.x + gridDim.x, ...
    auto plan = [&](int item) {
        tcs::TilePlan p;
        const int g = g_lo + (int)A.by_grid2.div(item), uh = (int)A.by_rt2.div(g), kt = g - uh * A.n_rt2;
        const int u = (int)A.by_hkv.div(uh), h = uh - u * A.Hkv;
        p.a1 = kt * A.keys2; p.a2 = h; p.a3 = u;
        p.h1 = tcs::kRows; p.h2 = 0;
        p.n_halves = A.keys2 > tcs::kRows && p.a1 + tcs::kRows < A.L ? 2 : 1;
        p.b1 = 0; p.b2 = h * A.G; p.b3 = u; p.step1 = 0; p.step2 = S::kCols / A.W;
        p.cols_total = A.GW;
        p.n_tiles = (A.GW + S::kCols - 1) / S::kCols;
        p.reuse_b = p.n_tiles <= S::kBStages && kt > 0 && g > g_lo;
        p.keep_b = p.n_tiles <= S::kBStages && kt + 1 < A.n_rt2 && g + 1 < g_hi;
        p.extra = nullptr;
        return p;
    };
    const uint32_t b_bytes = (uint32_t)A.b_heads * A.W * 256u;
    if (c.warp == 0) {
        S::producer(c, &k_map, &q_map, blockIdx.x + n_loop, tcs::kAHalf, b_bytes, plan, A.status);
    } else if (c.warp == 1) {
        S::template mma_issuer<true>(c, blockIdx.x + n_loop, plan, A.status);
    } else {
        // scratch: two sets of row constants by turns (up to 1024 rows), then the hand-over slots of the row halves, two by turns
        constexpr uint32_t kConstBytes = 4096, kXch = S::kSmemEpi + 2 * kConstBytes, kXchPart = tcs::kRows * 4;
        static_assert(2 * kConstBytes + 2 * 4 * kXchPart <= tcs::kEpiBytes, "scratch");
        const int lane = c.lane, row = c.quarter * 32 + lane, te = threadIdx.x - 64;
        const uint32_t xch = c.base + kXch + (uint32_t)part_of * kXchPart + (uint32_t)row * 4;
        int k = 0;
        bool ok = true;
        // the run's items one after the other: (unit u, KV head uh, its tile kt) step by step instead of by divisions, which
        // together with the rest of an item's start took a tenth of the epilogue's time
        const int n_tiles = (A.GW + S::kCols - 1) / S::kCols;
        int uh = (int)A.by_rt2.div(g_lo), kt = g_lo - uh * A.n_rt2, u = (int)A.by_hkv.div(uh), hk = uh - u * A.Hkv;
        uint32_t slot = 0, consts = c.base + S::kSmemEpi + kConstBytes;
        uint32_t both = 0;                                           // which words of 32 proxy tokens are of both modalities
        for (int g = g_lo; g < g_hi; ++g) {
            const int uh0 = uh, kt0 = kt;                            // this item
            if (g == g_lo || kt0 == 0) {                             // a new head: its row constants
                consts ^= (c.base + S::kSmemEpi) ^ (c.base + S::kSmemEpi + kConstBytes);
                const int n_rec = A.row_all ? 1 : runs_of_head(A, uh0);
                const uint8_t *proxy_mod = A.modality + (int64_t)(u + 1) * A.L - A.W;
                uint8_t of_lane[4];
#pragma unroll
                for (int w = 0; w < 4; ++w) of_lane[w] = proxy_mod[min(32 * w, A.W - 32) + lane];   // (the window is 32, 64 or 128 rows)
                for (int r = te; r < A.GW; r += 32 * tcs::kEpiWarps) {
                    const int64_t i0 = (int64_t)uh0 * A.GW + r;
                    const float4 *rec = A.row_all ? A.row_all + i0 : A.row_part + i0 * A.n_part;
                    RowStats s = {kNegBig, 0.f, 0.f};
                    for (int i = 0; i < n_rec; i += 8) {             // eight records on their way together
                        float4 o[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) o[e] = i + e < n_rec ? rec[i + e] : make_float4(kNegBig, 0.f, 0.f, 0.f);
                        const float m0 = s.m;
#pragma unroll
                        for (int e = 0; e < 8; ++e) s.m = fmaxf(s.m, o[e].x);
                        const float w0 = exp2f(m0 - s.m);
                        s.t *= w0; s.v *= w0;
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const float w = exp2f(o[e].x - s.m);
                            s.t += o[e].y * w; s.v += o[e].z * w;
                        }
                    }
                    const float z = s.t + s.v;
                    tc::sts32(consts + r * 4, -(s.m + log2f(z)));
                    if (kt0 == 0) {                                  // (one CTA per head)
                        const bool vis = proxy_mod[r & (A.W - 1)] != 0;
                        A.cross_part[((int64_t)u * A.Hq + hk * A.G) * A.W + r] = (vis ? s.t : s.v) / z;
                    }
                }
                both = 0;
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    const uint32_t vis = __ballot_sync(0xFFFFFFFFu, of_lane[w] != 0);
                    if (vis != 0u && vis != 0xFFFFFFFFu) both |= 1u << w;
                }
                // (the set written was read two heads ago, and every warp has been through the meeting of the head between)
                tcs::named_barrier(9, 32 * tcs::kEpiWarps);
            }
            if (++kt == A.n_rt2) {                                    // the next item
                kt = 0; ++uh;
                if (++hk == A.Hkv) { hk = 0; ++u; }
            }
            const int key0 = kt0 * A.keys2 + c.group * tcs::kRows;
            if (key0 >= A.L) continue;                               // no keys in this half
            const int key = key0 + row;
            const bool masked_tile = key0 + tcs::kRows > A.L - A.W + 1;   // some (key, proxy row) pair is masked
            const int first_proxy = A.L - A.W;
            uint64_t sum2 = 0;                                       // a packed pair of partial sums
            float imp = 0.f;
            // A wait that runs out changes no lane's way through the items (what follows is garbage, in bounds, and reported): the
            // reads of tensor memory and the meetings stay the whole warp's without a vote on every wait, which took 5 % (320
            // units of 8 heads, 512 proxy rows, 33 792 tokens 16.65 ms, 17.5 with the vote).  pair_meet tells all lanes.
            for (int t = 0; t < n_tiles; ++t) {
                const int ncols = min(S::kCols, A.GW - t * S::kCols);
                if (!S::takes_part(c, ncols)) continue;
                ok = ok && S::quad_extra_wait_lanes(c, k, -1, A.status);
                ++k;
                constexpr int kPerC = S::kCols / 64;                 // 32-column chunks a warp takes of a full tile
                int ch0 = kPerC * c.colhalf, n_ch = min((ncols + 31) >> 5, ch0 + kPerC) - ch0;   // >= 1
                if (kSplit) {
                    ch0 += share * (kPerC / 2);
                    n_ch = min(n_ch - share * (kPerC / 2), kPerC / 2);
                    if (n_ch <= 0) { S::quad_release(c); continue; }
                }
                const uint32_t nc = consts + (uint32_t)(t * S::kCols + ch0 * 32) * 4;
                if (!masked_tile && both == 0u) {
                    uint32_t a[2][32];
                    tc::tmem_ld32(S::acc_addr(c, ch0), a[0]);
#pragma unroll
                    for (int i = 0; i < kPerC; ++i) {
                        if (i >= n_ch) break;
                        tc::tmem_ld_wait(a[i & 1]);
                        if (i + 1 < kPerC && i + 1 < n_ch) tc::tmem_ld32(S::acc_addr(c, ch0 + i + 1), a[(i + 1) & 1]);
                        else S::quad_release(c);
                        colsum_chunk32(a[i & 1], nc + i * 128, A.scale_log2, sum2);
                    }
                    continue;
                }
                if (!masked_tile) {
                    // proxy tokens of both modalities, whose share a few rows can make up: by the exp2 unit alone (asking for it at every
                    // chunk of every call costs 4 % of the pass)
#pragma unroll 1
                    for (int i = 0; i < n_ch; ++i) {
                        uint32_t acc[32];
                        tc::tmem_ld32(S::acc_addr(c, ch0 + i), acc);
                        tc::tmem_ld_wait(acc);
                        if (i + 1 == n_ch) S::quad_release(c);
                        if (both >> (((ch0 + i) * 32 & (A.W - 1)) >> 5) & 1u) colsum_chunk32_exact(acc, nc + i * 128, A.scale_log2, sum2);
                        else colsum_chunk32(acc, nc + i * 128, A.scale_log2, sum2);
                    }
                    continue;
                }
                for (int i = 0; i < n_ch; ++i) {
                    const int a0 = (t * S::kCols + (ch0 + i) * 32) & (A.W - 1);   // the chunk's first proxy token
                    uint32_t acc[32];
                    tc::tmem_ld32(S::acc_addr(c, ch0 + i), acc);
                    tc::tmem_ld_wait(acc);
                    float s4[4] = {0.f, 0.f, 0.f, 0.f};              // (one sum over all rows would lose the small ones)
#pragma unroll
                    for (int q4 = 0; q4 < 8; ++q4) {
                        const float4 n4 = tc::lds128(nc + (i * 8 + q4) * 16);
                        const float nn[4] = {n4.x, n4.y, n4.z, n4.w};
#pragma unroll
                        for (int j = 0; j < 4; ++j) {                // causal mask inside the window, and keys >= L
                            const float e = tc::ex2(fmaf(__uint_as_float(acc[4 * q4 + j]), A.scale_log2, nn[j]));
                            s4[j] += key <= first_proxy + a0 + 4 * q4 + j ? e : 0.f;
                        }
                    }
                    imp += (s4[0] + s4[1]) + (s4[2] + s4[3]);
                }
                S::quad_release(c);
            }
            imp += __uint_as_float((uint32_t)sum2) + __uint_as_float((uint32_t)(sum2 >> 32));
            // the two column halves of a key meet (or their four shares): the others hand their partial sums to the first (kept even
            // after a wait ran out, so that no partner warp is left waiting).  Two sets of slots by turns: the next meeting keeps the
            // others from slots that are still being read.
            const bool owner = c.colhalf == 0 && share == 0;
            if (!owner) tc::sts32(xch + slot, imp);
            ok = !(kSplit ? tcs::meet_vote(1 + c.quarter, 128, !ok) : S::pair_meet(c, !ok));
            if (owner && ok && key < A.L) {
                float sum = imp + tc::lds32(xch + slot + kXchPart);
                if (kSplit) sum += tc::lds32(xch + slot + 2 * kXchPart) + tc::lds32(xch + slot + 3 * kXchPart);
                A.importance[(int64_t)uh0 * A.L + key] = sum / (float)A.G;   // group mean
            }
            slot ^= 4 * kXchPart;
        }
    }
    S::teardown(c);
}

}  // namespace flowmm
