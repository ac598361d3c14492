// Weighted merge (Eq. 5) + compaction, gather form, over the rows of a head in slot order (merge_lists.cuh): each slot's pivot
// row, then its members'.
//
// Persistent warps take windows of A.win rows: a warp merges the slots that begin in its window, to their ends, and leaves
// out a long slot; pieces of such slots are spread over the warps of the head's windows, or are items behind the windows, store
// fp32 partial sums, and the last one to arrive adds them up in order.  Sums are in fixed order throughout.
// Rows come through shared memory: a lane copies its own bytes of each row (cp.async; lanes 0-15 the K row's, 16-31 the V
// row's), in groups of a few rows, three of which are on their way while one is worked on, and reads back what it has copied
// itself, so no lane waits for another.  The window's tokens and weights wait in shared memory, fetched a window ahead.
// Bound by HBM in large calls, by the chain of a warp's groups in small ones (groups without a pivot are summed side by side, 4 to 9 %
// there).  A warp per slot or piece of 64 members, as before, spent 340 instructions on each beside 61 per row; here a window costs
// about 300 and a row 24.  Us, so and now: 64 heads of 2158 rows with 1444 slots 49 / 25, 200 of 2508 with 1662 165 / 74, 112 of
// 8448 with 1690 126 / 101 (5.7 TB/s), 128 of 33 792 with 1690 421 / 400 (5.8 TB/s), 8 of 33 792 51 / 43.
#pragma once
#include "common.cuh"
#include "merge_lists.cuh"
#include "tc_common.cuh"

namespace flowmm {
namespace mrow {

constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kChunk = 128;                                  // rows whose tokens and weights wait in shared memory
constexpr int kMaxWin = 64;                                  // rows of a window at most
static_assert(kChunk >= kMaxWin + kPiece, "the last slot that begins in a window ends among them");
constexpr int kStages = 4;
constexpr uint32_t kEntryBytes = kChunk * 8;
__host__ __device__ constexpr int group_rows(int bytes) { return bytes == 32 ? 2 : 4; }
__host__ __device__ constexpr uint32_t warp_bytes(int bytes) { return kEntryBytes + kStages * group_rows(bytes) * 32 * bytes; }

// kBytes: of a K row (a V row) per lane.
template <typename T, int kBytes>
__global__ void __launch_bounds__(kThreads, 3) merge_rows_kernel(const MergeArgs A, unsigned n_items, unsigned n_piece_items, int *status, const FastDiv by_win, const FastDiv by_heads, const FastDiv by_hkv) {
    constexpr int V = kBytes / (int)sizeof(T), kWords = kBytes / 4, kGroup = group_rows(kBytes);
    constexpr uint32_t kRow = 32 * kBytes, kStage = kGroup * kRow;
    extern __shared__ __align__(128) uint8_t mrow_smem[];
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    const uint32_t ents = tc::smem_u32(mrow_smem) + warp * warp_bytes(kBytes), bufs = ents + kEntryBytes + lane * kBytes;
    predecessor_done();
    const bool is_v = lane >= 16;
    const int c0 = (lane & 15) * V;
    const int64_t row_bytes = (is_v ? A.vs[2] : A.ks[2]) * (int64_t)sizeof(T);   // (two rows may be more than 4 GB apart)
    const unsigned n_warps = gridDim.x * kWarps;

    // (head, number) of a piece that is an item: all heads' first ones, then all heads' second ones, ...  Most possible pieces are none, and the
    // ones that are find warps without a window so (merge_window() leaves some).
    auto piece_of = [&](unsigned g) {
        const unsigned p = by_heads.div(g - n_items);
        return make_int2((int)(g - n_items - p * by_heads.d), (int)p);
    };
    // what an item needs from global memory, a word of 32 rows per register
    struct Item { int2 count; int first, x[4], y[4]; };
    auto fetch = [&](unsigned g, Item &it) {
        if (g >= n_items) {
            if (g - n_items < n_piece_items) it.count = A.row_count[piece_of(g).x];
            return;
        }
        const int uh = (int)by_win.div(g), w = (int)(g - (unsigned)uh * (unsigned)A.n_win);
        if (A.rows) {
            it.count = A.row_count[uh];
            it.first = A.first_slot[g];
        } else {
            it.count = make_int2(A.B, 0);
            it.first = w * A.win;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int r = w * A.win + 32 * k + lane;
            it.x[k] = kRowPivot; it.y[k] = 0;                        // (past the rows: as if another slot began)
            if (r < A.L) {
                if (A.rows) { const int2 e = A.rows[(int64_t)uh * A.L + r]; it.x[k] = e.x; it.y[k] = e.y; }
                else if (r < A.B) it.x[k] = A.retained[(int64_t)uh * A.B + r] | kRowPivot;
            }
        }
    };
    auto read_words = [&](uint32_t at, uint32_t (&w)[kWords]) {
        if constexpr (kWords == 2) tc::lds64(at, w[0], w[1]);
        else {
#pragma unroll
            for (int q = 0; q < kWords; q += 4) {
                const float4 f = tc::lds128(at + 4 * q);
                w[q] = __float_as_uint(f.x); w[q + 1] = __float_as_uint(f.y); w[q + 2] = __float_as_uint(f.z); w[q + 3] = __float_as_uint(f.w);
            }
        }
    };
    auto unpack = [&](const uint32_t (&w)[kWords], float (&x)[V]) {
        if constexpr (sizeof(T) == 2) {
#pragma unroll
            for (int i = 0; i < kWords; ++i) { x[2 * i] = __uint_as_float(w[i] << 16); x[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u); }
        } else {
#pragma unroll
            for (int i = 0; i < kWords; ++i) x[i] = __uint_as_float(w[i]);
        }
    };
    auto store = [&](T *dst, const uint32_t (&w)[kWords]) {
        if constexpr (kWords == 2) *reinterpret_cast<uint2 *>(dst) = make_uint2(w[0], w[1]);
        else {
#pragma unroll
            for (int q = 0; q < kWords; q += 4) reinterpret_cast<uint4 *>(dst)[q / 4] = make_uint4(w[q], w[q + 1], w[q + 2], w[q + 3]);
        }
    };

    // the slot being merged
    float acc[V], wsum = 0.f;
    uint32_t pivot[kWords];
    int members = 0;
    // Rows [r0, r1) of those in shared memory, in order: pivot() before a pivot's row is taken, member rows added up.
    auto add = [&](const uint32_t (&raw)[kWords], float w) {
        float x[V];
        unpack(raw, x);
        const float2 w2 = make_float2(w, w);
#pragma unroll
        for (int e = 0; e < V; e += 2) {
            const float2 a = tc::ffma2(w2, make_float2(x[e], x[e + 1]), make_float2(acc[e], acc[e + 1]));
            acc[e] = a.x; acc[e + 1] = a.y;
        }
        wsum += w;
    };
    // lo, hi: which of the rows are pivots
    auto walk = [&](const char *src, int r0, int r1, unsigned long long lo, unsigned long long hi, auto &&on_pivot) {
        const int n_groups = (r1 - r0 + kGroup - 1) / kGroup;
        auto issue = [&](int gi) {
            const int lo = r0 + gi * kGroup;
#pragma unroll
            for (int q = 0; q < kGroup; ++q)
                if (lo + q < r1) {
                    int tok = __float_as_int(tc::lds32(ents + (lo + q) * 8)) & kRowToken;
                    if (!index_ok(tok, A.L, status)) tok = 0;
                    const uint32_t dst = bufs + (gi & (kStages - 1)) * kStage + q * kRow;
                    const char *from = src + tok * row_bytes;
                    if constexpr (kBytes == 8) tc::copy8_async(dst, from);
                    else tc::copy16_async(dst, from);
                    if constexpr (kBytes == 32) tc::copy16_async(dst + 16, from + 16);
                }
            tc::copies_commit();
        };
#pragma unroll
        for (int gi = 0; gi < kStages - 1; ++gi) issue(gi);
        for (int gi = 0; gi < n_groups; ++gi) {
            issue(gi + kStages - 1);                                 // (where the group before this one was)
            tc::copies_wait<kStages - 1>();
            const int ra = r0 + gi * kGroup;
            const unsigned pivots = (unsigned)(ra == 0 ? lo : ra < 64 ? lo >> ra | hi << (64 - ra) : hi >> (ra - 64)) & ((1u << kGroup) - 1);
            if (pivots == 0 && ra + kGroup <= r1) {                  // members alone: side by side up to the sums
                uint32_t raw[kGroup][kWords];
                float w[kGroup];
#pragma unroll
                for (int q = 0; q < kGroup; ++q) {
                    w[q] = tc::lds32(ents + (ra + q) * 8 + 4);
                    read_words(bufs + (gi & (kStages - 1)) * kStage + q * kRow, raw[q]);
                }
#pragma unroll
                for (int q = 0; q < kGroup; ++q) add(raw[q], w[q]);
                members += kGroup;
                continue;
            }
#pragma unroll
            for (int q = 0; q < kGroup; ++q) {
                const int r = ra + q;
                if (r >= r1) break;
                uint32_t ex, ey, raw[kWords];
                tc::lds64(ents + r * 8, ex, ey);
                read_words(bufs + (gi & (kStages - 1)) * kStage + q * kRow, raw);
                if ((int)ex < 0) {
                    on_pivot();
#pragma unroll
                    for (int i = 0; i < kWords; ++i) pivot[i] = raw[i];
#pragma unroll
                    for (int e = 0; e < V; ++e) acc[e] = 0.f;
                    wsum = 0.f;
                    members = 0;
                } else {
                    add(raw, __uint_as_float(ey));
                    ++members;
                }
            }
        }
    };

    // A warp's first window is given, the others are drawn from a shared counter, two ahead (or taken with a stride, without one).
    Item it;
    unsigned g = blockIdx.x * kWarps + warp, g_next, g_after;
    // Pieces in a row go to the warps of one block after the other: with eight real ones on the warps of one block 32 heads of 1500 rows with
    // 64 long slots took 20.4 us, so 18.9; 12 of 4992 with 249 slots 18.6, 17.5.
    if (g >= n_items) {
        const unsigned blocks = min(n_piece_items, n_warps - n_items) / kWarps, o = g - n_items;
        if (o < blocks * kWarps) g = n_items + o % kWarps * blocks + o / kWarps;
    }
    auto draw = [&](unsigned from) { return A.ticket ? (lane == 0 ? n_warps + atomicAdd(A.ticket, 1u) : 0u) : from + n_warps; };
    fetch(g, it);
    g_next = __shfl_sync(0xFFFFFFFFu, draw(g), 0);
    for (; g < n_items + n_piece_items; g = g_next, g_next = __shfl_sync(0xFFFFFFFFu, g_after, 0)) {
        g_after = draw(g_next);
        const bool is_window = g < n_items;
        const int2 piece = is_window ? make_int2(0, 0) : piece_of(g);
        const int uh = is_window ? (int)by_win.div(g) : piece.x, w = is_window ? (int)(g - (unsigned)uh * (unsigned)A.n_win) : piece.y;   // window, or piece
        const int u = (int)by_hkv.div(uh), h = uh - u * A.Hkv;
        const int left = is_window ? it.count.x - w * A.win : 0, n_pieces = is_window && n_piece_items != 0 ? 0 : it.count.y;   // left: rows from the window's first on
        int slot = it.first;
        // the rows of a chunk go to shared memory; which of them begin a slot, or lie past the last row
        unsigned long long lo, hi;
        {
            uint32_t begins[4];
            __syncwarp();                                            // (the rows before have been read)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int r = 32 * k + lane, v = r < left ? it.x[k] : kRowPivot;
                begins[k] = __ballot_sync(0xFFFFFFFFu, v < 0);
                tc::sts64(ents + r * 8, (uint32_t)v, (uint32_t)it.y[k]);
            }
            __syncwarp();
            lo = begins[0] | (unsigned long long)begins[1] << 32;
            hi = begins[2] | (unsigned long long)begins[3] << 32;
        }
        fetch(g_next, it);
        const char *src = reinterpret_cast<const char *>((is_v ? static_cast<const T *>(A.v) + u * A.vs[0] + h * A.vs[1]
                                                               : static_cast<const T *>(A.k) + u * A.ks[0] + h * A.ks[1]) + c0);
        const int n_own = min(A.win, left);
        const unsigned long long own = n_own <= 0 ? 0ull : lo & (~0ull >> (64 - n_own));
        if (own) {
            const int last = 63 - __clzll((long long)own);
            const int r0 = __ffsll((long long)own) - 1;
            int r1 = last;         // a long slot, which is the window's last, is left to its pieces
            if (!(__float_as_int(tc::lds32(ents + last * 8)) & kRowLong)) {
                const unsigned long long next = last == 63 ? 0ull : lo & (~0ull << (last + 1));
                r1 = next ? __ffsll((long long)next) - 1 : hi ? 64 + __ffsll((long long)hi) - 1 : kChunk;
            }
            T *out = is_v ? static_cast<T *>(A.v_out) + u * A.vos[0] + h * A.vos[1] : static_cast<T *>(A.k_out) + u * A.kos[0] + h * A.kos[1];
            const int64_t ostride = is_v ? A.vos[2] : A.kos[2];
            out += c0 + (slot - 1) * ostride;                        // (the first pivot steps to the first slot)
            bool open = false;
            auto finish = [&]() {
                if (members == 0) { store(out, pivot); return; }     // nothing merged in: the pivot row, bit for bit
                const float inv = 1.f / (1.f + wsum);
                float x[V];
                unpack(pivot, x);
#pragma unroll
                for (int e = 0; e < V; ++e) x[e] = (x[e] + acc[e]) * inv;
                uint32_t o[kWords];
                if constexpr (sizeof(T) == 2) {
#pragma unroll
                    for (int i = 0; i < kWords; ++i) {
                        const __nv_bfloat162 b = __floats2bfloat162_rn(x[2 * i], x[2 * i + 1]);
                        o[i] = *reinterpret_cast<const uint32_t *>(&b);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < kWords; ++i) o[i] = __float_as_uint(x[i]);
                }
                store(out, o);
            };
            auto begin = [&]() {
                if (open) finish();
                open = true;
                out += ostride;
            };
            walk(src, r0, r1, lo, hi, begin);
            if (open) finish();
        }
        for (int p = w; p < n_pieces; p += is_window ? A.n_win : A.max_parts) {   // this window's share of the head's pieces, or the piece
            const int4 d = A.pieces[(int64_t)uh * A.max_parts + p];
            __syncwarp();
#pragma unroll
            for (int k = 0; k < kPiece / 32; ++k) {
                const int r = 32 * k + lane;
                if (r < d.z) { const int2 e = A.rows[(int64_t)uh * A.L + d.y + r]; tc::sts64(ents + r * 8, (uint32_t)e.x, (uint32_t)e.y); }
            }
            __syncwarp();
#pragma unroll
            for (int e = 0; e < V; ++e) acc[e] = 0.f;
            wsum = 0.f;
            members = 0;
            walk(src, 0, d.z, 0ull, 0ull, []() {});
            float *rec = A.partial + ((int64_t)uh * A.max_parts + d.w) * (2 * A.D + 4);
#pragma unroll
            for (int e = 0; e < V; ++e) rec[(is_v ? A.D : 0) + c0 + e] = acc[e];
            if (lane == 0) rec[2 * A.D] = wsum;
            __threadfence();                                         // was this the slot's last piece to arrive?
            __syncwarp();
            int prev = 0;
            if (lane == 0) prev = atomicAdd(&A.slot_done[(int64_t)uh * A.B + d.x], 1);
            prev = __shfl_sync(0xFFFFFFFFu, prev, 0);
            const int *poff = A.part_off + (int64_t)uh * (A.B + 1);
            if (prev == poff[d.x + 1] - poff[d.x] - 1) {
                __threadfence();
                merge_finish_slot<T>(A, uh, d.x, lane);
            }
        }
    }
}

}  // namespace mrow
}  // namespace flowmm
