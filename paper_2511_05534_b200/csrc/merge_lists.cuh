// The merge / compaction stage.
#pragma once
#include "common.cuh"

namespace flowmm {

// ---------------------------------------------------------------------------------------------
// Merge stage.  The match array maps non-pivot j to a slot (or -1).  The members of every slot
// are needed in a fixed order, so the non-pivot positions j are sorted by slot, stably
// (ascending j inside a slot).  What comes out is the sequence of a head's rows in slot order: each slot's
// pivot, then its members, with token position and Eq. 5 weight; slot s begins at row off[s] + s, off[s] being the
// number of members of the slots before it.  The merge kernel (merge_rows.cuh) takes the sequence a window of rows at a time.
// A slot of more than kPiece members is left out there: it is cut into pieces of kPiece, so that many warps share it and no sum is
// a longer chain than that.
// ---------------------------------------------------------------------------------------------
constexpr int kPiece = 64;

struct CsrArgs {
    const int *match;        // [UH, E]
    const int *evicted;      // [UH, E]
    const float *match_sim;  // [UH, E]
    int *sort_a, *sort_b;    // [UH, E] ping-pong buffers of non-pivot positions
    const int *retained;     // [UH, B]
    int2 *rows;              // [UH, B + E] (token, weight bits) of the head's rows in slot order; pivots with kRowPivot, of a long slot with kRowLong
    int2 *row_count;         // [UH] (rows, pieces of long slots)
    int *off;                // [UH, B+1] first member of each slot in the sorted order
    int *first_slot;         // [UH, n_win] first slot that begins in a window of `win` rows, for windows in which one does
    int *part_off;           // [UH, B+1] first piece of each slot (long slots only)
    int4 *pieces;            // [UH, max_parts] (slot, first row, rows, number of the piece)
    unsigned *ticket;        // work counter of the merge kernel, cleared here
    int *slot_done;          // [UH, B] pieces of a slot that have stored their partial sums, cleared here
    int B, E, n_pass, max_parts, merge_mode, win, n_win;
};
constexpr int kRowPivot = (int)0x80000000u, kRowLong = 1 << 30, kRowToken = kRowLong - 1;

__device__ __forceinline__ int csr_key(int m, int B) { return m < 0 ? B : m; }   // dropped tokens sort last

constexpr int kCsrBits = 6, kCsrBins = 1 << kCsrBits;      // digit width of the sort

// Lanes of the warp that hold the same digit as this one, among the valid lanes: a vote per bit and as many logic
// operations (the match instruction gives the same set, but its unit is slow and shared by the SM's warps).
__device__ __forceinline__ uint32_t digit_peers(int digit, bool valid) {
    uint32_t mine = __ballot_sync(0xFFFFFFFFu, valid);
#pragma unroll
    for (int b = 0; b < kCsrBits; ++b) {
        const uint32_t vote = __ballot_sync(0xFFFFFFFFu, (digit >> b) & 1);
        mine &= ((digit >> b) & 1) ? vote : ~vote;
    }
    return mine;
}

// What the merge kernel needs beside the members' rows: the pivots' rows and the windows' first slots, of the slots [s_lo, s_hi) ...
// off[s] = first member of slot s (s <= B).
template <int kThreads>
__device__ __forceinline__ void csr_write_pivots(const CsrArgs &A, int uh, const int *off, int s_lo, int s_hi) {
    const int *ret = A.retained + (int64_t)uh * A.B;
    int2 *rows = A.rows + (int64_t)uh * (A.B + A.E);
    int *first_slot = A.first_slot + (int64_t)uh * A.n_win;
    for (int s = s_lo + threadIdx.x; s < s_hi; s += kThreads) {
        const int row = off[s] + s;
        rows[row] = make_int2(ret[s] | kRowPivot | (off[s + 1] - off[s] > kPiece ? kRowLong : 0), 0);
        for (int w = s == 0 ? 0 : (off[s - 1] + s - 1) / A.win + 1; w <= row / A.win; ++w) first_slot[w] = s;
        A.slot_done[(int64_t)uh * A.B + s] = 0;
    }
}
// ... and the head's pieces of long slots.
template <int kThreads>
__device__ __forceinline__ void csr_write_pieces(const CsrArgs &A, int uh, const int *off, int *scratch) {
    const int tid = threadIdx.x;
    int *part_off = A.part_off + (int64_t)uh * (A.B + 1);
    int4 *pieces = A.pieces + (int64_t)uh * A.max_parts;
    int longest = 0, seen = 0;
    for (int s = tid; s < A.B; s += kThreads) longest = max(longest, off[s + 1] - off[s]);
    const bool any = __syncthreads_or(longest > kPiece);             // (mostly none: then there is nothing to add up)
    for (int base = 0; base <= A.B; base += kThreads) {
        const int s = base + tid;
        int n = 0, np = 0, total = 0, part = 0;
        if (s < A.B) {
            n = off[s + 1] - off[s];
            np = n > kPiece ? (n + kPiece - 1) / kPiece : 0;
        }
        if (any) part = seen + block_exclusive_scan(np, scratch, total);
        if (s <= A.B) part_off[s] = part;
        for (int q = 0; q < np; ++q) pieces[part + q] = make_int4(s, off[s] + s + 1 + q * kPiece, min(kPiece, n - q * kPiece), part + q);
        seen += total;
    }
    if (tid == 0) A.row_count[uh] = make_int2(off[A.B] + A.B, seen);
    if (uh == 0 && tid == 0) *A.ticket = 0u;
}
template <int kThreads>
__device__ __forceinline__ void csr_write_slots(const CsrArgs &A, int uh, const int *off, int *scratch) {
    csr_write_pivots<kThreads>(A, uh, off, 0, A.B);
    csr_write_pieces<kThreads>(A, uh, off, scratch);
}

// n words from global to shared memory, eight per thread on their way together.
template <int kThreads, typename T>
__device__ __forceinline__ void copy_batched(T *dst, const T *src, int n) {
    for (int i = threadIdx.x; i < n; i += 8 * kThreads) {
        T v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = i + e * kThreads < n ? src[i + e * kThreads] : T(0);
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (i + e * kThreads < n) dst[i + e * kThreads] = v[e];
    }
}

// grid = U*Hkv, block = 32 * NW threads (warp w owns a contiguous range of the input).  n_pass passes of kCsrBits bits.
// For heads too large for build_csr_count_kernel below: keys are gathered by position and positions scattered through
// global memory, which an SM takes at about one access per clock.
template <int NW>
__global__ void __launch_bounds__(32 * NW) build_csr_kernel(const CsrArgs A) {
    constexpr int kThreads = 32 * NW;
    constexpr int kBatch = 8;                       // steps of 32 positions whose loads are in flight together
    __shared__ int counters[NW][kCsrBins + 1];      // [warp][digit], padded
    __shared__ int scratch[33];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int uh = blockIdx.x;
    predecessor_done();
    const int *match = A.match + (int64_t)uh * A.E;
    int *bufs[2] = {A.sort_a + (int64_t)uh * A.E, A.sort_b + (int64_t)uh * A.E};
    auto key_of = [&](int j) -> int { return csr_key(match[j], A.B); };
    const int per_warp = ((A.E + NW - 1) / NW + 31) / 32 * 32;     // multiple of 32
    const int lo = warp * per_warp, hi = min(A.E, lo + per_warp);
    const int end = min(lo + per_warp, ((hi + 31) / 32) * 32);

    for (int pass = 0; pass < A.n_pass; ++pass) {
        const int shift = kCsrBits * pass;
        const int *src = pass == 0 ? nullptr : bufs[(pass - 1) & 1];
        int *dst = bufs[pass & 1];
        // The positions and their keys are fetched kBatch steps at a time (the loads of a step depend on each other,
        // those of different steps do not); a step past the warp's range has no valid lane and changes nothing.
        auto fetch = [&](int t0, int (&jv)[kBatch], int (&dg)[kBatch]) {
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int idx = t0 + 32 * b + lane;
                jv[b] = idx < hi ? (src ? (int)src[idx] : idx) : -1;
            }
#pragma unroll
            for (int b = 0; b < kBatch; ++b) dg[b] = jv[b] >= 0 ? (key_of(jv[b]) >> shift) & (kCsrBins - 1) : 0;
        };
        // count the warp's positions by digit (order does not matter here: shared-memory atomics on the warp's own counters)
        for (int d = lane; d < kCsrBins; d += 32) counters[warp][d] = 0;
        __syncwarp();
        for (int t0 = lo; t0 < end; t0 += 32 * kBatch) {
            int jv[kBatch], dg[kBatch];
            fetch(t0, jv, dg);
#pragma unroll
            for (int b = 0; b < kBatch; ++b)
                if (jv[b] >= 0) atomicAdd(&counters[warp][dg[b]], 1);
        }
        __syncthreads();
        // exclusive scan in (digit, warp) order: thread t holds the kPerThread consecutive entries from kPerThread t on,
        // entry e being digit = e / NW, warp = e % NW
        {
            constexpr int kPerThread = kCsrBins / 32;
            int vals[kPerThread], sum = 0;
#pragma unroll
            for (int e = 0; e < kPerThread; ++e) {
                const int idx = tid * kPerThread + e;
                vals[e] = counters[idx % NW][idx / NW];
                sum += vals[e];
            }
            int total;
            int run = block_exclusive_scan(sum, scratch, total);
            __syncthreads();
#pragma unroll
            for (int e = 0; e < kPerThread; ++e) {
                const int idx = tid * kPerThread + e;
                counters[idx % NW][idx / NW] = run;
                run += vals[e];
            }
        }
        __syncthreads();
        // scatter, in order inside each warp's range: the warp's counters now hold the next free place of each digit
        for (int t0 = lo; t0 < end; t0 += 32 * kBatch) {
            int jv[kBatch], dg[kBatch];
            fetch(t0, jv, dg);
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const bool valid = jv[b] >= 0;
                const uint32_t mine = digit_peers(dg[b], valid);
                if (valid) dst[counters[warp][dg[b]] + __popc(mine & lanemask_lt())] = jv[b];
                __syncwarp();
                if (valid && lane == __ffs(mine) - 1) counters[warp][dg[b]] += __popc(mine);
                __syncwarp();
            }
        }
        __syncthreads();
        __threadfence_block();
    }
    const int *sorted = bufs[(A.n_pass - 1) & 1];
    int *off = A.off + (int64_t)uh * (A.B + 1);
    // token position and weight of every member, in slot order
    {
        const int *evi = A.evicted + (int64_t)uh * A.E;
        const float *sim = A.match_sim + (int64_t)uh * A.E;
        int2 *rows = A.rows + (int64_t)uh * (A.B + A.E);
        // ... and off[s] = number of sorted entries with key < s: entry i starts every slot above its predecessor's
        // key up to its own, the last entry also ends the slots above its key (E > 0: the kernel is not launched otherwise)
        for (int i = tid; i < A.E; i += kThreads) {
            const int j = sorted[i];
            const int key = key_of(j);
            const int prev = i > 0 ? key_of(sorted[i - 1]) : -1;
            if (key < A.B) rows[i + key + 1] = make_int2(evi[j], __float_as_int(A.merge_mode == 1 ? 1.f : __expf(sim[j] - 1.f)));
            for (int s2 = prev + 1; s2 <= key; ++s2) off[s2] = i;
            if (i == A.E - 1)
                for (int s2 = key + 1; s2 <= A.B; ++s2) off[s2] = A.E;
        }
    }
    __syncthreads();
    csr_write_slots<kThreads>(A, uh, off, scratch);
}

// The same lists for heads whose sort fits in shared memory: one counting pass over the whole slot number instead of a
// digit at a time.  Every warp owns a contiguous range of positions and 16-bit counters for all B + 1 slots.
//   1. warps count their ranges;  2. a thread per pair of slots turns the counts into every warp's start inside the slot,
//   one prefix sum over the slots gives the slots' starts;  3. warps walk their ranges again, in order, and place the
//   positions (lanes of the same slot rank themselves by votes);  4. token positions and similarities are staged in the
//   counters' place and written out in slot order;  5. what csr_write_slots adds.
// Bound by issue slots and shared-memory latency of one CTA per head (two walks of E positions, 11 votes per step at
// B = 1690): 8 heads of 32 102 positions 77 us with two 6-bit digits in shared memory, 58 us so; 112 heads of 6 758 32 and
// 25 us.  Dynamic shared memory: csr_count_smem().
__host__ __device__ constexpr size_t csr_count_smem(int E, int B, int n_warps) {
    const size_t Ep = ((size_t)E + 7) & ~(size_t)7, Lp = ((size_t)E + B + 7) & ~(size_t)7, cnt = (size_t)n_warps * (((size_t)B + 2) & ~(size_t)1) * 2;
    return 2 * Lp + 4 * (((size_t)B + 4) & ~(size_t)3) + (4 * Ep > cnt ? 4 * Ep : cnt) + 16;
}
// (Two blocks of 32 warps to an SM, of 32 registers: 284 heads of 9000 tokens with 37 registers 104.9 us for the step, so 97.0.  Blocks of 8 warps
// are left to the compiler's 48 registers: with 80 registers 576 heads of 4300 117.5 us instead of 107.7; held to 48, it spills.)
template <int NW>
__global__ void __launch_bounds__(32 * NW, NW == 32 ? 2 : 0) build_csr_count_kernel(const CsrArgs A, int n_bits) {
    constexpr int kThreads = 32 * NW, kBatch = 8;
    extern __shared__ __align__(16) uint8_t csr_raw[];
    __shared__ int scratch[33];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, uh = blockIdx.x, E = A.E, B = A.B;
    const size_t Lp = ((size_t)E + B + 7) & ~(size_t)7;
    uint16_t *sorted = reinterpret_cast<uint16_t *>(csr_raw);                        // [Lp] positions in slot order, a place before each slot's for its pivot
    int *off = reinterpret_cast<int *>(csr_raw + 2 * Lp);                            // [B + 1] first member of every slot
    uint8_t *region = csr_raw + 2 * Lp + 4 * (((size_t)B + 4) & ~(size_t)3);
    const int pitch = (B + 2) & ~1;                                                  // counters of a warp, an even number
    uint16_t *cnt = reinterpret_cast<uint16_t *>(region) + warp * pitch;
    for (int i = tid; i < NW * pitch / 2; i += kThreads) reinterpret_cast<uint32_t *>(region)[i] = 0u;
    __syncthreads();
    predecessor_done();
    const int *match = A.match + (int64_t)uh * E;
    const int per_warp = ((E + NW - 1) / NW + 31) / 32 * 32, lo = min(E, warp * per_warp), hi = min(E, lo + per_warp);
    auto fetch = [&](int t0, int (&key)[kBatch]) {                                   // -1: no such position
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int j = t0 + 32 * b + lane;
            key[b] = j < hi ? csr_key(match[j], B) : -1;
        }
    };
    auto count = [&](const int (&key)[kBatch]) {
#pragma unroll
        for (int b = 0; b < kBatch; ++b)
            if (key[b] >= 0) atomicAdd(reinterpret_cast<uint32_t *>(cnt) + (key[b] >> 1), (key[b] & 1) ? 0x10000u : 1u);
    };
    const int *evi = A.evicted + (int64_t)uh * E;
    const float *sim = A.match_sim + (int64_t)uh * E;
    int2 *rows = A.rows + (int64_t)uh * (B + E);
    // A warp's positions are one batch (up to 2048 for the head): it keeps them with their tokens and weights from the first walk and
    // writes the rows straight to their places, without the staging's four rounds through memory.  The call, us, staged and so: 112
    // caches of 640 rows with 423 slots 81.2, 79.6; 112 of 1900 with 1000 152.5, 148.1; 112 heads of 2400 with 480 150.9, 144.5.  (For 32
    // warps, up to 8192 positions: 112 heads of 6758 the same, 160 of 6400 911, 963: the registers leave one block to an SM.)
    const bool one = NW == 8 && E <= 32 * kBatch * NW;
    int key1[kBatch], tok1[kBatch];
    float w1[kBatch];
    if (one) {
        fetch(lo, key1);
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            tok1[b] = key1[b] >= 0 ? evi[lo + 32 * b + lane] : 0;
            w1[b] = key1[b] >= 0 ? sim[lo + 32 * b + lane] : 0.f;
        }
        count(key1);
    } else
        for (int t0 = lo; t0 < hi; t0 += 32 * kBatch) {
            int key[kBatch];
            fetch(t0, key);
            count(key);
        }
    __syncthreads();
    for (int i0 = 0, seen = 0; i0 < pitch / 2; i0 += kThreads) {                     // (one round up to 2 kThreads slots)
        const int i = i0 + tid;
        uint32_t run = 0;
        if (i < pitch / 2) {
            uint32_t *col = reinterpret_cast<uint32_t *>(region) + i;
#pragma unroll 8
            for (int w = 0; w < NW; ++w) {                                           // two slots at a time, no carry between them: E < 65536
                const uint32_t x = col[w * (pitch / 2)];
                col[w * (pitch / 2)] = run;
                run += x;
            }
        }
        int total;
        const int first = seen + block_exclusive_scan((int)(run & 0xFFFFu) + (int)(run >> 16), scratch, total);
        if (2 * i <= B) off[2 * i] = first;
        if (2 * i + 1 <= B) off[2 * i + 1] = first + (int)(run & 0xFFFFu);
        seen += total;
    }
    __syncthreads();
    auto place = [&](const int (&key)[kBatch], auto &&put) {                         // put(batch entry, the member's row in slot order)
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const bool valid = key[b] >= 0;
            uint32_t mine = __ballot_sync(0xFFFFFFFFu, valid);                       // lanes of the same slot
            if (mine == 0u) break;
            for (int q = 0; q < n_bits; ++q) {
                const uint32_t vote = __ballot_sync(0xFFFFFFFFu, (key[b] >> q) & 1);
                mine &= ((key[b] >> q) & 1) ? vote : ~vote;
            }
            if (valid && key[b] < B) put(b, off[key[b]] + key[b] + 1 + cnt[key[b]] + __popc(mine & lanemask_lt()));
            __syncwarp();
            if (valid && lane == __ffs(mine) - 1) cnt[key[b]] += (uint16_t)__popc(mine);
            __syncwarp();
        }
    };
    if (one) {
        place(key1, [&](int b, int row) { rows[row] = make_int2(tok1[b], __float_as_int(A.merge_mode == 1 ? 1.f : __expf(w1[b] - 1.f))); });
    } else {
        for (int t0 = lo; t0 < hi; t0 += 32 * kBatch) {
            int key[kBatch];
            fetch(t0, key);
            place(key, [&](int b, int row) { sorted[row] = (uint16_t)(t0 + 32 * b + lane); });
        }
        for (int s = tid; s < B; s += kThreads) sorted[off[s] + s] = 0xFFFF;         // the pivots' places (E < 65536: no position is that)
        __syncthreads();
        const int n_rows = off[B] + B;
        int *stage = reinterpret_cast<int *>(region);
        copy_batched<kThreads>(stage, evi, E);
        __syncthreads();
        for (int i = tid; i < n_rows; i += kThreads) {
            const int j = sorted[i];
            if (j != 0xFFFF) rows[i].x = stage[j];
        }
        float *stage_f = reinterpret_cast<float *>(region);
        if (A.merge_mode != 1) {
            __syncthreads();
            copy_batched<kThreads>(stage_f, sim, E);
            __syncthreads();
        }
        for (int i = tid; i < n_rows; i += kThreads) {
            const int j = sorted[i];
            if (j != 0xFFFF) rows[i].y = __float_as_int(A.merge_mode == 1 ? 1.f : __expf(stage_f[j] - 1.f));
        }
    }
    csr_write_slots<kThreads>(A, uh, off, scratch);
}

// The counting sort with a head's positions shared among the CTAs of a cluster, for calls whose heads do not fill the GPU.
// As above, but every CTA counts its part of the positions, reads the other CTAs' totals per slot out of their shared
// memory, and writes its members' token positions and weights straight to their places (8 heads of 32 102 positions:
// 59 -> 22 us).  Bound by its chain of loads: where a warp's positions are one batch, all that is needed of them is fetched at the
// start, the other CTAs' totals are read together, and every CTA writes its share of the slots (the whole call: 8 heads of 33 792 tokens
// 231 -> 227 us, of 12 000 102.3 -> 101.1, 4 of 10 800 with 2160 pivots 88.6 -> 85.6).
// grid = (U*Hkv * ctas), cluster = ctas along x.  Dynamic shared memory: csr_cluster_smem().
constexpr int kCsrClusterWarps = 16, kMaxCsrCtas = 8;
__host__ __device__ constexpr size_t csr_cluster_smem(int B) {
    const size_t pitch = ((size_t)B + 2) & ~(size_t)1;
    return kCsrClusterWarps * pitch * 2 + pitch * 2 + 2 * pitch * 4 + 16;
}
__global__ void __launch_bounds__(32 * kCsrClusterWarps) build_csr_cluster_kernel(const CsrArgs A, int n_bits, int ctas) {
    constexpr int NW = kCsrClusterWarps, kThreads = 32 * NW, kBatch = 8;
    extern __shared__ __align__(16) uint8_t csr_raw[];
    __shared__ int scratch[33];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, E = A.E, B = A.B;
    const int uh = blockIdx.x / ctas, rank = blockIdx.x % ctas;
    const int pitch = (B + 2) & ~1;                                                  // counters of a warp, an even number
    uint32_t *words = reinterpret_cast<uint32_t *>(csr_raw);                         // [NW][pitch / 2] pairs of 16-bit counters
    uint32_t *totals = words + NW * pitch / 2;                                       // [pitch / 2] this CTA's counts
    int *off = reinterpret_cast<int *>(totals + pitch / 2);                          // [B + 1] first member of every slot
    int *base = off + pitch;                                                         // ... of this CTA's part of it
    uint16_t *cnt = reinterpret_cast<uint16_t *>(csr_raw) + warp * pitch;
    for (int i = tid; i < NW * pitch / 2; i += kThreads) words[i] = 0u;
    __syncthreads();
    predecessor_done();
    const int *match = A.match + (int64_t)uh * E, *evi = A.evicted + (int64_t)uh * E;
    const float *sim = A.match_sim + (int64_t)uh * E;
    const int per_warp = ((E + ctas * NW - 1) / (ctas * NW) + 31) / 32 * 32;
    const int lo = min(E, (rank * NW + warp) * per_warp), hi = min(E, lo + per_warp);
    // a batch of the warp's positions (key -1: no such position); what its rows need comes along
    auto fetch = [&](int t0, int (&key)[kBatch], int (&tok)[kBatch], float (&w)[kBatch], bool rows_too) {
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int j = t0 + 32 * b + lane;
            key[b] = j < hi ? csr_key(match[j], B) : -1;
            tok[b] = rows_too && j < hi ? evi[j] : 0;
            w[b] = rows_too && j < hi ? sim[j] : 0.f;
        }
    };
    const bool one = per_warp <= 32 * kBatch;                                        // the first batch is the only one, and stays in registers
    int key[kBatch], tok[kBatch];
    float w[kBatch];
    for (int t0 = lo; t0 < hi || t0 == lo; t0 += 32 * kBatch) {
        fetch(t0, key, tok, w, one);
#pragma unroll
        for (int b = 0; b < kBatch; ++b)
            if (key[b] >= 0) atomicAdd(reinterpret_cast<uint32_t *>(cnt) + (key[b] >> 1), (key[b] & 1) ? 0x10000u : 1u);
    }
    __syncthreads();
    for (int i = tid; i < pitch / 2; i += kThreads) {                                // two slots at a time, no carry between them: E < 65536
        uint32_t run = 0;
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            const uint32_t x = words[q * (pitch / 2) + i];
            words[q * (pitch / 2) + i] = run;
            run += x;
        }
        totals[i] = run;
    }
    cluster_sync();
    const uint32_t totals_at = (uint32_t)__cvta_generic_to_shared(totals);
    for (int i0 = 0, seen = 0; i0 < pitch / 2; i0 += kThreads) {
        const int i = i0 + tid;
        uint32_t part[kMaxCsrCtas], all = 0, before = 0;
#pragma unroll
        for (int r = 0; r < kMaxCsrCtas; ++r) part[r] = r < ctas && i < pitch / 2 ? ld_cluster_u32(totals_at + 4 * i, r) : 0u;   // (on their way together)
#pragma unroll
        for (int r = 0; r < kMaxCsrCtas; ++r) {
            before = r == rank ? all : before;
            all += part[r];
        }
        int total;
        const int first = seen + block_exclusive_scan((int)(all & 0xFFFFu) + (int)(all >> 16), scratch, total);
        const int second = first + (int)(all & 0xFFFFu);
        if (2 * i <= B) { off[2 * i] = first; base[2 * i] = first + (int)(before & 0xFFFFu); }
        if (2 * i + 1 <= B) { off[2 * i + 1] = second; base[2 * i + 1] = second + (int)(before >> 16); }
        seen += total;
    }
    __syncthreads();
    cluster_arrive();                                                                // the other CTAs' totals have been read
    int2 *rows = A.rows + (int64_t)uh * (B + E);
    for (int t0 = lo; t0 < hi; t0 += 32 * kBatch) {
        if (!one) fetch(t0, key, tok, w, true);
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const bool valid = key[b] >= 0;
            uint32_t mine = __ballot_sync(0xFFFFFFFFu, valid);                       // lanes of the same slot
            if (mine == 0u) break;
            for (int q = 0; q < n_bits; ++q) {
                const uint32_t vote = __ballot_sync(0xFFFFFFFFu, (key[b] >> q) & 1);
                mine &= ((key[b] >> q) & 1) ? vote : ~vote;
            }
            if (valid && key[b] < B) {                                               // (dropped tokens have no place)
                const int at = base[key[b]] + cnt[key[b]] + __popc(mine & lanemask_lt());
                rows[at + key[b] + 1] = make_int2(tok[b], __float_as_int(A.merge_mode == 1 ? 1.f : __expf(w[b] - 1.f)));
            }
            __syncwarp();
            if (valid && lane == __ffs(mine) - 1) cnt[key[b]] += (uint16_t)__popc(mine);
            __syncwarp();
        }
    }
    // the slots in even shares, the pieces by the last CTA, which has the fewest positions
    csr_write_pivots<kThreads>(A, uh, off, B * rank / ctas, B * (rank + 1) / ctas);
    if (rank == ctas - 1) csr_write_pieces<kThreads>(A, uh, off, scratch);
    __syncwarp();
    cluster_wait();                                                                  // nobody's totals go away while they are read
}

struct MergeArgs {
    const void *k, *v;
    void *k_out, *v_out;
    const int *retained;              // [UH, B]
    const int2 *rows;                 // [UH, L] as in CsrArgs; nullptr when E == 0: the pivots alone
    const int2 *row_count;            // [UH]
    const int *first_slot;            // [UH, n_win]
    const int4 *pieces;               // [UH, max_parts]
    const int *part_off;              // [UH, B+1]
    float *partial;                   // [UH, max_parts, 2*D + 4] fp32 partial sums
    unsigned *ticket;                 // shared work counter; nullptr: windows are taken with a stride
    int *slot_done;                   // [UH, B] arrival counters of long slots
    int Hkv, D, L, B, E, max_parts, win, n_win;
    int64_t ks[3], vs[3], kos[3], vos[3];
};

// A slot whose members were cut into several pieces: add the pieces' partial sums in piece order,
// then the pivot row, normalise and store.  Run by the warp whose piece was the last to arrive;
// the partial records come from other SMs, so they are read past L1.
template <typename T>
__device__ __forceinline__ void merge_finish_slot(const MergeArgs &A, int uh, int slot, int lane) {
    constexpr int V = Elem<T>::kVec;
    const int u = uh / A.Hkv, h = uh % A.Hkv;
    const int *poff = A.part_off + (int64_t)uh * (A.B + 1);
    const int part_base = poff[slot], n_pieces = poff[slot + 1] - part_base;
    const float *rec0 = A.partial + ((int64_t)uh * A.max_parts + part_base) * (2 * A.D + 4);
    const int rv = A.D / V;
    const int r = A.retained[(int64_t)uh * A.B + slot];
    float wsum = 0.f;
    for (int p = 0; p < n_pieces; ++p) wsum += __ldcg(rec0 + (int64_t)p * (2 * A.D + 4) + 2 * A.D);
    const float inv = 1.f / (1.f + wsum);
    for (int vec = lane; vec < 2 * rv; vec += 32) {
        const bool is_v = vec >= rv;
        const int c0 = (is_v ? vec - rv : vec) * V;
        float acc[V];
#pragma unroll
        for (int e = 0; e < V; ++e) acc[e] = 0.f;
        for (int p = 0; p < n_pieces; ++p) {
            const float *rec = rec0 + (int64_t)p * (2 * A.D + 4) + (is_v ? A.D : 0) + c0;
#pragma unroll
            for (int e = 0; e < V; ++e) acc[e] += __ldcg(rec + e);
        }
        const T *src = is_v ? static_cast<const T *>(A.v) + u * A.vs[0] + h * A.vs[1] + (int64_t)r * A.vs[2]
                            : static_cast<const T *>(A.k) + u * A.ks[0] + h * A.ks[1] + (int64_t)r * A.ks[2];
        T *dst = is_v ? static_cast<T *>(A.v_out) + u * A.vos[0] + h * A.vos[1] + (int64_t)slot * A.vos[2]
                      : static_cast<T *>(A.k_out) + u * A.kos[0] + h * A.kos[1] + (int64_t)slot * A.kos[2];
        float x[V], o[V];
        Elem<T>::load16(src + c0, x);
#pragma unroll
        for (int e = 0; e < V; ++e) o[e] = (x[e] + acc[e]) * inv;
        Elem<T>::store16(dst + c0, o);
    }
}

constexpr int kMergeBatch = 8;        // member rows a warp keeps in flight

// Short lists (up to kShortList non-pivots per head): no member lists.  A block holds the head's matches,
// tokens and weights in shared memory, a warp finds the members of its slot by ballots over them, in ascending order, and
// sums their rows, 8 on their way at a time.  A slot of more than kSoloMembers is shared
// by the block's warps, each with an eighth of the members; the parts are added in order.
// Bound by latency: a chain of three loads, where the sort of the lists and the tables around it took a launch of its own.  The
// call of 4 heads of 192 tokens (fp32) 40.6 -> 31.4 us, 8 of 950 62 -> 50, 112 of 640 with 423 slots (bf16) 110 -> 102.
constexpr int kShortList = 1024, kSoloMembers = 64;

// grid = (UH, slots / (8 * kPer)), 256 threads; a warp takes kPer consecutive slots and finds the members of all of them in one
// walk over the list (a walk per slot took 69.6 us for a call of 8 heads with 1000 entries and 1500 slots, this 61.9).  The slots'
// counts wait in shared memory, and bf16 takes the slots one after the other: in registers and unrolled, 64 registers a thread did not
// hold them (112 heads of 217 entries and 423 slots 23.3 -> 21.8 us, 448 of 217 and 300 87 -> 79; three blocks per SM with 75
// registers 24.8 and 99).  fp32, two vectors per lane and row, gains from overlapping the slots (43.6 us, one after the other 47.8).
template <typename T, int kPer>
__global__ void __launch_bounds__(256, 4) merge_short_kernel(const MergeArgs A, const int *match, const int *evicted, const float *match_sim,
                                                             int merge_mode) {
    constexpr int V = Elem<T>::kVec, kWarps = 8;
    __shared__ int e_slot[kShortList], e_tok[kShortList];
    __shared__ float e_w[kShortList];
    __shared__ uint16_t members[kWarps][kPer][kSoloMembers], counts[kWarps][kPer];
    __shared__ float part[kWarps][32][V + 1];
    __shared__ int popular;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int uh = blockIdx.x, u = uh / A.Hkv, h = uh % A.Hkv, s0 = blockIdx.y * kWarps * kPer, s1 = min(A.B, s0 + kWarps * kPer);
    const int rv = A.D / V, n_vec = 2 * rv;                              // 16-byte vectors of a row, of a K row and its V row
    const T *kb = static_cast<const T *>(A.k) + u * A.ks[0] + h * A.ks[1], *vb = static_cast<const T *>(A.v) + u * A.vs[0] + h * A.vs[1];
    const int *ret = A.retained + (int64_t)uh * A.B;
    if (tid == 0) popular = 0;
    predecessor_done();
    for (int j = tid; j < A.E; j += 256) {
        const int64_t i = (int64_t)uh * A.E + j;
        const float sim = merge_mode == 1 ? 1.f : match_sim[i];
        e_slot[j] = match[i];
        e_tok[j] = evicted[i];
        e_w[j] = merge_mode == 1 ? 1.f : __expf(sim - 1.f);
    }
    __syncthreads();
    auto finish = [&](int slot, bool is_v, int c0, const uint4 &pivot, const float (&acc)[V], float wsum, int count) {
        T *dst = (is_v ? static_cast<T *>(A.v_out) + u * A.vos[0] + h * A.vos[1] + (int64_t)slot * A.vos[2]
                       : static_cast<T *>(A.k_out) + u * A.kos[0] + h * A.kos[1] + (int64_t)slot * A.kos[2]) + c0;
        if (count == 0) { *reinterpret_cast<uint4 *>(dst) = pivot; return; }   // nothing merged in: the pivot row, bit for bit
        const float inv = 1.f / (1.f + wsum);
        float xf[V], o[V];
        Elem<T>::unpack(pivot, xf);
#pragma unroll
        for (int e = 0; e < V; ++e) o[e] = (xf[e] + acc[e]) * inv;
        Elem<T>::store16(dst, o);
    };
    const int mine = s0 + warp * kPer;                                   // this warp's first slot
    int n_members[kPer];
#pragma unroll
    for (int p = 0; p < kPer; ++p) n_members[p] = 0;
#pragma unroll 4
    for (int b = 0; b < A.E; b += 32) {
        const int which = b + lane < A.E ? e_slot[b + lane] - mine : -1;
        if (kPer > 1 && __ballot_sync(0xFFFFFFFFu, which >= 0 && which < kPer) == 0u) continue;
#pragma unroll
        for (int p = 0; p < kPer; ++p) {
            const uint32_t hits = __ballot_sync(0xFFFFFFFFu, which == p);
            const int at = n_members[p] + __popc(hits & lanemask_lt());
            if (which == p && at < kSoloMembers) members[warp][p][at] = (uint16_t)(b + lane);
            n_members[p] += __popc(hits);
        }
    }
    if constexpr (kPer > 1) {
#pragma unroll
        for (int p = 0; p < kPer; ++p)
            if (lane == p) counts[warp][p] = (uint16_t)n_members[p];
    }
    __syncwarp();
#pragma unroll (sizeof(T) == 4 ? kPer : 1)
    for (int p = 0; p < kPer; ++p) {
        const int slot = mine + p, count = kPer > 1 ? counts[warp][p] : n_members[0];
        if (slot >= s1) break;
        const int r = ret[slot];
        if (count > kSoloMembers) {
            if (lane == 0) popular = 1;
        } else {
            for (int vec = lane; vec < n_vec; vec += 32) {
                const bool is_v = vec >= rv;
                const int c0 = (is_v ? vec - rv : vec) * V;
                const T *src = (is_v ? vb : kb) + c0;
                const int64_t stride = is_v ? A.vs[2] : A.ks[2];
                const uint4 pivot = load_raw16(src + (int64_t)r * stride);
                float acc[V], wsum = 0.f;
#pragma unroll
                for (int e = 0; e < V; ++e) acc[e] = 0.f;
                for (int t0 = 0; t0 < count; t0 += kMergeBatch) {
                    uint4 x[kMergeBatch];
#pragma unroll
                    for (int q = 0; q < kMergeBatch; ++q)                // the batch's row loads, back to back
                        x[q] = t0 + q < count ? load_raw16(src + (int64_t)e_tok[members[warp][p][t0 + q]] * stride) : make_uint4(0, 0, 0, 0);
#pragma unroll
                    for (int q = 0; q < kMergeBatch; ++q)                // fixed order: ascending member index
                        if (t0 + q < count) {
                            const float w = e_w[members[warp][p][t0 + q]];
                            float xf[V];
                            Elem<T>::unpack(x[q], xf);
                            wsum += w;
#pragma unroll
                            for (int e = 0; e < V; ++e) acc[e] = fmaf(w, xf[e], acc[e]);
                        }
                }
                finish(slot, is_v, c0, pivot, acc, wsum, count);
            }
        }
    }
    __syncthreads();
    if (!popular) return;
    for (int slot = s0; slot < s1; ++slot) {                             // the popular slots, by all warps
        int count = 0;
        for (int b = 0; b < A.E; b += 32) count += __popc(__ballot_sync(0xFFFFFFFFu, b + lane < A.E && e_slot[b + lane] == slot));
        if (count <= kSoloMembers) continue;                             // (the same for the whole block)
        const int first = count * warp / kWarps, last = count * (warp + 1) / kWarps;
        for (int vec0 = 0; vec0 < n_vec; vec0 += 32) {
            const int vec = vec0 + lane;
            const bool on = vec < n_vec, is_v = vec >= rv;
            const int c0 = on ? (is_v ? vec - rv : vec) * V : 0;
            const T *src = (is_v ? vb : kb) + c0;
            const int64_t stride = is_v ? A.vs[2] : A.ks[2];
            float acc[V], wsum = 0.f;
#pragma unroll
            for (int e = 0; e < V; ++e) acc[e] = 0.f;
            int seen = 0;
            for (int b = 0; b < A.E && seen < last; b += 32) {
                uint32_t hits = __ballot_sync(0xFFFFFFFFu, b + lane < A.E && e_slot[b + lane] == slot);
                for (; hits != 0u && seen < last; hits &= hits - 1, ++seen) {
                    if (seen < first) continue;
                    const int i = b + __ffs(hits) - 1;
                    const float w = e_w[i];
                    float xf[V];
                    Elem<T>::unpack(load_raw16(src + (int64_t)e_tok[i] * stride), xf);
                    wsum += w;
#pragma unroll
                    for (int e = 0; e < V; ++e) acc[e] = fmaf(w, xf[e], acc[e]);
                }
            }
#pragma unroll
            for (int e = 0; e < V; ++e) part[warp][lane][e] = acc[e];
            part[warp][lane][V] = wsum;
            __syncthreads();
            if (warp == 0) {
                for (int w = 1; w < kWarps; ++w) {
#pragma unroll
                    for (int e = 0; e < V; ++e) acc[e] += part[w][lane][e];
                    wsum += part[w][lane][V];
                }
                if (on) finish(slot, is_v, c0, load_raw16(src + (int64_t)ret[slot] * stride), acc, wsum, count);
            }
            __syncthreads();
        }
    }
}

}  // namespace flowmm
