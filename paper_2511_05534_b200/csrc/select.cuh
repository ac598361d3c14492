// Pivot selection (top-B per KV head, Section 3.3.1) with what rides along with it: the layer flow of Eq. 6, the theta
// rule, and the candidate layout of the tensor-core matching step.
#pragma once
#include "common.cuh"
#include "match_tc.cuh"

#include <type_traits>

namespace flowmm {

// Order-preserving integer key of an importance (a non-negative float); window tokens forced
// into the pivot set get the largest key.  31 bits: bit 31 of a staged word holds the token's modality.
constexpr uint32_t kKeyMask = 0x7FFFFFFFu;
__device__ __forceinline__ uint32_t select_key(float v, bool forced) {
    if (forced) return kKeyMask;
    const uint32_t b = __float_as_uint(v);
    return (b & 0x80000000u) ? 0u : b;        // -0 and (never expected) negatives sort lowest
}

// Eq. 6 and the theta rule riding along with the selection: one extra block per unit, behind those of the heads.
struct SelectFlow {
    const float *cross_part;     // nullptr, or [n_units * Hq, n_parts] partial masses that are first added up into cross_mass
    int n_parts;
    float *cross_mass;           // [n_units, Hq] per-head masses (read; written first when cross_part is given)
    float *rho;                  // [n_units] or nullptr
    int *strategy;               // [n_units]
    int *strategy_h;             // nullptr, or [n_units, n_rep]: the unit's strategy once more for each of its KV heads
    int n_units, Hq, n_rep;
    float theta;
    int flow_mode;
};

struct SelectArgs {
    const float *importance;     // [n_heads, L]
    int *retained, *evicted;     // [n_heads, B], [n_heads, L - B]
    uint8_t *row_mod_out;        // nullptr, or [n_heads, B]: the pivots' modalities (one modality map per head: P.Hkv == 1)
    int n_heads, L, B, W, keep_window;
    int lets_in;                 // the successor may be set up beside this kernel
    int chunk;                   // positions handled at a time, a multiple of 32: the whole context if it fits in shared memory, or a CTA's part of it
};

// The extra block of unit u.  Sums as in cross_mass_reduce and layer_flow_kernel, term for term.
__device__ __forceinline__ void select_flow_block(const SelectFlow &F, int u, int W, float *masses) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    if (F.cross_part) {
        for (int g = warp; g < F.Hq; g += nwarps) {
            const int64_t i = (int64_t)u * F.Hq + g;
            const float s = head_mass(F.cross_part + i * F.n_parts, F.n_parts);
            if (lane == 0) F.cross_mass[i] = s;
        }
        __syncthreads();
    }
    float s = 0.f;
    for (int g0 = 0; g0 < F.Hq; g0 += blockDim.x) {              // (one round unless a unit has more heads than threads)
        const int g = g0 + threadIdx.x;
        if (g < F.Hq) masses[threadIdx.x] = F.cross_mass[(int64_t)u * F.Hq + g] / (float)W;   // a head's total mass is W
        __syncthreads();
        if (threadIdx.x == 0)
            for (int j = 0; j < min((int)blockDim.x, F.Hq - g0); ++j) s += masses[j];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const float r = s / (float)F.Hq;
        const int st = F.flow_mode == 1 ? 0 : F.flow_mode == 2 ? 1 : ((r > F.theta) != (F.flow_mode == 3) ? 1 : 0);
        if (F.rho) F.rho[u] = r;
        F.strategy[u] = st;
        if (F.strategy_h)
            for (int h = 0; h < F.n_rep; ++h) F.strategy_h[(int64_t)u * F.n_rep + h] = st;
    }
}

constexpr int kSelBits = 11, kSelBins = 1 << kSelBits;           // digit width of the radix select
// dynamic shared memory: two sets of counters; the chunk's words; six values per 32 positions
__host__ __device__ constexpr size_t select_smem(int chunk) { return 4 * (2 * (size_t)kSelBins + chunk + 6 * (size_t)(chunk / 32)); }
constexpr int kSelMaxChunk = 45248;
static_assert(select_smem(kSelMaxChunk) <= 232448 - 1024, "shared memory budget");


// The block of one head (blocks below n_heads).
//   1. The importances are staged in shared memory as 31-bit keys with the token's modality in the top bit, and counted
//      by their 11 highest key bits on the way.
//   2. The digit that holds the B-th largest key is found from the counts; the next 11 (then 9) bits are only counted
//      among the keys that share it.  Two digits decide nearly always: as soon as all keys of the last digit belong to
//      the B, its lower bits do not matter.
//   3. Warps mark the pivots (and, of those, the matching candidates by modality) of 32 positions at a time, one prefix
//      sum over the words of marks numbers them, warps write the lists, all ascending.  Ties at the threshold go to the
//      lower positions.
// Bound by latency: one block per head, a few dependent rounds over shared memory.  The marks and
// one prefix sum replace block-wide scans per 1024 to 4096 positions, four counting passes over global memory and a separate
// preparation pass over the lists: 128 heads of 33 792 tokens 118 -> 42 us, 32 heads of 640 tokens 20 -> 10 us.
// kCtas > 1: the CTAs of a cluster share a head, A.chunk positions each (a multiple of 256).  The counts of all of them are
// added up through distributed shared memory in every pass, their totals before the lists are written.  For calls of few
// heads, whose blocks would leave most SMs idle: 8 heads of 33 792 tokens 31 -> 18 us, 4 heads of 8448 14 -> 12.
template <int kThreads, bool kOneChunk, int kCtas, bool kFew>
__global__ void __launch_bounds__(kThreads, kThreads <= 256 ? 1024 / kThreads : kThreads == 512 && kCtas == 1 ? 2 : 1)
select_topb_kernel(const SelectArgs A, const SelectFlow F, const MatchPrepArgs P, int with_prepare) {
    static_assert(kCtas == 1 || (kOneChunk && kThreads == 512), "a CTA's part is one chunk; four counters per thread");
    constexpr int kWarps = kThreads / 32, kPer = kSelBins / kThreads;
    static_assert(!kFew || (kOneChunk && kCtas == 1), "a warp's words in registers");   // (kFew: launched for up to 1024 or 4096 positions)
    extern __shared__ __align__(16) int sel_smem[];
    __shared__ int wtot[kWarps], res[3];
    __shared__ unsigned long long wsum[kWarps];
    __shared__ uint32_t xtot[3];                                     // a CTA's totals, for the others of the cluster
    int *hist = sel_smem;
    uint32_t *words = reinterpret_cast<uint32_t *>(sel_smem + 2 * kSelBins);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int head = blockIdx.x / kCtas, rank_c = kCtas > 1 ? (int)(blockIdx.x % kCtas) : 0;
    const int i0 = rank_c * A.chunk;                                 // first position of this CTA's part (kCtas == 1: 0)
    const int L = kCtas > 1 ? max(0, min(A.chunk, A.L - i0)) : A.L;  // positions this CTA looks at; counted from i0 below
    for (int i = tid; i < 2 * kSelBins / 4; i += kThreads) reinterpret_cast<int4 *>(hist)[i] = make_int4(0, 0, 0, 0);
    __syncthreads();
    predecessor_done();
    if (A.lets_in) successor_may_start();
    if (head >= A.n_heads) {
        if (rank_c == 0) select_flow_block(F, head - A.n_heads, A.W, reinterpret_cast<float *>(hist));
        return;
    }
    const float *imp = A.importance + (int64_t)head * A.L + i0;
    const uint8_t *mod = P.modality + (int64_t)(head / P.Hkv) * A.L + i0;   // (not read unless with_prepare or row_mod_out)
    const int first_forced = (A.keep_window ? A.L - A.W : A.L) - i0;
    auto word = [&](int i) -> uint32_t {
        if (kOneChunk) return words[i];
        return select_key(imp[i], i >= first_forced) | (with_prepare && mod[i] ? 0x80000000u : 0u);
    };

    // keys that agree with `prefix` in the bits of `mask`, counted by the `width` bits at `shift`
    uint32_t prefix = 0, mask = 0;
    auto count = [&](uint32_t key, int *h, int shift, int width) {
        if ((key & mask) == prefix) atomicAdd(h + ((int)(key >> shift) & ((1 << width) - 1)), 1);
    };
    for (int base = 0; base < L; base += 8 * kThreads) {
        float v[8];
        uint8_t m[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int i = base + e * kThreads + tid;
            v[e] = i < L ? imp[i] : 0.f;
            m[e] = with_prepare && i < L ? mod[i] : 0;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            if (base + e * kThreads >= L) break;                     // (the same for the whole block)
            const int i = base + e * kThreads + tid;
            if (i < L) {
                const uint32_t key = select_key(v[e], i >= first_forced);
                if (kOneChunk) words[i] = key | (m[e] ? 0x80000000u : 0u);
                count(key, hist, 20, 11);
            }
        }
    }
    int need = A.B, n_eq = 0;                                        // keys still to take among those that match the prefix; their number
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
        const int shift = pass == 0 ? 20 : pass == 1 ? 9 : 0, width = pass == 2 ? 9 : 11;
        int *h = hist + (pass & 1) * kSelBins;
        if (pass > 0) {
            for (int i = tid; i < L; i += kThreads) count(word(i) & kKeyMask, h, shift, width);
        }
        if (kCtas > 1) cluster_sync(); else __syncthreads();
        // counters from the largest digit down, kPer per thread; thread t holds digits hi - kPer + 1 .. hi
        const int hi = kSelBins - 1 - tid * kPer;
        int c[kPer], sum = 0;
        if constexpr (kCtas > 1) {
            const uint32_t at = (uint32_t)__cvta_generic_to_shared(h + hi - (kPer - 1));
            uint4 part[kCtas];
#pragma unroll
            for (int q = 0; q < kCtas; ++q) part[q] = ld_cluster_u128(at, q);   // (scalar reads took four times as long)
            c[0] = c[1] = c[2] = c[3] = 0;
#pragma unroll
            for (int q = 0; q < kCtas; ++q) { c[0] += (int)part[q].w; c[1] += (int)part[q].z; c[2] += (int)part[q].y; c[3] += (int)part[q].x; }
            sum = (c[0] + c[1]) + (c[2] + c[3]);
        } else {
            // (16 bytes at a time: word by word, lanes kPer words apart are kPer deep in a bank)
            constexpr int kVec = kPer < 4 ? kPer : 4;
            using Vec = std::conditional_t<kVec == 4, int4, int2>;
#pragma unroll
            for (int e = 0; e < kPer; e += kVec) {
                const Vec v = *reinterpret_cast<const Vec *>(h + hi - e - (kVec - 1));
                c[e + kVec - 1] = v.x; c[e + kVec - 2] = v.y;
                if constexpr (kVec == 4) { c[e + 1] = v.z; c[e] = v.w; }
            }
#pragma unroll
            for (int e = 0; e < kPer; ++e) sum += c[e];
        }
        int incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wtot[warp] = incl;
        __syncthreads();
        int w = lane < kWarps && lane < warp ? wtot[lane] : 0;       // totals of the warps before this one
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xFFFFFFFFu, w, o);
        int acc = w + incl - sum;                                    // keys with a larger digit than this thread's first
        if (acc < need && need <= acc + sum) {
            int e = 0;
#pragma unroll
            for (int q = 0; q < kPer - 1; ++q)
                if (e == q && acc + c[q] < need) { acc += c[q]; ++e; }
            int ce = c[0];
#pragma unroll
            for (int q = 1; q < kPer; ++q) ce = e == q ? c[q] : ce;
            res[0] = hi - e; res[1] = need - acc; res[2] = ce;
        }
        __syncthreads();
        prefix |= (uint32_t)res[0] << shift;
        need = res[1];
        n_eq = res[2];
        mask |= ((1u << width) - 1u) << shift;
        if (need == n_eq) break;                                     // all of them are kept: lower bits do not matter
        if (pass == 1)                                               // the third digit takes the first one's counters, which every CTA has read
            for (int i = tid; i < kSelBins; i += kThreads) hist[i] = 0;
        __syncthreads();
    }
    const bool all_eq = need == n_eq;

    // 3. the positions of a chunk in ascending order, 32 to a word
    const int chunk_w = A.chunk >> 5;
    uint32_t *keep_w = words + A.chunk;                              // which of a word's 32 positions are pivots,
    uint32_t *text_w = keep_w + chunk_w, *vis_w = text_w + chunk_w;  // which of those are candidates, by modality,
    int *pos_w = reinterpret_cast<int *>(vis_w + chunk_w);           // how many pivots come before the word,
    int *pt_w = pos_w + chunk_w, *pv_w = pt_w + chunk_w;             // and how many candidates
    const uint32_t lt = lanemask_lt();
    int *ret = A.retained + (int64_t)head * A.B;
    int *evi = A.evicted + (int64_t)head * (A.L - A.B) + i0;
    int *rank = P.rank + (int64_t)head * A.L + i0;
    uint8_t *evi_mod = P.evi_mod + (int64_t)head * (A.L - A.B) + i0;
    int *cand_tok = hist;                                            // token of every candidate column (copy_here: up to 256)
    int *slot_out = P.cand_slot + (int64_t)head * P.Ctot;
    float *scale_out = P.cand_scale + (int64_t)head * P.Ctot;
    const bool copy_here = with_prepare && P.copy_here, by_list = with_prepare && !P.copy_here;
    // modalities in every tile of 256 non-pivots (by_list; the counters' place, as far as it goes)
    uint32_t *tiles = reinterpret_cast<uint32_t *>(hist);
    const bool tiles_here = by_list && P.n_rt <= 2 * kSelBins;
    if (kCtas == 1 && tiles_here)
        for (int t = tid; t < P.n_rt; t += kThreads) tiles[t] = 0;
    // Up to 4096 positions: a warp's words, one run of them, stay in registers, and what comes before them is added up over the warps'
    // totals behind one barrier; the candidates' key rows are fetched while the lists are written.  (With marks in shared memory and
    // a prefix sum over all words, which every warp took for itself, the block of 1471 positions spent 1900 clocks on the marks, 2800 on
    // the sum, 2400 on the lists and 3600 on the rows, of 15 600.  The whole call, us: 4 heads of 192 positions 22.3 -> 21.3, 32 of 640
    // 26.4 -> 25.7, 8 of 1471 36.0 -> 35.0, 112 of 2176 112.7 -> 111.0, 1024 of 640 156.3 -> 153.4.)  Four blocks of 256 threads to an
    // SM: with five or six a thread has too few registers for four rows, with more rows too many.
    if constexpr (kFew) {
        constexpr int kE = kThreads == 256 || kThreads == 1024 ? 4 : 8;   // words of a warp: 1024 positions by up to 256 threads, else 4096
        const int n_w = (L + 31) >> 5, per = (n_w + kWarps - 1) / kWarps, w0 = warp * per;
        uint32_t wd[kE], keep[kE], text[kE], vis[kE];
#pragma unroll
        for (int e = 0; e < kE; ++e) {
            const int i = 32 * (w0 + e) + lane;
            wd[e] = e < per && i < L ? words[i] : 0u;
        }
        int ties = 0;                                                // equal keys before this warp's: the lower positions are taken
        if (!all_eq) {
            int n = 0;
#pragma unroll
            for (int e = 0; e < kE; ++e)
                if (e < per) n += __popc(__ballot_sync(0xFFFFFFFFu, 32 * (w0 + e) + lane < L && (wd[e] & kKeyMask) == prefix));
            if (lane == 0) wtot[warp] = n;
            __syncthreads();
            ties = (int)__reduce_add_sync(0xFFFFFFFFu, lane < warp ? (unsigned)wtot[lane] : 0u);
        }
        uint32_t n_keep_text = 0, n_vis = 0;                         // pivots, and admissible text ones from bit 16 on; admissible visual ones
#pragma unroll
        for (int e = 0; e < kE; ++e) {
            keep[e] = text[e] = vis[e] = 0;
            if (e >= per) continue;
            const int i = 32 * (w0 + e) + lane;
            const uint32_t mk = wd[e] & kKeyMask & mask;
            bool take = i < L && mk >= prefix;
            if (!all_eq) {
                const bool eq = i < L && mk == prefix;
                const uint32_t m = __ballot_sync(0xFFFFFFFFu, eq);
                if (eq) take = ties + __popc(m & lt) < need;
                ties += __popc(m);
            }
            keep[e] = __ballot_sync(0xFFFFFFFFu, take);
            n_keep_text += __popc(keep[e]);
            if (with_prepare) {                                      // Eq. 10: pivots above tau are kept out of merging
                const bool adm = take && (i < first_forced ? __uint_as_float(wd[e] & kKeyMask) : imp[i]) <= P.tau_eff;
                const uint32_t cand = __ballot_sync(0xFFFFFFFFu, adm), seen_vis = __ballot_sync(0xFFFFFFFFu, wd[e] >> 31);
                text[e] = cand & ~seen_vis; vis[e] = cand & seen_vis;
                n_keep_text += __popc(text[e]) << 16;
                n_vis += __popc(vis[e]);
            }
        }
        if (lane == 0) wsum[warp] = n_keep_text | (unsigned long long)n_vis << 32;
        __syncthreads();
        const unsigned long long mine = lane < kWarps ? wsum[lane] : 0ull;
        const uint32_t kt_all = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)mine), v_all = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)(mine >> 32));
        const uint32_t kt = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? (uint32_t)mine : 0u);
        const int n_text = (int)(kt_all >> 16), n_vis_all = (int)v_all, t0 = (n_text + 31) & ~31;   // text group first, visual group from the next multiple of 32
        int s = (int)(kt & 0xFFFF), pt = (int)(kt >> 16), pv = t0 + (int)__reduce_add_sync(0xFFFFFFFFu, lane < warp ? (uint32_t)(mine >> 32) : 0u);
        if (with_prepare) {                                          // the candidates, and the columns without one
            int s1 = s;
#pragma unroll
            for (int e = 0; e < kE; ++e) {
                const uint32_t bit = 1u << lane;
                const int c = text[e] & bit ? pt + __popc(text[e] & lt) : vis[e] & bit ? pv + __popc(vis[e] & lt) : -1;
                if (c >= 0 && index_ok(c, P.Ctot, P.status)) {
                    slot_out[c] = s1 + __popc(keep[e] & lt);
                    if (copy_here) cand_tok[c] = 32 * (w0 + e) + lane;
                }
                s1 += __popc(keep[e]); pt += __popc(text[e]); pv += __popc(vis[e]);
            }
            for (int c = n_text + tid; c < P.Ctot; c += kThreads)
                if (c < t0 || c >= t0 + n_vis_all) {
                    slot_out[c] = -1;
                    scale_out[c] = __int_as_float(0x7FC00000);       // NaN: no candidate here
                    if (copy_here) cand_tok[c] = -1;
                }
            if (tid == 0) { P.cand_count[2 * head] = n_text; P.cand_count[2 * head + 1] = n_vis_all; }
        }
        if (copy_here) __syncthreads();                              // every candidate's token is in place
        constexpr int kRows = 4;                          // candidates' rows per thread on their way together
        MatchGather<kRows> gather(P, head, tid, kThreads);
        int p0 = tid >> 4;
        if (copy_here) gather.start(cand_tok, p0, P.Ctot);
#pragma unroll
        for (int e = 0; e < kE; ++e) {
            if (e >= per) break;
            const int i = 32 * (w0 + e) + lane, sl = s + __popc(keep[e] & lt);
            const bool out = i < L && !((keep[e] >> lane) & 1u), seen = by_list && i < L && words[i] >> 31;
            if (out) {
                evi[i - sl] = i;
                if (copy_here) rank[i] = i - sl;
                else if (by_list) evi_mod[i - sl] = seen;
            } else if (i < L) {
                ret[sl] = i;
                if (A.row_mod_out) A.row_mod_out[(int64_t)head * A.B + sl] = mod[i];
                if (copy_here) rank[i] = -(sl + 2);
            }
            if (by_list) {
                // A word's non-pivots are neighbours in the list, of one tile or of two (a word of both modalities at a tile's
                // edge may claim both for each: such a tile is then visited as a mixed one, with the same result).
                const uint32_t o = __ballot_sync(0xFFFFFFFFu, out), m = __ballot_sync(0xFFFFFFFFu, seen);
                const int first = 32 * (w0 + e) - s;
                if (lane == 0 && o) {
                    const uint32_t what = (o & ~m ? 1u : 0u) | (o & m ? 2u : 0u);
                    atomicOr(&tiles[first / kMtItemRows], what);
                    if (first % kMtItemRows + __popc(o) > kMtItemRows) atomicOr(&tiles[first / kMtItemRows + 1], what);
                }
            }
            s += __popc(keep[e]);
        }
        if (copy_here) {
            gather.finish(p0, P.Ctot);
            for (p0 += kRows * gather.stride; p0 < P.Ctot; p0 += kRows * gather.stride) {   // (uniform trip count within a warp)
                gather.start(cand_tok, p0, P.Ctot);
                gather.finish(p0, P.Ctot);
            }
        } else if (by_list) {
            __syncthreads();
            for (int t = tid; t < P.n_rt; t += kThreads) P.tile_mod[(int64_t)head * P.n_rt + t] = (uint8_t)tiles[t];
        }
        return;
    }
    auto block_sum = [&](unsigned long long v, unsigned long long &total) -> unsigned long long {   // exclusive prefix sum
        unsigned long long incl_v = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long t = __shfl_up_sync(0xFFFFFFFFu, incl_v, o);
            if (lane >= o) incl_v += t;
        }
        __syncthreads();                                             // the totals of the call before have been read
        if (lane == 31) wsum[warp] = incl_v;
        __syncthreads();
        const unsigned long long mine = lane < kWarps ? wsum[lane] : 0ull;
        unsigned long long b = lane < warp ? mine : 0ull, all = mine;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            b += __shfl_xor_sync(0xFFFFFFFFu, b, o);
            all += __shfl_xor_sync(0xFFFFFFFFu, all, o);
        }
        total = all;
        return b + incl_v - v;
    };
    // the same across the cluster: what the CTAs before this one hold, and all of them together
    auto cluster_sum = [&](unsigned long long v, unsigned long long &total) -> unsigned long long {
        if (tid == 0) { xtot[0] = (uint32_t)v; xtot[1] = (uint32_t)(v >> 32); }
        cluster_sync();
        const uint32_t at = (uint32_t)__cvta_generic_to_shared(xtot);
        unsigned long long b = 0, all = 0;
#pragma unroll
        for (int q = 0; q < kCtas; ++q) {
            const unsigned long long x = (unsigned long long)ld_cluster_u32(at, q) | (unsigned long long)ld_cluster_u32(at + 4, q) << 32;
            if (q < rank_c) b += x;
            all += x;
        }
        total = all;
        return b;
    };
    int t0 = 0;                                                      // first column of the visual candidates
    // (a context longer than a chunk is walked once more beforehand, for the number of its text candidates)
    for (int walk = kOneChunk || !with_prepare ? 1 : 0; walk < 2; ++walk) {
        int seen = 0, seen_t = 0, seen_v = 0, seen_eq = 0;           // before the chunk (kCtas > 1: in the CTAs before this one)
        for (int c0 = 0; c0 < L || (kCtas > 1 && c0 == 0); c0 += A.chunk) {   // (a CTA without positions takes part all the same)
            const int n_w = (min(A.chunk, L - c0) + 31) >> 5, per = (n_w + kThreads - 1) / kThreads;
            if (!all_eq) {                                           // ties at the threshold go to the lower positions:
                for (int w = warp; w < n_w; w += kWarps) {           // mark the equal keys, then number them
                    const int i = c0 + 32 * w + lane;
                    const uint32_t eq = __ballot_sync(0xFFFFFFFFu, i < L && (word(i) & kKeyMask) == prefix);
                    if (lane == 0) text_w[w] = eq;
                }
                __syncthreads();
                const int w_lo = min(n_w, tid * per), w_hi = min(n_w, w_lo + per);   // words whose counts this thread adds up
                unsigned long long n_mine = 0, tot;
                for (int w = w_lo; w < w_hi; ++w) n_mine += __popc(text_w[w]);
                int r = (int)block_sum(n_mine, tot);
                if (kCtas > 1) {
                    if (tid == 0) xtot[2] = (uint32_t)tot;
                    cluster_sync();
                    const uint32_t at = (uint32_t)__cvta_generic_to_shared(xtot + 2);
                    for (int q = 0; q < rank_c; ++q) seen_eq += (int)ld_cluster_u32(at, q);
                }
                r += seen_eq;
                for (int w = w_lo; w < w_hi; ++w) { pos_w[w] = r; r += __popc(text_w[w]); }
                seen_eq += (int)tot;
                __syncthreads();
            }
#pragma unroll 4
            for (int w = warp; w < n_w; w += kWarps) {               // marks, a word per warp and step
                const int i = c0 + 32 * w + lane;
                const uint32_t wd = i < L ? word(i) : 0u, mk = wd & kKeyMask & mask;
                bool take = i < L && mk >= prefix;
                if (!all_eq && take && mk == prefix) take = pos_w[w] + __popc(text_w[w] & lt) < need;
                const uint32_t keep = __ballot_sync(0xFFFFFFFFu, take);
                uint32_t text = 0, vis = 0;
                if (with_prepare) {                                  // Eq. 10: pivots above tau are kept out of merging
                    const bool adm = take && (i < first_forced ? __uint_as_float(wd & kKeyMask) : imp[i]) <= P.tau_eff;
                    const uint32_t cand = __ballot_sync(0xFFFFFFFFu, adm), seen_vis = __ballot_sync(0xFFFFFFFFu, wd >> 31);
                    text = cand & ~seen_vis; vis = cand & seen_vis;
                }
                __syncwarp();
                if (lane == 0) { keep_w[w] = keep; text_w[w] = text; vis_w[w] = vis; }
            }
            __syncthreads();
            // Pivots (24 bits), admissible text pivots (20) and admissible visual ones (20) before each word: one prefix sum
            // for all three.
            auto counts = [&](int w) -> unsigned long long {
                return (unsigned long long)__popc(keep_w[w]) | (unsigned long long)__popc(text_w[w]) << 24 | (unsigned long long)__popc(vis_w[w]) << 44;
            };
            const int w_lo = min(n_w, tid * per), w_hi = min(n_w, w_lo + per);
            unsigned long long mine = 0, all;
            for (int w = w_lo; w < w_hi; ++w) mine += counts(w);
            const unsigned long long before = block_sum(mine, all);
            if (kCtas > 1) {                                         // (from here on `all` is the head's)
                const unsigned long long ahead = cluster_sum(all, all);
                seen = (int)(ahead & 0xFFFFFF); seen_t = (int)(ahead >> 24) & 0xFFFFF; seen_v = (int)(ahead >> 44);
                if (!with_prepare) cluster_arrive();                 // the other CTAs' totals have been read
                if (tiles_here) {                                    // (every CTA of the cluster has read the counters)
                    for (int t = tid; t < P.n_rt; t += kThreads) tiles[t] = 0;
                    __syncthreads();
                }
            }
            const int n_text = (int)(all >> 24) & 0xFFFFF, n_vis = (int)(all >> 44);
            if (kOneChunk) t0 = (n_text + 31) & ~31;                 // text group first, visual group from the next multiple of 32
            if (walk == 1) {
                int s = seen + (int)(before & 0xFFFFFF), pt = seen_t + ((int)(before >> 24) & 0xFFFFF), pv = t0 + seen_v + (int)(before >> 44);
                for (int w = w_lo; w < w_hi; ++w) {
                    pos_w[w] = s; pt_w[w] = pt; pv_w[w] = pv;
                    const unsigned long long c = counts(w);
                    s += (int)(c & 0xFFFFFF); pt += (int)(c >> 24) & 0xFFFFF; pv += (int)(c >> 44);
                }
                __syncthreads();
                // The lists, a word per warp and step: coalesced.  A selection alone has a loop of its own: the other's stores to shared
                // memory keep its steps apart.
                if (!with_prepare) {
#pragma unroll 4
                    for (int w = warp; w < n_w; w += kWarps) {
                        const uint32_t keep = keep_w[w];
                        const int i = c0 + 32 * w + lane, sl = pos_w[w] + __popc(keep & lt);
                        if (i >= L) continue;
                        if (!((keep >> lane) & 1u)) { evi[i - sl] = i0 + i; continue; }
                        ret[sl] = i0 + i;
                        if (A.row_mod_out) A.row_mod_out[(int64_t)head * A.B + sl] = mod[i];
                    }
                } else
#pragma unroll 4
                for (int w = warp; w < n_w; w += kWarps) {
                    const uint32_t keep = keep_w[w];
                    const int i = c0 + 32 * w + lane, sl = pos_w[w] + __popc(keep & lt);
                    bool is_vis = false;
                    if (by_list) {
                        is_vis = i < L && word(i) >> 31;
                        const uint32_t m = __ballot_sync(0xFFFFFFFFu, is_vis);
                        if (lane == 0) words[32 * w] = m;                // (nobody reads these keys any more)
                    }
                    if (i >= L) continue;
                    if (!((keep >> lane) & 1u)) {
                        evi[i - sl] = i0 + i;
                        if (copy_here) rank[i] = i0 + i - sl;
                        if (by_list) evi_mod[i - sl] = is_vis;
                        continue;
                    }
                    ret[sl] = i0 + i;
                    if (A.row_mod_out) A.row_mod_out[(int64_t)head * A.B + sl] = mod[i];
                    if (copy_here) rank[i] = -(sl + 2);
                    const uint32_t text = text_w[w], vis = vis_w[w];
                    const int c = ((text >> lane) & 1u) ? pt_w[w] + __popc(text & lt) : ((vis >> lane) & 1u) ? pv_w[w] + __popc(vis & lt) : -1;
                    if (c >= 0 && index_ok(c, P.Ctot, P.status)) {
                        slot_out[c] = sl;
                        if (copy_here) {
                            if (kCtas > 1) {
                                const uint32_t at = (uint32_t)__cvta_generic_to_shared(cand_tok + c);
#pragma unroll
                                for (int q = 0; q < kCtas; ++q) st_cluster_u32(at, q, (uint32_t)(i0 + i));
                            } else cand_tok[c] = i;
                        }
                    }
                }
                if (tiles_here) {
                    // A word's non-pivots are neighbours in the list, of one tile or of two (a word of both modalities at a tile's
                    // edge may claim both for each: such a tile is then visited as a mixed one, with the same result).
                    __syncthreads();
                    for (int w = tid; w < n_w; w += kThreads) {
                        const int left = L - c0 - 32 * w;
                        const uint32_t out = ~keep_w[w] & (left < 32 ? (1u << left) - 1u : 0xFFFFFFFFu), m = words[32 * w];
                        if (out == 0u) continue;
                        const uint32_t what = (out & ~m ? 1u : 0u) | (out & m ? 2u : 0u);
                        const int e = i0 + c0 + 32 * w - pos_w[w];
                        atomicOr(&tiles[e / kMtItemRows], what);
                        if (e % kMtItemRows + __popc(out) > kMtItemRows) atomicOr(&tiles[e / kMtItemRows + 1], what);
                    }
                }
                if (!kOneChunk) __syncthreads();                     // (the next chunk's words go into the same place)
            }
            if (kCtas > 1) { seen_t = n_text; seen_v = n_vis; }
            else { seen += (int)(all & 0xFFFFFF); seen_t += n_text; seen_v += n_vis; }
        }
        if (walk == 0) t0 = (seen_t + 31) & ~31;
        else if (with_prepare) {
            // columns without a candidate: between the groups and behind them
            for (int c = seen_t + tid; c < P.Ctot; c += kThreads)
                if (c < t0 || c >= t0 + seen_v) {
                    if (rank_c == 0) {
                        slot_out[c] = -1;
                        scale_out[c] = __int_as_float(0x7FC00000);   // NaN: no candidate here
                    }
                    if (copy_here) cand_tok[c] = -1;
                }
            if (tid == 0 && rank_c == 0) { P.cand_count[2 * head] = seen_t; P.cand_count[2 * head + 1] = seen_v; }
        }
    }
    if (by_list) {
        if (kCtas > 1) cluster_sync(); else __syncthreads();         // every CTA's tiles are marked
        if (rank_c == 0)
            for (int t = tid; t < P.n_rt; t += kThreads) {
                uint32_t m = tiles_here ? tiles[t] : 3u;
                if (kCtas > 1 && tiles_here) {
                    const uint32_t at = (uint32_t)__cvta_generic_to_shared(tiles + t);
#pragma unroll
                    for (int q = 1; q < kCtas; ++q) m |= ld_cluster_u32(at, q);
                }
                P.tile_mod[(int64_t)head * P.n_rt + t] = (uint8_t)m;
            }
    }
    if (copy_here) {
        if (kCtas > 1) cluster_sync(); else __syncthreads();         // every candidate's token is in place, in every CTA
        const int lo = P.Ctot / 32 * rank_c / kCtas * 32, hi = P.Ctot / 32 * (rank_c + 1) / kCtas * 32;
        match_gather_rows<8>(P, head, cand_tok, lo, hi, tid, kThreads);
    } else if (kCtas > 1) {                                          // nobody's totals and tiles go away while they are read
        if (with_prepare) cluster_arrive();
        cluster_wait();
    }
}

}  // namespace flowmm
