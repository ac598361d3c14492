// SIMT fp32 kernels for the two dense contractions (window scoring and pivot matching).
// They serve fp32 inputs and head_dim 64, and any shape the tensor-core kernels do not take.
// Products of the inputs are accumulated in fp32; for bf16 inputs every product is exact.
#pragma once
#include "common.cuh"

namespace flowmm {

constexpr int kTile = 64;       // rows and columns of a CTA tile
constexpr int kDChunk = 32;     // head_dim slice held in shared memory
constexpr int kPitch = 68;      // row pitch of a slice (floats): 16-byte aligned, breaks bank strides
constexpr int kSimtThreads = 256;

struct SimtTiles {
    float a[kDChunk][kPitch];
    float b[kDChunk][kPitch];
    float norm_a[kTile], norm_b[kTile];      // kNorms: reciprocal norms of the tile's rows (0 for a zero row)
};

// acc[i][j] = sum_d A[ty*kR+i][d] * B[tx*4+j][d] for a tile of 16 kR x 64, kR = 4 or 1; rowA(r) / rowB(r) give the
// address of tile row r (nullptr: a row of zeros).  All 256 threads of the CTA take part.
// Small calls wait for their loads more than they compute: a slice of the head dimension is fetched while the one before it
// is multiplied, and with kNorms the threads that bring the rows in take their norms on the way (left in sm.norm_a / norm_b
// at the function's end, behind a barrier).
template <typename T, bool kNorms = false, int kR, typename FA, typename FB>
__device__ __forceinline__ void simt_tile_dot(SimtTiles &sm, int D, FA rowA, FB rowB, float (&acc)[kR][4]) {
    static_assert(kR == 4 || kR == 1, "a thread's rows are read 16 bytes at a time, or it has one");
    constexpr int V = Elem<T>::kVec;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
#pragma unroll
    for (int i = 0; i < kR; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    const int lr = tid >> 2, ld = (tid & 3) * V;       // this thread loads 8 elements of row lr, 16 bytes at a time
    const bool has_a = lr < 16 * kR;
    const T *pa = has_a ? rowA(lr) : nullptr;
    const T *pb = rowB(lr);
    float va[8 / V][V], vb[8 / V][V], na = 0.f, nb = 0.f;
    auto fetch = [&](int d0) {
#pragma unroll
        for (int half = 0; half < 8 / V; ++half) {
#pragma unroll
            for (int e = 0; e < V; ++e) va[half][e] = vb[half][e] = 0.f;
            if (pa) Elem<T>::load16(pa + d0 + ld + half * 4 * V, va[half]);
            if (pb) Elem<T>::load16(pb + d0 + ld + half * 4 * V, vb[half]);
        }
    };
    fetch(0);
    for (int d0 = 0; d0 < D; d0 += kDChunk) {
        __syncthreads();
#pragma unroll
        for (int half = 0; half < 8 / V; ++half) {
#pragma unroll
            for (int e = 0; e < V; ++e) {
                if (has_a) sm.a[ld + half * 4 * V + e][lr] = va[half][e];
                sm.b[ld + half * 4 * V + e][lr] = vb[half][e];
                if (kNorms) {
                    na = fmaf(va[half][e], va[half][e], na);
                    nb = fmaf(vb[half][e], vb[half][e], nb);
                }
            }
        }
        __syncthreads();
        if (d0 + kDChunk < D) fetch(d0 + kDChunk);
#pragma unroll 8
        for (int d = 0; d < kDChunk; ++d) {
            float a[kR];
            if constexpr (kR == 4) {
                const float4 a4 = *reinterpret_cast<const float4 *>(&sm.a[d][ty * 4]);
                a[0] = a4.x; a[1] = a4.y; a[2] = a4.z; a[3] = a4.w;
            } else a[0] = sm.a[d][ty];
            const float4 b4 = *reinterpret_cast<const float4 *>(&sm.b[d][tx * 4]);
            const float b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
            for (int i = 0; i < kR; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
    }
    if (kNorms) {                                      // the four threads of a row sit side by side
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            na += __shfl_xor_sync(0xFFFFFFFFu, na, o);
            nb += __shfl_xor_sync(0xFFFFFFFFu, nb, o);
        }
        if ((tid & 3) == 0) {
            sm.norm_a[lr] = na > 0.f ? rsqrtf(na) : 0.f;
            sm.norm_b[lr] = nb > 0.f ? rsqrtf(nb) : 0.f;
        }
        __syncthreads();
    }
}

struct ScoreArgs {
    const void *q, *k;
    const uint8_t *modality;      // [U, L]
    float *importance;            // [U, Hkv, L]
    float2 *row_part;             // [U*Hq*W, n_chunk1]: (max, sum) of a row over one key chunk, log2 domain
    float *cross_part;            // [U*Hq, n_chunk2]
    int Hq, Hkv, G, D, L, W;
    int n_chunk1, chunk1;         // pass 1: key chunks per row, keys per chunk (multiple of 64)
    int n_chunk2, chunk2;         // pass 2
    float scale_log2;             // softmax scale * log2(e)
    int64_t qs[3], ks[3];
};

// Pass 1 of Eq. 8: per proxy row the running maximum and exp-sum of its causal logits over one
// chunk of keys.  grid = (U*Hkv, row tiles of G*W, n_chunk1).
template <typename T>
__global__ void __launch_bounds__(kSimtThreads) score_stats_simt(const ScoreArgs A) {
    predecessor_done();
    __shared__ SimtTiles sm;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const int uh = blockIdx.x, u = uh / A.Hkv, h = uh % A.Hkv;
    const int GW = A.G * A.W;
    const int row0 = blockIdx.y * kTile;
    const int key_lo = blockIdx.z * A.chunk1, key_hi = min(A.L, key_lo + A.chunk1);
    const T *q = static_cast<const T *>(A.q) + u * A.qs[0];
    const T *k = static_cast<const T *>(A.k) + u * A.ks[0] + h * A.ks[1];

    float m[4], l[4];
    int pa[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        m[i] = kNegBig; l[i] = 0.f;
        const int r = row0 + ty * 4 + i;
        pa[i] = r < GW ? A.L - A.W + (r % A.W) : -1;
    }
    auto rowA = [&](int lr) -> const T * {
        const int r = row0 + lr;
        if (r >= GW) return nullptr;
        return q + (int64_t)(h * A.G + r / A.W) * A.qs[1] + (int64_t)(r % A.W) * A.qs[2];
    };
    for (int kt = key_lo; kt < key_hi; kt += kTile) {
        auto rowB = [&](int lr) -> const T * {
            const int i = kt + lr;
            return i < key_hi ? k + (int64_t)i * A.ks[2] : nullptr;
        };
        float acc[4][4];
        simt_tile_dot<T>(sm, A.D, rowA, rowB, acc);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float s[4], mx = m[i];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int key = kt + tx * 4 + j;
                const bool ok = key < key_hi && key <= pa[i];       // causal inside the window
                s[j] = ok ? acc[i][j] * A.scale_log2 : kNegBig;
                mx = fmaxf(mx, s[j]);
            }
            float add = 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) add += s[j] > 0.5f * kNegBig ? exp2f(s[j] - mx) : 0.f;
            l[i] = l[i] * exp2f(m[i] - mx) + add;
            m[i] = mx;
        }
    }
    // the 16 threads that share a row sit in one half-warp
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            const float mo = __shfl_xor_sync(0xFFFFFFFFu, m[i], o);
            const float lo = __shfl_xor_sync(0xFFFFFFFFu, l[i], o);
            const float mx = fmaxf(m[i], mo);
            l[i] = l[i] * exp2f(m[i] - mx) + lo * exp2f(mo - mx);
            m[i] = mx;
        }
        const int r = row0 + ty * 4 + i;
        if (tx == 0 && r < GW)
            A.row_part[((int64_t)uh * GW + r) * A.n_chunk1 + blockIdx.z] = make_float2(m[i], l[i]);
    }
}

// Pass 2 of Eq. 8 and the modality split of Eq. 7: logits are recomputed, normalised with the
// row statistics of pass 1, summed down the columns into the importance, and summed per head
// over the keys of the other modality.  grid = (U*Hkv, n_chunk2); dynamic shared memory:
// 3*G*W floats.
template <typename T>
__global__ void __launch_bounds__(kSimtThreads) score_colsum_simt(const ScoreArgs A) {
    predecessor_done();
    __shared__ SimtTiles sm;
    __shared__ float colpart[16][kTile];
    extern __shared__ float dyn[];
    const int GW = A.G * A.W;
    float *row_max = dyn, *row_inv = dyn + GW, *row_cross = dyn + 2 * GW;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const int uh = blockIdx.x, u = uh / A.Hkv, h = uh % A.Hkv;
    const int key_lo = blockIdx.y * A.chunk2, key_hi = min(A.L, key_lo + A.chunk2);
    const T *q = static_cast<const T *>(A.q) + u * A.qs[0];
    const T *k = static_cast<const T *>(A.k) + u * A.ks[0] + h * A.ks[1];
    const uint8_t *mod = A.modality + (int64_t)u * A.L;

    for (int r = tid; r < GW; r += kSimtThreads) {      // combine the chunk statistics of pass 1
        const float2 *part = A.row_part + ((int64_t)uh * GW + r) * A.n_chunk1;
        float mx = kNegBig;
        for (int c = 0; c < A.n_chunk1; ++c) mx = fmaxf(mx, part[c].x);
        float z = 0.f;
        for (int c = 0; c < A.n_chunk1; ++c) z += part[c].y * exp2f(part[c].x - mx);
        row_max[r] = mx;
        row_inv[r] = 1.f / z;
        row_cross[r] = 0.f;
    }
    __syncthreads();

    for (int kt = key_lo; kt < key_hi; kt += kTile) {
        auto rowB = [&](int lr) -> const T * {
            const int i = kt + lr;
            return i < key_hi ? k + (int64_t)i * A.ks[2] : nullptr;
        };
        float colacc[4] = {0.f, 0.f, 0.f, 0.f};
        uint8_t mk[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int key = kt + tx * 4 + j;
            mk[j] = key < key_hi ? mod[key] : 0;
        }
        for (int row0 = 0; row0 < GW; row0 += kTile) {
            auto rowA = [&](int lr) -> const T * {
                const int r = row0 + lr;
                if (r >= GW) return nullptr;
                return q + (int64_t)(h * A.G + r / A.W) * A.qs[1] + (int64_t)(r % A.W) * A.qs[2];
            };
            uint8_t mqs[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {                        // (fetched along with the rows)
                const int r = row0 + ty * 4 + i;
                mqs[i] = r < GW ? mod[A.L - A.W + (r % A.W)] : 0;
            }
            float acc[4][4];
            simt_tile_dot<T>(sm, A.D, rowA, rowB, acc);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = row0 + ty * 4 + i;
                float cr = 0.f;
                if (r < GW) {
                    const int pa = A.L - A.W + (r % A.W);
                    const uint8_t mq = mqs[i];
                    const float mx = row_max[r], inv = row_inv[r];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int key = kt + tx * 4 + j;
                        if (key < key_hi && key <= pa) {
                            const float p = exp2f(acc[i][j] * A.scale_log2 - mx) * inv;
                            colacc[j] += p;
                            if (mk[j] != mq) cr += p;
                        }
                    }
                }
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) cr += __shfl_xor_sync(0xFFFFFFFFu, cr, o);
                if (tx == 0 && r < GW) row_cross[r] += cr;      // one owner per row: fixed order
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j) colpart[ty][tx * 4 + j] = colacc[j];
        __syncthreads();
        if (tid < kTile) {
            float s = 0.f;
#pragma unroll
            for (int t = 0; t < 16; ++t) s += colpart[t][tid];
            const int key = kt + tid;
            if (key < key_hi) A.importance[(int64_t)uh * A.L + key] = s / (float)A.G;   // group mean
        }
    }
    __syncthreads();
    for (int g = tid; g < A.G; g += kSimtThreads) {
        float s = 0.f;
        for (int a = 0; a < A.W; ++a) s += row_cross[g * A.W + a];
        A.cross_part[((int64_t)u * A.Hq + h * A.G + g) * A.n_chunk2 + blockIdx.y] = s;
    }
}

// Both passes in one launch for short contexts with one tile of proxy rows (G*W <= 64, at most 16 key tiles): the CTAs of a
// cluster take the key tiles of a head by turns, keep the logits in registers, exchange the row statistics through distributed
// shared memory and go on with the probabilities.  grid = (U*Hkv * ctas), cluster = ctas <= 8, kTiles key tiles per CTA.
// Bound by latency: against two launches that compute the logits twice, 4 heads of 192 tokens 29.8 -> 23.2 us for the call, 8 of
// 950 46.6 -> 43.0.
// With up to 16 proxy rows a thread has one row (kR = 1), as tiles of 64 would be zeros for three quarters: with the same in the matching, 4
// heads of 192 tokens 21.5 -> 17.9 us for the call, of 1000 59.4 -> 56.2.
constexpr int kClusterScoreTiles = 16;
template <typename T, int kTiles, int kR>
__global__ void __launch_bounds__(kSimtThreads) score_cluster_simt(const ScoreArgs A, int ctas) {
    __shared__ SimtTiles sm;
    __shared__ float colpart[16][kTile];
    __shared__ float stat_m[kTile], stat_l[kTile], row_max[kTile], row_inv[kTile], row_cross[kTile];
    predecessor_done();
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const int uh = blockIdx.x / ctas, rank = blockIdx.x % ctas, u = uh / A.Hkv, h = uh % A.Hkv;
    const int GW = A.G * A.W;
    const T *q = static_cast<const T *>(A.q) + u * A.qs[0];
    const T *k = static_cast<const T *>(A.k) + u * A.ks[0] + h * A.ks[1];
    const uint8_t *mod = A.modality + (int64_t)u * A.L;

    float acc[kTiles][kR][4], m[kR], l[kR];
    int pa[kR];
    uint8_t mq[kR], mk[kTiles][4];
#pragma unroll
    for (int i = 0; i < kR; ++i) {
        m[i] = kNegBig; l[i] = 0.f;
        const int r = ty * kR + i;
        pa[i] = r < GW ? A.L - A.W + (r % A.W) : -1;
        mq[i] = r < GW ? mod[pa[i]] : 0;
    }
    auto rowA = [&](int r) -> const T * {
        return r < GW ? q + (int64_t)(h * A.G + r / A.W) * A.qs[1] + (int64_t)(r % A.W) * A.qs[2] : nullptr;
    };
#pragma unroll
    for (int t = 0; t < kTiles; ++t) {
        const int kt = (rank + t * ctas) * kTile;
#pragma unroll
        for (int j = 0; j < 4; ++j) mk[t][j] = kt + tx * 4 + j < A.L ? mod[kt + tx * 4 + j] : 0;
        if (kt >= A.L) break;                                    // (the same for the whole CTA)
        auto rowB = [&](int lr) -> const T * { return kt + lr < A.L ? k + (int64_t)(kt + lr) * A.ks[2] : nullptr; };
        simt_tile_dot<T>(sm, A.D, rowA, rowB, acc[t]);
#pragma unroll
        for (int i = 0; i < kR; ++i) {
            float mx = m[i], add = 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const bool ok = kt + tx * 4 + j <= pa[i];        // causal inside the window
                acc[t][i][j] = ok ? acc[t][i][j] * A.scale_log2 : kNegBig;
                mx = fmaxf(mx, acc[t][i][j]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) add += acc[t][i][j] > 0.5f * kNegBig ? exp2f(acc[t][i][j] - mx) : 0.f;
            l[i] = l[i] * exp2f(m[i] - mx) + add;
            m[i] = mx;
        }
    }
#pragma unroll
    for (int i = 0; i < kR; ++i) {                                // the 16 threads that share a row sit in one half-warp
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            const float mo = __shfl_xor_sync(0xFFFFFFFFu, m[i], o);
            const float lo = __shfl_xor_sync(0xFFFFFFFFu, l[i], o);
            const float mx = fmaxf(m[i], mo);
            l[i] = l[i] * exp2f(m[i] - mx) + lo * exp2f(mo - mx);
            m[i] = mx;
        }
        if (tx == 0) { stat_m[ty * kR + i] = m[i]; stat_l[ty * kR + i] = l[i]; }
    }
    cluster_sync();
    if (tid < GW) {
        const uint32_t at_m = (uint32_t)__cvta_generic_to_shared(stat_m + tid), at_l = (uint32_t)__cvta_generic_to_shared(stat_l + tid);
        float mr[8], lr[8], mx = kNegBig, z = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            mr[c] = c < ctas ? ld_cluster(at_m, c) : kNegBig;
            lr[c] = c < ctas ? ld_cluster(at_l, c) : 0.f;
            mx = fmaxf(mx, mr[c]);
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) z += lr[c] * exp2f(mr[c] - mx);
        row_max[tid] = mx;
        row_inv[tid] = 1.f / z;
    }
    cluster_arrive();                                            // the other CTAs' statistics have been read
    __syncthreads();
    float cross[kR] = {};
#pragma unroll
    for (int t = 0; t < kTiles; ++t) {
        const int kt = (rank + t * ctas) * kTile;
        if (kt >= A.L) break;
        float colacc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < kR; ++i) {
            const int r = ty * kR + i;
            if (r >= GW) break;
            const float mx = row_max[r], inv = row_inv[r];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float p = acc[t][i][j] > 0.5f * kNegBig ? exp2f(acc[t][i][j] - mx) * inv : 0.f;
                colacc[j] += p;
                cross[i] += mk[t][j] != mq[i] ? p : 0.f;
            }
        }
        if (t > 0) __syncthreads();
#pragma unroll
        for (int j = 0; j < 4; ++j) colpart[ty][tx * 4 + j] = colacc[j];
        __syncthreads();
        if (tid < kTile && kt + tid < A.L) {
            float s = 0.f;
#pragma unroll
            for (int y = 0; y < 16; ++y) s += colpart[y][tid];
            A.importance[(int64_t)uh * A.L + kt + tid] = s / (float)A.G;   // group mean
        }
    }
#pragma unroll
    for (int i = 0; i < kR; ++i) {
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) cross[i] += __shfl_xor_sync(0xFFFFFFFFu, cross[i], o);
        if (tx == 0) row_cross[ty * kR + i] = cross[i];
    }
    __syncthreads();
    for (int g = tid; g < A.G; g += kSimtThreads) {
        float s = 0.f;
        for (int a = 0; a < A.W; ++a) s += row_cross[g * A.W + a];
        A.cross_part[((int64_t)u * A.Hq + h * A.G + g) * ctas + rank] = s;
    }
    cluster_wait();                                              // nobody's statistics go away while they are read
}

// cross_mass[u, g] = sum of the per-chunk partial masses; one warp per head.
__global__ void cross_mass_reduce(const float *cross_part, int n_chunk, int n, float *cross_mass) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    predecessor_done();
    if (i >= n) return;
    const float s = head_mass(cross_part + (int64_t)i * n_chunk, n_chunk);
    if (lane_id() == 0) cross_mass[i] = s;
}

// Eq. 6 and the theta rule: one thread per unit.
__global__ void layer_flow_kernel(const float *cross_mass, int U, int Hq, int W, float theta, int flow_mode,
                                  float *rho, int *strategy) {
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    predecessor_done();
    if (u >= U) return;
    float s = 0.f;
    for (int g = 0; g < Hq; ++g) s += cross_mass[(int64_t)u * Hq + g] / (float)W;   // a head's total mass is W
    const float r = s / (float)Hq;
    if (rho) rho[u] = r;
    strategy[u] = flow_mode == 1 ? 0 : flow_mode == 2 ? 1 : ((r > theta) != (flow_mode == 3) ? 1 : 0);
}

// Full-prefill flow: the parts of every head's mass added up (lanes take parts with a stride of 32, then a shuffle tree:
// a fixed order), then Eq. 6 over all L rows and the theta rule.  parts [n_parts][U * Hq]; one block per unit, a warp per head.
__global__ void full_flow_reduce_kernel(const float *parts, int n_parts, int n, int Hq, int L, float theta, int flow_mode,
                                        float *cross_mass, float *rho, int *strategy) {
    predecessor_done();
    const int u = blockIdx.x, lane = lane_id();
    for (int g = threadIdx.x >> 5; g < Hq; g += blockDim.x >> 5) {
        float s = 0.f;
        for (int t = lane; t < n_parts; t += 32) s += parts[(int64_t)t * n + (int64_t)u * Hq + g];
        s = warp_sum(s);
        if (lane == 0) cross_mass[(int64_t)u * Hq + g] = s;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        float s = 0.f;
        for (int g = lane; g < Hq; g += 32) s += cross_mass[(int64_t)u * Hq + g] / (float)L;   // a head's total mass is L
        const float r = warp_sum(s) / (float)Hq;
        if (lane == 0) {
            if (rho) rho[u] = r;
            strategy[u] = flow_mode == 1 ? 0 : flow_mode == 2 ? 1 : ((r > theta) != (flow_mode == 3) ? 1 : 0);
        }
    }
}

struct MatchArgs {
    const void *k;
    const float *importance;      // [U, Hkv, L]
    const uint8_t *modality;      // [U, L]
    const int *retained, *evicted, *strategy;
    int *match;
    float *match_sim;
    int Hkv, D, L, B, E;
    float tau_eff;
    int64_t ks[3];
};

// Eq. 9 and Eq. 10: cosine similarity of 16 kR non-pivots against every pivot, gated argmax per row.
// grid = (U*Hkv, ceil(E / (16 kR))).
template <typename T, int kR>
__global__ void __launch_bounds__(kSimtThreads) match_simt(const MatchArgs A) {
    predecessor_done();
    __shared__ SimtTiles sm;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const int uh = blockIdx.x, u = uh / A.Hkv, h = uh % A.Hkv;
    const T *k = static_cast<const T *>(A.k) + u * A.ks[0] + h * A.ks[1];
    const int *ret = A.retained + (int64_t)uh * A.B;
    const int *evi = A.evicted + (int64_t)uh * A.E;
    const float *imp = A.importance + (int64_t)uh * A.L;
    const uint8_t *mod = A.modality + (int64_t)u * A.L;
    const bool intra = A.strategy[u] == 0;
    const int j0 = blockIdx.y * (16 * kR);

    float best[kR];
    int bests[kR];
    uint8_t me[kR];
#pragma unroll
    for (int i = 0; i < kR; ++i) {
        const int j = j0 + ty * kR + i;
        const int e = j < A.E ? evi[j] : -1;
        me[i] = e >= 0 ? mod[e] : 0;
        best[i] = -INFINITY;
        bests[i] = 0x7FFFFFFF;
    }
    auto rowA = [&](int lr) -> const T * {
        const int j = j0 + lr;
        return j < A.E ? k + (int64_t)evi[j] * A.ks[2] : nullptr;
    };
    for (int s0 = 0; s0 < A.B; s0 += kTile) {
        auto rowB = [&](int lr) -> const T * {
            const int s = s0 + lr;
            return s < A.B ? k + (int64_t)ret[s] * A.ks[2] : nullptr;
        };
        bool adm[4];
        uint8_t mr[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {                        // (fetched along with the rows)
            const int s = s0 + tx * 4 + j, r = s < A.B ? ret[s] : -1;
            adm[j] = r >= 0 && imp[r] <= A.tau_eff;          // a highly sensitive pivot is never a merge target
            mr[j] = r >= 0 ? mod[r] : 0;
        }
        float acc[kR][4];
        simt_tile_dot<T, true>(sm, A.D, rowA, rowB, acc);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int s = s0 + tx * 4 + j;
            if (!adm[j]) continue;
            const float rnr = sm.norm_b[tx * 4 + j];
#pragma unroll
            for (int i = 0; i < kR; ++i) {
                if (intra && mr[j] != me[i]) continue;
                const float uval = acc[i][j] * sm.norm_a[ty * kR + i] * rnr;
                if (uval > best[i] || (uval == best[i] && s < bests[i])) { best[i] = uval; bests[i] = s; }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < kR; ++i) {
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            const float bo = __shfl_xor_sync(0xFFFFFFFFu, best[i], o);
            const int so = __shfl_xor_sync(0xFFFFFFFFu, bests[i], o);
            if (bo > best[i] || (bo == best[i] && so < bests[i])) { best[i] = bo; bests[i] = so; }
        }
        const int j = j0 + ty * kR + i;
        if (tx == 0 && j < A.E) {
            const bool none = bests[i] == 0x7FFFFFFF;
            A.match[(int64_t)uh * A.E + j] = none ? -1 : bests[i];
            A.match_sim[(int64_t)uh * A.E + j] = none ? 0.f : best[i];
        }
    }
}

}  // namespace flowmm
