// C ABI of the FlowMM compression library: validation, workspace layout and kernel launches.
// Declarations and the meaning of every argument are in include/flowmm.h.
#include "flowmm.h"

#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <mutex>

#include "common.cuh"
#include "decode.cuh"
#include "decode_tc.cuh"
#include "flow_tc.cuh"
#include "match_merge_tc.cuh"
#include "match_small_tc.cuh"
#include "merge_rows.cuh"
#include "merge_tc.cuh"
#include "score_cluster_tc.cuh"
#include "score_fused_tc.cuh"
#include "match_tc.cuh"
#include "merge_lists.cuh"
#include "score_tc.cuh"
#include "select.cuh"
#include "simt_kernels.cuh"
#include "tc_host.cuh"

using namespace flowmm;

namespace {

thread_local int32_t g_launches = 0;

// Optional per-kernel timing: one event before the first kernel of an entry point, one after each.
constexpr int kMaxProfiled = 32;
struct Profile {
    bool on = false, have_events = false;
    cudaEvent_t ev[kMaxProfiled + 1];
    const char *name[kMaxProfiled];
    int n = 0;
};
thread_local Profile g_prof;

inline void profile_begin(cudaStream_t st) {
    g_launches = 0;
    g_prof.n = 0;
    if (g_prof.on) cudaEventRecord(g_prof.ev[0], st);
}
inline void profile_mark(const char *name, cudaStream_t st) {
    if (g_prof.on && g_prof.n < kMaxProfiled) {
        g_prof.name[g_prof.n] = name;
        cudaEventRecord(g_prof.ev[++g_prof.n], st);
    }
}

// Launches a kernel as a programmatic dependent of the one before it in the stream: its blocks are set up while that
// kernel drains, and predecessor_done() in the kernel holds them back from the data (common.cuh).  A launch boundary
// costs 2 us less than with a plain launch (13 launches of a re-compression: 163 to 135 us) and the host no more.  An
// error stays in cudaGetLastError() for FLOWMM_LAUNCHED.
template <typename... Params, typename... Args>
void launch_cluster(dim3 cluster, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args &&...args) {
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster.x; attr[1].val.clusterDim.y = cluster.y; attr[1].val.clusterDim.z = cluster.z;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cfg.attrs = attr; cfg.numAttrs = cluster.x * cluster.y * cluster.z > 1 ? 2 : 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}
template <typename... Params, typename... Args>
void launch(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args &&...args) {
    launch_cluster(dim3(1), kernel, grid, block, smem, st, args...);
}

#define FLOWMM_LAUNCHED(name)                                          \
    do {                                                               \
        ++g_launches;                                                  \
        if (cudaGetLastError() != cudaSuccess) return FLOWMM_ERR_CUDA; \
        profile_mark(name, st);                                        \
    } while (0)

#define FLOWMM_TRY(expr)                         \
    do {                                         \
        const flowmm_status _s = (expr);         \
        if (_s != FLOWMM_OK) return _s;          \
    } while (0)

// Lets a kernel have all of a block's shared memory beside `static_bytes` of its own.  The same for every call: function attributes are the
// device's, and a call's own size could be lowered by another thread's between here and the launch.
constexpr int kBlockSmem = 227 * 1024;
template <typename... Params>
bool allow_smem(void (*kernel)(Params...), int static_bytes = 0) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBlockSmem - static_bytes) == cudaSuccess;
}

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// (unit, head) pairs per call: they index grid.x of several launches and 32-bit item counters
// (items = pairs x row tiles), so the bound is generous rather than a grid limit of 65535.
constexpr int64_t kMaxHeadsPerCall = 1 << 22;

// Blocks that the scoring is cut for: one per SM of a B200, and about two of the SIMT kernels.  (By hand: the size of a workspace is
// asked for without a GPU.)
constexpr int kScoreCtas = 148, kSimtCtas = 2 * kScoreCtas;

// Where everything lives inside the caller's workspace.  One layout serves every entry point.
struct Layout {
    size_t status, importance, cross_mass, rho, strategy, retained, evicted, match, match_sim;
    size_t row_part, cross_part, sort_a, sort_b, rows, row_count, off, first_slot, part_off, pieces, partial, ticket, slot_done;
    size_t cand_k, cand_scale, cand_slot, cand_count, rank, evi_mod, tile_mod, row_all;
    size_t tokmap;             // [UH, L] (slot, weight) of every token position, for the tensor-core merge
    size_t merge_status;       // status word the merge kernels report to (the workspace's own, or one of the merge scratch)
    int tc_q_rows, tc_keys2, tc_n_qt, tc_runs, tc_n_part;
    size_t total;
    int n_chunk1, chunk1, n_chunk2, chunk2, max_parts, csr_passes, merge_win, n_win, c_tot, n_rt, n_et;
};

int chunks_for(int L, int other_ctas, int &chunk) {
    // enough CTAs to fill the GPU about twice, at least 64 keys per chunk
    int want = (kSimtCtas + other_ctas - 1) / other_ctas;
    const int max_chunks = (L + kTile - 1) / kTile;
    if (want < 1) want = 1;
    if (want > max_chunks) want = max_chunks;
    chunk = ((L + want - 1) / want + kTile - 1) / kTile * kTile;
    return (L + chunk - 1) / chunk;
}

// Rows of a window of the merge kernel (merge_rows.cuh).  Long windows cost less per row, short ones give every warp one: 1.2 million
// rows at most leave 3552 warps five windows of 64.  34 000 rows by 32 and 16: 77.7 and 76.4 us for the call, 43 000 84.3 and 87.3,
// 270 000 231.5 and 240.6.
// From kManyRows on warps draw their windows from a counter, else windows are taken with a stride.  The merge by windows of 32 with a
// stride, and of 64 from the counter, us: 300 000 rows 44 to 53, 53 to 64; 0.8 million 83, 86; 1.0 million 109 to 123, 113 to 124;
// 1.3 million 154, 156; 1.6 million 165, 164; 2.5 million 257, 248; 4.3 million 422, 392 (fp32 rows of 64 within 1 %, equal from 0.8 million on).
// While every warp has one window at most and warps are left for the pieces of long slots, one per 256 members (members seldom make more; the
// first ones of all heads get them, merge_rows.cuh), the windows are as short as leaves it so, by groups of four rows (other lengths misalign the
// reads of the list: 64 heads of 1688 rows by 31 were 1.3 % slower).  The merge step, us, by windows of 32, so, and with the pieces left out of
// account, head by head behind the windows, so that a warp with a window and a piece set the pace: 32 heads of 2500 with 250 slots, one of
// them long, 19.8, 19.5, 23.1; 16 of 3500 with 350 18.6, 19.0, 22.0; 24 of 4296 with 430 26.6, 21.5, 26.5; 32 of 1500 with 300, 64 of them long,
// 19.5, 18.9, 23.6; none long 12 of 6000 with 1200 19.8, 18.3, 18.3.  Windows shorter than two slots would often be empty: 4 heads of 10 822
// rows with 542 slots by 16 instead of 32 81.8 -> 85.2 for the call.  (Equal numbers of longer windows, 39 rows for 270 000, 232 -> 243.)
constexpr int64_t kManyRows = 1300000;
constexpr int kMinWin = 16, kMergeCtas = 3 * kScoreCtas;
int merge_window(const flowmm_params &p) {
    const int64_t heads = (int64_t)p.n_units * p.n_kv_heads, rows = heads * p.seq_len;
    if (rows >= kManyRows) return mrow::kMaxWin;
    if (rows < 40000) return kMinWin;
    const int parts = (p.seq_len - p.n_keep) / 256;
    int win = kMinWin;
    while (win < 32 && (win * (int64_t)p.n_keep < 2 * (int64_t)p.seq_len || heads * ((p.seq_len + win - 1) / win + parts) > kMergeCtas * mrow::kWarps)) win += 4;
    return win;
}

// The part of the workspace that the merge step uses (rows in slot order, windows, pieces, partial sums).
template <class Take>
void layout_merge(Layout &y, const flowmm_params &p, Take take) {
    const size_t UH = (size_t)p.n_units * p.n_kv_heads, B = p.n_keep, L = p.seq_len, E = L - B, D = p.head_dim;
    y.max_parts = (int)(2 * (E / kPiece) + 2);
    y.csr_passes = 1;                                        // digits of kCsrBits bits over the keys 0 .. B
    while (y.csr_passes < 6 && (B >> (kCsrBits * y.csr_passes)) != 0) ++y.csr_passes;
    y.merge_win = merge_window(p);
    y.n_win = (int)((L + y.merge_win - 1) / y.merge_win);
    y.sort_a = take(UH * E * 4);
    y.sort_b = take(UH * E * 4);
    y.rows = take(UH * L * 8);
    y.row_count = take(UH * 8);
    y.off = take(UH * (B + 1) * 4);
    y.first_slot = take(UH * ((L + kMinWin - 1) / kMinWin) * 4);   // (of the shortest windows, so that more rows never need less room)
    y.part_off = take(UH * (B + 1) * 4);
    y.pieces = take(UH * (size_t)y.max_parts * 16);
    y.partial = take(UH * (size_t)y.max_parts * (2 * D + 4) * 4);
    y.ticket = take(256);
    y.slot_done = take(UH * B * 4);
    y.merge_status = take(256);
    y.tokmap = take(UH * L * 8);
}

Layout make_layout(const flowmm_params &p) {
    Layout y;
    const size_t U = p.n_units, Hq = p.n_q_heads, Hkv = p.n_kv_heads, L = p.seq_len, W = p.window;
    const size_t B = p.n_keep, E = L - B, G = Hq / Hkv;
    const int row_tiles = (int)((G * W + kTile - 1) / kTile);
    y.n_chunk1 = chunks_for((int)L, (int)(U * Hkv) * row_tiles, y.chunk1);
    y.n_chunk2 = chunks_for((int)L, (int)(U * Hkv), y.chunk2);
    size_t o = 0;
    auto take = [&](size_t bytes) { const size_t at = o; o += align256(bytes); return at; };
    y.status = take(256);
    y.importance = take(U * Hkv * L * 4);
    y.cross_mass = take(U * Hq * 4);
    y.rho = take(U * 4);
    y.strategy = take(U * 4);
    y.retained = take(U * Hkv * B * 4);
    y.evicted = take(U * Hkv * E * 4);
    y.match = take(U * Hkv * E * 4);
    y.match_sim = take(U * Hkv * E * 4);
    y.n_rt = (int)((L + tcs::kItemRows - 1) / tcs::kItemRows);
    // Items of 256 proxy rows (pass 1) or keys (pass 2) take two halves of 128 against every operand tile.  Where that leaves SMs
    // idle and items of one half still have an SM each, they are of one half: their products and exponentials then take half as
    // long.  The whole call, us, 256 and 128: 8 heads of 1471 tokens, 224 rows 34.8, 32.8; 4 of 500 30.6, 28.1; 4 of 2300 45.1, 43.4;
    // 4 of 4500 51.8, 50.1; 8 of 1000, 512 rows 35.7, 32.8; 4 caches of 640 rows 37.2, 34.8; where pass 2 alone is cut finer 8 of
    // 2300 42.2, 41.1.
    y.tc_q_rows = G * W > tcs::kRows && U * Hkv * (size_t)y.n_rt * ((G * W + tcs::kRows - 1) / tcs::kRows) <= kScoreCtas ? tcs::kRows : tcs::kItemRows;
    // Pass 2 by items of 128 as well, on which all warps of a CTA work, where the longest run of them is at most two thirds of the longest of
    // items of 256: heads that end in half an item, few items per CTA.  The scoring, us, by 256 and by 128, 224 rows: runs of half the length
    // 56 heads of 640 tokens 21.7, 20.1, 96 of 300 21.0, 19.6; of two thirds 112 of 640 26.9, 25.7, 64 of 1150 27.0, 25.6, 168 of 300 25.5, 25.5; of
    // three quarters 16 of 2312 21.6, 23.2, 40 of 900 20.9, 21.8, 64 of 1664 29.8, 31.6, 32 of 1400 21.7, 21.6, 24 of 2000 24.0, 23.5.
    const size_t halves2 = U * Hkv * ((L + tcs::kRows - 1) / tcs::kRows), items2 = U * Hkv * (size_t)y.n_rt;
    const size_t run_items = (items2 + kScoreCtas - 1) / kScoreCtas, run_halves = (halves2 + kScoreCtas - 1) / kScoreCtas;
    y.tc_keys2 = halves2 <= kScoreCtas || 3 * run_halves <= 4 * run_items ? tcs::kRows : tcs::kItemRows;
    // pass 1 of the tensor-core scoring: the key tiles of all heads in equal runs, one per SM and tile of proxy rows
    y.tc_n_qt = (int)((G * W + y.tc_q_rows - 1) / y.tc_q_rows);
    {
        const size_t tiles = U * Hkv * (size_t)y.n_rt, runs = kScoreCtas > y.tc_n_qt ? kScoreCtas / y.tc_n_qt : 1;
        y.tc_runs = (int)(tiles < runs ? tiles : runs);
        const size_t spread = (size_t)y.tc_runs / (U * Hkv) + 2;          // runs that a head's tiles can be in
        y.tc_n_part = (int)(spread < (size_t)y.n_rt ? spread : (size_t)y.n_rt);
    }
    // Row statistics and partial masses: bounds of what the cuts above come to for all heads (records of 16 bytes, of the SIMT kernels of
    // 8, per proxy row) that, unlike those, never fall when units or tokens are added.
    const size_t UH = U * Hkv, key_tiles = (L + kTile - 1) / kTile, qt = (G * W + tcs::kItemRows - 1) / tcs::kItemRows;
    const size_t parts = std::min(UH * (size_t)y.n_rt, std::max<size_t>(kScoreCtas / qt, 1) + 2 * UH);
    const size_t simt1 = std::min(UH * key_tiles, kSimtCtas / row_tiles + 1 + UH), simt2 = std::min(UH * key_tiles, kSimtCtas + UH);
    y.row_part = take(G * W * std::max(16 * parts, 8 * simt1));
    y.cross_part = take(G * std::max(simt2, UH * std::max<size_t>(W, 8)) * 4);
    y.row_all = take(U * Hq * W * 16);
    layout_merge(y, p, take);
    y.merge_status = y.status;
    y.c_tot = (int)((B + 31) / 32 * 32 + 32);
    y.cand_k = take(U * Hkv * (size_t)y.c_tot * 128 * 2);
    y.cand_scale = take(U * Hkv * (size_t)y.c_tot * 4 + 1024);   // + one tile of slack: whole 256-column slices are copied
    y.cand_slot = take(U * Hkv * (size_t)y.c_tot * 4);
    y.cand_count = take(U * Hkv * 2 * 4);
    y.rank = take(U * Hkv * L * 4);
    y.evi_mod = take(U * Hkv * E);
    y.n_et = (int)((E + kMtItemRows - 1) / kMtItemRows);
    y.tile_mod = take(U * Hkv * (size_t)y.n_et);
    y.total = o;
    return y;
}

flowmm_status validate(const flowmm_params *p) {
    if (!p) return FLOWMM_ERR_NULL;
    if (p->n_units < 1 || p->n_q_heads < 1 || p->n_kv_heads < 1) return FLOWMM_ERR_SHAPE;
    if (p->n_q_heads % p->n_kv_heads != 0) return FLOWMM_ERR_SHAPE;
    if (p->head_dim != 64 && p->head_dim != 128) return FLOWMM_ERR_SHAPE;
    if (p->seq_len < 1 || p->window < 1 || p->window > p->seq_len) return FLOWMM_ERR_SHAPE;
    if ((int64_t)p->n_units * p->n_kv_heads > kMaxHeadsPerCall) return FLOWMM_ERR_SHAPE;
    {   // work items (pairs x 128-row tiles of the context x 128-row tiles of a head's proxy rows) are counted in 32 bits
        const int64_t tiles = (int64_t)p->n_units * p->n_kv_heads * ((p->seq_len + 127) / 128) *
                              (((int64_t)p->n_q_heads / p->n_kv_heads * p->window + 127) / 128);
        if (tiles > 0x7FFFFFFFll) return FLOWMM_ERR_SHAPE;
    }
    if (p->n_keep < 1 || p->n_keep > p->seq_len) return FLOWMM_ERR_BUDGET;
    if (p->keep_window && p->n_keep < p->window) return FLOWMM_ERR_BUDGET;
    if (p->dtype != FLOWMM_F32 && p->dtype != FLOWMM_BF16) return FLOWMM_ERR_DTYPE;
    if (p->tau_mode < 0 || p->tau_mode > 1 || p->flow_mode < 0 || p->flow_mode > 3 || p->merge_mode < 0 ||
        p->merge_mode > 1 || p->path < 0 || p->path > 1)
        return FLOWMM_ERR_SHAPE;
    if (!(p->softmax_scale >= 0.f) || isnan(p->theta) || isnan(p->tau)) return FLOWMM_ERR_SHAPE;
    return FLOWMM_OK;
}

bool strides_ok(const int64_t s[3], int head_dim) {
    for (int i = 0; i < 3; ++i)
        if (s[i] < 0 || s[i] % 8 != 0) return false;
    return s[2] >= head_dim;
}
bool aligned16(const void *ptr) { return (reinterpret_cast<uintptr_t>(ptr) & 15) == 0; }

flowmm_status check_device() {
    int dev = 0, major = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return FLOWMM_ERR_CUDA;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) return FLOWMM_ERR_CUDA;
    return major == 10 ? FLOWMM_OK : FLOWMM_ERR_UNSUPPORTED_DEVICE;
}

flowmm_status check_ws(const flowmm_params *p, const void *ws, size_t ws_bytes, Layout &y) {
    if (!ws) return FLOWMM_ERR_NULL;
    if (reinterpret_cast<uintptr_t>(ws) & 255) return FLOWMM_ERR_ALIGN;
    y = make_layout(*p);
    if (ws_bytes < y.total) return FLOWMM_ERR_WORKSPACE;
    return FLOWMM_OK;
}

template <typename X> X *at(void *ws, size_t off) { return reinterpret_cast<X *>(static_cast<char *>(ws) + off); }

float tau_effective(const flowmm_params &p) {
    return p.tau_mode == FLOWMM_TAU_REL ? (float)((double)p.tau * (double)p.window / (double)p.seq_len) : p.tau;
}

// ---- debug build: the index lists a caller hands in are checked before any kernel uses them ---------
#ifdef FLOWMM_DEBUG
// One block per (unit, head): pivots and non-pivots inside [0, L) and strictly ascending, matches inside [-1, B).
__global__ void debug_check_lists_kernel(const int32_t *retained, const int32_t *evicted, const int32_t *match,
                                         int L, int B, int E, int *status) {
    predecessor_done();
    const int uh = blockIdx.x;
    bool bad = false;
    if (retained)
        for (int s = threadIdx.x; s < B; s += blockDim.x) {
            const int r = retained[(int64_t)uh * B + s];
            bad |= r < 0 || r >= L || (s > 0 && retained[(int64_t)uh * B + s - 1] >= r);
        }
    if (evicted)
        for (int j = threadIdx.x; j < E; j += blockDim.x) {
            const int e = evicted[(int64_t)uh * E + j];
            bad |= e < 0 || e >= L || (j > 0 && evicted[(int64_t)uh * E + j - 1] >= e);
        }
    if (match)
        for (int j = threadIdx.x; j < E; j += blockDim.x) {
            const int m = match[(int64_t)uh * E + j];
            bad |= m < -1 || m >= B;
        }
    if (bad) atomicCAS(status, 0, kStatusIndex);
}

// Runs the check, waits for it and reports: the entry point launches nothing else when a list is bad.
flowmm_status debug_check_lists(const flowmm_params &p, const int32_t *retained, const int32_t *evicted,
                                const int32_t *match, int *status, cudaStream_t st) {
    launch(debug_check_lists_kernel, p.n_units * p.n_kv_heads, 256, 0, st, retained, evicted, match, p.seq_len, p.n_keep,
                                                                        p.seq_len - p.n_keep, status);
    if (cudaGetLastError() != cudaSuccess) return FLOWMM_ERR_CUDA;
    int32_t word = 0;
    if (cudaMemcpyAsync(&word, status, sizeof(word), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return FLOWMM_ERR_CUDA;
    return word == kStatusIndex ? FLOWMM_ERR_INDEX : FLOWMM_OK;
}
#define FLOWMM_DEBUG_LISTS(p, ret, evi, mt, status, st) FLOWMM_TRY(debug_check_lists(p, ret, evi, mt, status, st))
#else
#define FLOWMM_DEBUG_LISTS(p, ret, evi, mt, status, st) do { } while (0)
#endif

// ---- step launchers (no validation; the entry points below validate) --------------------------

bool use_tc(const flowmm_params &p) {
    return p.path == FLOWMM_PATH_AUTO && p.dtype == FLOWMM_BF16 && p.head_dim == 128;
}
bool use_tc_score(const flowmm_params &p) {
    const int gw = p.n_q_heads / p.n_kv_heads * p.window;
    return use_tc(p) && (p.window == 32 || p.window == 64 || p.window == 128) && gw <= 1024;
}

// Row records of a head that the CTAs of the second scoring pass join themselves when they come to it; more are joined by a launch
// in between, which costs 2 to 3 us.  The whole call, us, without and with it: 6 records of 224 rows 36.5, 38.7; 11 of 224 86.0, 86.6;
// 11 of 512 98.0, 96.8 and 249.5, 248.5.
constexpr int kMaxHeadRecords = 4096;

flowmm_status run_score_tc(const flowmm_params &p, const Layout &y, const void *q, const void *k, const uint8_t *mod,
                           float *importance, float *cross_mass, void *ws, cudaStream_t st, int *parts_out) {
    const int UH = p.n_units * p.n_kv_heads, G = p.n_q_heads / p.n_kv_heads, W = p.window;
    ScoreTcArgs a;
    a.row_part = at<float4>(ws, y.row_part); a.modality = mod;
    a.importance = importance; a.cross_part = at<float>(ws, y.cross_part); a.status = at<int>(ws, y.status);
    a.Hq = p.n_q_heads; a.Hkv = p.n_kv_heads; a.G = G; a.W = W; a.L = p.seq_len; a.GW = G * W;
    a.q_rows = y.tc_q_rows; a.n_qt = y.tc_n_qt; a.n_runs1 = y.tc_runs; a.n_part = y.tc_n_part; a.n_rt = y.n_rt;
    a.a_heads = G < tcs::kRows / W ? G : tcs::kRows / W;        // one A half holds 128 proxy rows
    // pass 2 streams the keys as the A operand; with up to 256 proxy rows per KV head the shapes with two A stages keep
    // the key loads in flight across items
    const bool small2 = a.GW <= 128 && W <= 64, resident2 = !small2 && a.GW <= 256;
    const int nb2 = small2 ? tcs::Small::kCols : tcs::Big::kCols;
    a.b_heads = G < nb2 / W ? G : nb2 / W;
    a.n_tiles1 = UH * a.n_rt;
    a.keys2 = y.tc_keys2; a.n_rt2 = (p.seq_len + a.keys2 - 1) / a.keys2; a.n_items2 = UH * a.n_rt2;
    const int grid1 = a.n_runs1 * a.n_qt;
    const int grid2 = a.n_items2 < tc::sm_count() ? a.n_items2 : tc::sm_count();
    a.by_grid1 = make_fastdiv((uint32_t)grid1); a.by_grid2 = make_fastdiv((uint32_t)grid2);
    a.by_hkv = make_fastdiv((uint32_t)p.n_kv_heads); a.by_rt = make_fastdiv((uint32_t)a.n_rt); a.by_rt2 = make_fastdiv((uint32_t)a.n_rt2);
    a.by_tiles = make_fastdiv((uint32_t)a.n_tiles1);
    const float scale = p.softmax_scale != 0.f ? p.softmax_scale : 1.f / sqrtf((float)p.head_dim);
    a.scale_log2 = scale * kLog2e;

    CUtensorMap qa, qb, k128, k256;
    const uint64_t qd[4] = {128, (uint64_t)W, (uint64_t)p.n_q_heads, (uint64_t)p.n_units};
    const uint64_t qs[3] = {(uint64_t)p.q_stride[2] * 2, (uint64_t)p.q_stride[1] * 2, (uint64_t)p.q_stride[0] * 2};
    const uint64_t kd[4] = {128, (uint64_t)p.seq_len, (uint64_t)p.n_kv_heads, (uint64_t)p.n_units};
    const uint64_t ks[3] = {(uint64_t)p.k_stride[2] * 2, (uint64_t)p.k_stride[1] * 2, (uint64_t)p.k_stride[0] * 2};
    const uint32_t bqa[4] = {64, (uint32_t)W, (uint32_t)a.a_heads, 1}, bqb[4] = {64, (uint32_t)W, (uint32_t)a.b_heads, 1};
    const uint32_t bk128[4] = {64, tcs::kRows, 1, 1}, bk256[4] = {64, tcs::Big::kCols, 1, 1};
    if (!tc::make_bf16_map(&qa, q, 4, qd, qs, bqa) || !tc::make_bf16_map(&qb, q, 4, qd, qs, bqb) ||
        !tc::make_bf16_map(&k128, k, 4, kd, ks, bk128) || !tc::make_bf16_map(&k256, k, 4, kd, ks, bk256))
        return FLOWMM_ERR_CUDA;
    const bool split2 = a.keys2 == tcs::kRows;
    auto pass2 = small2 ? (split2 ? score_colsum_tc_kernel<tcs::Small, true> : score_colsum_tc_kernel<tcs::Small, false>)
                 : resident2 ? (split2 ? score_colsum_tc_kernel<tcs::Resident, true> : score_colsum_tc_kernel<tcs::Resident, false>)
                             : (split2 ? score_colsum_tc_kernel<tcs::Big, true> : score_colsum_tc_kernel<tcs::Big, false>);
    const uint32_t smem2 = small2 ? tcs::Small::kSmemBytes : resident2 ? tcs::Resident::kSmemBytes : tcs::Big::kSmemBytes;
    if (cudaFuncSetAttribute(score_stats_tc_kernel<tcs::Big>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)tcs::Big::kSmemBytes) != cudaSuccess ||
        cudaFuncSetAttribute(pass2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2) != cudaSuccess)
        return FLOWMM_ERR_CUDA;
    launch(score_stats_tc_kernel<tcs::Big>, grid1, tcs::kThreads, tcs::Big::kSmemBytes, st, qa, k256, a);
    FLOWMM_LAUNCHED("score_stats_tc");
    a.row_all = nullptr;
    if (a.n_part * a.GW > kMaxHeadRecords) {
        float4 *all = at<float4>(ws, y.row_all);
        const int n_rows = UH * a.GW;
        launch(score_combine_kernel<4>, (n_rows + 63) / 64, 256, 0, st, a, n_rows, all);
        FLOWMM_LAUNCHED("score_combine");
        a.row_all = all;
    }
    launch(pass2, grid2, tcs::kThreads, smem2, st, k128, qb, a);
    FLOWMM_LAUNCHED("score_colsum_tc");
    if (parts_out) { *parts_out = W; return FLOWMM_OK; }              // the caller adds the rows' shares up itself
    const int n = p.n_units * p.n_q_heads;
    launch(cross_mass_reduce, (n + 7) / 8, 256, 0, st, a.cross_part, W, n, cross_mass);
    FLOWMM_LAUNCHED("cross_mass_reduce");
    return FLOWMM_OK;
}

// Short contexts with 32 proxy rows per KV head: every logit of a head fits in half of TMEM, K is read once.
bool use_fused_score(const flowmm_params &p) {
    const int gw = p.n_q_heads / p.n_kv_heads * p.window, nt = (p.seq_len + sft::kTile - 1) / sft::kTile;
    return use_tc(p) && gw == sft::kRows && nt <= sft::kMaxTiles;
}

flowmm_status run_score_fused(const flowmm_params &p, const Layout &y, const void *q, const void *k, const uint8_t *mod,
                              float *importance, float *cross_mass, void *ws, cudaStream_t st) {
    const int UH = p.n_units * p.n_kv_heads, G = p.n_q_heads / p.n_kv_heads, W = p.window;
    CUtensorMap qmap, kmap;
    const uint64_t qd[4] = {128, (uint64_t)W, (uint64_t)p.n_q_heads, (uint64_t)p.n_units};
    const uint64_t qs[3] = {(uint64_t)p.q_stride[2] * 2, (uint64_t)p.q_stride[1] * 2, (uint64_t)p.q_stride[0] * 2};
    const uint64_t kd[4] = {128, (uint64_t)p.seq_len, (uint64_t)p.n_kv_heads, (uint64_t)p.n_units};
    const uint64_t ks[3] = {(uint64_t)p.k_stride[2] * 2, (uint64_t)p.k_stride[1] * 2, (uint64_t)p.k_stride[0] * 2};
    const uint32_t bq[4] = {64, (uint32_t)W, (uint32_t)G, 1}, bk[4] = {64, sft::kTile, 1, 1};
    if (!tc::make_bf16_map(&qmap, q, 4, qd, qs, bq) || !tc::make_bf16_map(&kmap, k, 4, kd, ks, bk)) return FLOWMM_ERR_CUDA;
    sft::Args a;
    a.modality = mod; a.importance = importance; a.cross_mass = cross_mass; a.status = at<int>(ws, y.status);
    a.Hq = p.n_q_heads; a.Hkv = p.n_kv_heads; a.G = G; a.W = W; a.L = p.seq_len; a.n_items = UH;
    const float scale = p.softmax_scale != 0.f ? p.softmax_scale : 1.f / sqrtf((float)p.head_dim);
    a.scale_log2 = scale * kLog2e;
    if (cudaFuncSetAttribute(sft::score_fused_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sft::kSmemBytes) != cudaSuccess)
        return FLOWMM_ERR_CUDA;
    const int grid = UH < tc::sm_count() ? UH : tc::sm_count();
    launch(sft::score_fused_tc_kernel, grid, sft::kThreads, sft::kSmemBytes, st, qmap, kmap, a);
    FLOWMM_LAUNCHED("score_fused_tc");
    return FLOWMM_OK;
}

// Clusters of `ctas` CTAs of the one-pass scoring that run at once on the current device, an SM for each CTA (score_cluster_tc.cuh asks for too
// much shared memory for two).  A cluster's CTAs are in one group of SMs, so by fours 132 of 148 find room, by sevens 105.  Clusters of an odd size
// do not always find the last places: a sixteenth less (the call by two passes and so: 42 heads of 730 tokens by threes 32.5, 28.7, 44 of 704 31.1,
// 33.0, 45 of 678 32.7, 34.5; 26 of 625 by fives 30.8, 29.2, 25 of 606 31.2, 26.9; by an even size to the last, 74 of 223 by twos 28.5, 24.0).
// Asked for once per device and size (a benign race: every thread would store the same value).
int score_clusters_at_once(int ctas) {
    constexpr int kSlots = 64;
    static std::atomic<int> known[kSlots][sct::kMaxCtas + 1];            // one more than the answer; 0: not asked for yet
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 0;
    if (dev < kSlots && (n = known[dev][ctas].load(std::memory_order_relaxed)) != 0) return n - 1;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = ctas; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas); cfg.blockDim = dim3(sct::kThreads); cfg.dynamicSmemBytes = sct::kMinSmem; cfg.attrs = &attr; cfg.numAttrs = 1;
    if (!allow_smem(sct::score_cluster_tc_kernel) ||
        cudaOccupancyMaxActiveClusters(&n, sct::score_cluster_tc_kernel, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (ctas > 1 && ctas % 2 == 1) n -= n / 16;
    if (dev < kSlots) known[dev][ctas].store(n + 1, std::memory_order_relaxed);
    return n;
}

// One pass by clusters (score_cluster_tc.cuh) where all of them run at once: a cluster's CTAs take 9 us one after the other what the two passes
// take side by side.  The scoring, us, by two passes and so: 20 heads of 709 tokens, 128 rows, by sixes 12.0, 9.1; 28 of 986, 224 rows, by
// fours 15.9, 12.4; where some clusters come second 16 of 791, 128 rows, by sevens 11.9, 14.9; 48 of 306, 96 rows, by threes 11.9, 13.6.
// Rows short of a tile leave lanes without one.  64 rows: 4 heads of 640 tokens 11.3, 8.6, 28 of 2000 17.6, 12.9; by four key tiles to a CTA, beyond
// 2048 tokens, 4 of 3000 11.9, 12.4, so not there.  32 rows: 4 of 1500 11.0, 9.5, of 3000 11.5, 11.7, 32 of 2000, whole call, 45.2, 51.8.  Key tiles
// per CTA: the fewest that fit; returns the CTAs per head (0: not so).
int cluster_score_split(const flowmm_params &p, int &kt) {
    const int gw = p.n_q_heads / p.n_kv_heads * p.window, rt = (gw + sct::kTile - 1) / sct::kTile, nt = (p.seq_len + sct::kTile - 1) / sct::kTile;
    const int64_t heads = (int64_t)p.n_units * p.n_kv_heads;
    if (!use_tc_score(p) || gw < 64 || rt > sct::kMaxAcc || heads > kScoreCtas) return 0;
    for (kt = 1; rt * kt <= sct::kMaxAcc && (gw >= 96 || kt <= 2); kt *= 2) {
        const int ctas = (nt + kt - 1) / kt;
        if (ctas <= sct::kMaxCtas && heads <= score_clusters_at_once(ctas)) return ctas;
    }
    return 0;
}

flowmm_status run_score_cluster(const flowmm_params &p, const Layout &y, const void *q, const void *k, const uint8_t *mod, float *importance, int kt,
                                int ctas, void *ws, cudaStream_t st) {
    const int UH = p.n_units * p.n_kv_heads, G = p.n_q_heads / p.n_kv_heads, W = p.window;
    sct::Args a;
    a.modality = mod; a.importance = importance; a.cross_part = at<float>(ws, y.cross_part); a.status = at<int>(ws, y.status);
    a.Hq = p.n_q_heads; a.Hkv = p.n_kv_heads; a.G = G; a.W = W; a.L = p.seq_len; a.GW = G * W;
    a.rt = (a.GW + sct::kTile - 1) / sct::kTile; a.kt = kt; a.ctas = ctas;
    const int q_heads = G < sct::kTile / W ? G : sct::kTile / W;      // of a tile of proxy rows
    a.q_bytes = (uint32_t)(q_heads * W) * 256u;
    const float scale = p.softmax_scale != 0.f ? p.softmax_scale : 1.f / sqrtf((float)p.head_dim);
    a.scale_log2 = scale * kLog2e;
    CUtensorMap qmap, kmap;
    const uint64_t qd[4] = {128, (uint64_t)W, (uint64_t)p.n_q_heads, (uint64_t)p.n_units};
    const uint64_t qs[3] = {(uint64_t)p.q_stride[2] * 2, (uint64_t)p.q_stride[1] * 2, (uint64_t)p.q_stride[0] * 2};
    const uint64_t kd[4] = {128, (uint64_t)p.seq_len, (uint64_t)p.n_kv_heads, (uint64_t)p.n_units};
    const uint64_t ks[3] = {(uint64_t)p.k_stride[2] * 2, (uint64_t)p.k_stride[1] * 2, (uint64_t)p.k_stride[0] * 2};
    const uint32_t bq[4] = {64, (uint32_t)W, (uint32_t)q_heads, 1}, bk[4] = {64, sct::kTile, 1, 1};
    if (!tc::make_bf16_map(&qmap, q, 4, qd, qs, bq) || !tc::make_bf16_map(&kmap, k, 4, kd, ks, bk)) return FLOWMM_ERR_CUDA;
    const uint32_t smem = sct::smem_bytes(a.rt, kt);
    if (!allow_smem(sct::score_cluster_tc_kernel)) return FLOWMM_ERR_CUDA;
    launch_cluster(dim3(ctas), sct::score_cluster_tc_kernel, UH * ctas, sct::kThreads, smem, st, qmap, kmap, a);
    FLOWMM_LAUNCHED("score_cluster_tc");
    return FLOWMM_OK;
}

// The scoring of short contexts in one launch: a key tile per CTA or two, a row per thread or four.
template <typename T>
auto cluster_score_kernel(bool one_tile, bool one_row) {
    return one_tile ? (one_row ? score_cluster_simt<T, 1, 1> : score_cluster_simt<T, 1, 4>) : (one_row ? score_cluster_simt<T, 2, 1> : score_cluster_simt<T, 2, 4>);
}

// parts_out: the caller reduces the partial cross-modal masses itself; set to 0 when cross_mass is already final
flowmm_status run_score(const flowmm_params &p, const Layout &y, const void *q, const void *k, const uint8_t *mod,
                        float *importance, float *cross_mass, void *ws, cudaStream_t st, int *parts_out = nullptr) {
    if (use_fused_score(p)) {
        if (parts_out) *parts_out = 0;
        return run_score_fused(p, y, q, k, mod, importance, cross_mass, ws, st);
    }
    int kt = 0;
    if (const int ctas = cluster_score_split(p, kt)) {
        FLOWMM_TRY(run_score_cluster(p, y, q, k, mod, importance, kt, ctas, ws, st));
        if (parts_out) { *parts_out = p.window; return FLOWMM_OK; }  // the caller adds the rows' shares up itself
        const int n = p.n_units * p.n_q_heads;
        launch(cross_mass_reduce, (n + 7) / 8, 256, 0, st, at<float>(ws, y.cross_part), p.window, n, cross_mass);
        FLOWMM_LAUNCHED("cross_mass_reduce");
        return FLOWMM_OK;
    }
    if (use_tc_score(p)) return run_score_tc(p, y, q, k, mod, importance, cross_mass, ws, st, parts_out);
    ScoreArgs a;
    a.q = q; a.k = k; a.modality = mod; a.importance = importance;
    a.row_part = at<float2>(ws, y.row_part);
    a.cross_part = at<float>(ws, y.cross_part);
    a.Hq = p.n_q_heads; a.Hkv = p.n_kv_heads; a.G = p.n_q_heads / p.n_kv_heads;
    a.D = p.head_dim; a.L = p.seq_len; a.W = p.window;
    a.n_chunk1 = y.n_chunk1; a.chunk1 = y.chunk1; a.n_chunk2 = y.n_chunk2; a.chunk2 = y.chunk2;
    const float scale = p.softmax_scale != 0.f ? p.softmax_scale : 1.f / sqrtf((float)p.head_dim);
    a.scale_log2 = scale * kLog2e;
    for (int i = 0; i < 3; ++i) { a.qs[i] = p.q_stride[i]; a.ks[i] = p.k_stride[i]; }
    const int GW = a.G * a.W;
    const int UH = p.n_units * p.n_kv_heads;
    const int key_tiles = (p.seq_len + kTile - 1) / kTile;
    int n_parts = y.n_chunk2;
    if (GW <= kTile && key_tiles <= kClusterScoreTiles) {    // the logits fit the registers of a cluster
        const int ctas = key_tiles <= 8 ? key_tiles : (key_tiles + 1) / 2;
        n_parts = ctas;                                      // (8 parts per head always have room)
        auto kernel = p.dtype == FLOWMM_BF16 ? cluster_score_kernel<__nv_bfloat16>(key_tiles <= 8, GW <= 16) : cluster_score_kernel<float>(key_tiles <= 8, GW <= 16);
        launch_cluster(dim3(ctas), kernel, UH * ctas, kSimtThreads, 0, st, a, ctas);
        FLOWMM_LAUNCHED("score_cluster_simt");
    } else {
        const dim3 g1(UH, (GW + kTile - 1) / kTile, y.n_chunk1), g2(UH, y.n_chunk2);
        const size_t dyn = (size_t)3 * GW * sizeof(float);
        if (p.dtype == FLOWMM_BF16) {
            launch(score_stats_simt<__nv_bfloat16>, g1, kSimtThreads, 0, st, a);
            FLOWMM_LAUNCHED("score_stats_simt");
            launch(score_colsum_simt<__nv_bfloat16>, g2, kSimtThreads, dyn, st, a);
            FLOWMM_LAUNCHED("score_colsum_simt");
        } else {
            launch(score_stats_simt<float>, g1, kSimtThreads, 0, st, a);
            FLOWMM_LAUNCHED("score_stats_simt");
            launch(score_colsum_simt<float>, g2, kSimtThreads, dyn, st, a);
            FLOWMM_LAUNCHED("score_colsum_simt");
        }
    }
    if (parts_out) { *parts_out = n_parts; return FLOWMM_OK; }
    const int n = p.n_units * p.n_q_heads;
    launch(cross_mass_reduce, (n + 7) / 8, 256, 0, st, a.cross_part, n_parts, n, cross_mass);
    FLOWMM_LAUNCHED("cross_mass_reduce");
    return FLOWMM_OK;
}

flowmm_status run_layer_flow(const flowmm_params &p, const float *cross_mass, float *rho, int32_t *strategy,
                             cudaStream_t st) {
    launch(layer_flow_kernel, (p.n_units + 127) / 128, 128, 0, st, cross_mass, p.n_units, p.n_q_heads, p.window, p.theta,
                                                                p.flow_mode, rho, strategy);
    FLOWMM_LAUNCHED("layer_flow");
    return FLOWMM_OK;
}

// What the preparation of the tensor-core matching step needs (candidate layout per head; see match_tc.cuh).
MatchPrepArgs match_prep_args(const flowmm_params &p, const Layout &y, const void *k, const float *importance,
                              const uint8_t *mod, const int32_t *retained, const int32_t *evicted, void *ws) {
    MatchPrepArgs g;
    g.k = k; g.importance = importance; g.modality = mod;
    g.retained = retained; g.evicted = evicted;
    g.cand_k = at<__nv_bfloat16>(ws, y.cand_k); g.cand_scale = at<float>(ws, y.cand_scale);
    g.cand_slot = at<int>(ws, y.cand_slot); g.cand_count = at<int>(ws, y.cand_count);
    g.rank = at<int>(ws, y.rank); g.evi_mod = at<uint8_t>(ws, y.evi_mod); g.tile_mod = at<uint8_t>(ws, y.tile_mod);
    g.Hkv = p.n_kv_heads; g.L = p.seq_len; g.B = p.n_keep; g.E = p.seq_len - p.n_keep; g.Ctot = y.c_tot; g.n_rt = y.n_et;
    g.tau_eff = tau_effective(p);
    for (int i = 0; i < 3; ++i) g.ks[i] = p.k_stride[i];
    g.copy_here = y.c_tot <= 256;
    g.status = at<int>(ws, y.status);
    return g;
}

template <int kThreads, bool kOneChunk, int kCtas = 1, bool kFew = false>
flowmm_status launch_select(const SelectArgs &a, const SelectFlow &f, const MatchPrepArgs &g, int with_prepare, cudaStream_t st) {
    const size_t smem = select_smem(a.chunk);
    if (!allow_smem(select_topb_kernel<kThreads, kOneChunk, kCtas, kFew>, 1024)) return FLOWMM_ERR_CUDA;
    launch_cluster(dim3(kCtas), select_topb_kernel<kThreads, kOneChunk, kCtas, kFew>, (a.n_heads + f.n_units) * kCtas, kThreads, smem, st, a, f, g, with_prepare);
    FLOWMM_LAUNCHED("select_topb");
    return FLOWMM_OK;
}

bool use_match_merge(const flowmm_params &p);

// flow != nullptr: the launch also applies Eq. 6 and the theta rule (SelectFlow's comments).
// prep != nullptr: each block goes on to prepare its head's matching candidates (tensor-core matching).
// row_mod, row_mod_out: the pivots' modalities are written as well, from one modality map per head.
flowmm_status run_select(const flowmm_params &p, const float *importance, int32_t *retained, int32_t *evicted,
                         cudaStream_t st, const SelectFlow *flow = nullptr, const MatchPrepArgs *prep = nullptr,
                         const uint8_t *row_mod = nullptr, uint8_t *row_mod_out = nullptr) {
    SelectArgs a;
    a.importance = importance; a.retained = retained; a.evicted = evicted; a.row_mod_out = row_mod_out;
    a.n_heads = p.n_units * p.n_kv_heads; a.L = p.seq_len; a.B = p.n_keep; a.W = p.window; a.keep_window = p.keep_window;
    a.chunk = p.seq_len <= kSelMaxChunk ? (p.seq_len + 31) / 32 * 32 : kSelMaxChunk;
    const SelectFlow no_flow = {};
    // Heads that leave SMs free, the short-list matching behind them (a block per SM; not the small blocks that gather long lists) and up to
    // five tiles of 128 tokens per SM for it.  The whole call, with and without: 32 heads of 640 tokens 23.1, 23.5 us; 16 of 2000 36.1, 36.4, with
    // 7 query heads each 41.6, 42.4; one of 206 16.4, 16.8; but 72 of 1500 49.3, 45.9; 52 of 2500 54.4, 51.5; 40 of 3500 61.5, 58.6; with the
    // matching and the merge in one launch 76 of 640 25.0, 23.6, of 2600 66.7, 62.8.  (4 heads whose keys and queries are still in L2 from the call
    // before: of 400 23.3, 22.4.)
    const int64_t tiles = (int64_t)a.n_heads * ((p.seq_len + mst::kTile - 1) / mst::kTile);
    a.lets_in = prep && prep->copy_here && !use_match_merge(p) && 3 * (a.n_heads + p.n_units) <= 2 * tc::sm_count() &&
                tiles <= 5 * tc::sm_count();
    MatchPrepArgs g = {};
    g.Hkv = 1; g.modality = row_mod;
    if (prep) g = *prep;
    const SelectFlow &f = flow ? *flow : no_flow;
    // Warps per head: a block's latency is its rounds of shared-memory work, which shrink with more warps until the
    // barriers outweigh them (640 tokens) or other heads' blocks no longer fit beside it
    // Long contexts of few heads: four CTAs for each (from about 6000 positions on their shares outweigh the cluster's
    // barriers; two save less, eight no more)
    const int part = (p.seq_len + 1023) / 1024 * 256;
    if (p.seq_len >= 6144 && part <= kSelMaxChunk && 4 * a.n_heads <= tc::sm_count()) {
        a.chunk = part;
        return launch_select<512, true, 4>(a, f, g, prep != nullptr, st);
    }
    // More heads than four blocks of 256 threads per SM would be in two rounds; of 128 threads an SM holds eight.  (1024 heads of 640
    // positions 151.4 -> 149.5 us for the call, of 1000 222.7 -> 221.4; of 400, where a block's rounds are short, 110.4 -> 111.5.)  Not beyond
    // 64 query heads a unit, which its own block takes by warps, one chain of loads after the other: 864 heads of 600 positions with 64, 128 and
    // 256 query heads a unit 142.1, 159.8, 205.2 us by 256 threads, 140.2, 162.4, 218.7 by 128.
    if (p.seq_len > 512 && p.seq_len <= 1024 && a.n_heads > 4 * tc::sm_count() && (f.n_units == 0 || f.Hq <= 64))
        return launch_select<128, true, 1, true>(a, f, g, prep != nullptr, st);
    // A block that has an SM for itself takes twice the warps: 32 heads of 640 positions 23.5 -> 23.0 us for the call, 4 of 3000 42.5 -> 41.7, 112
    // of 900 67.1 -> 65.4, of 2176 110.6 -> 109.5; of 4 heads of 192 17.9 -> 18.3, so from 257 positions on.
    const bool alone = a.n_heads + p.n_units <= tc::sm_count();
    if (p.seq_len <= (alone ? 256 : 1024)) return launch_select<256, true, 1, true>(a, f, g, prep != nullptr, st);
    if (p.seq_len <= (alone ? 1024 : 4096)) return launch_select<512, true, 1, true>(a, f, g, prep != nullptr, st);
    if (p.seq_len <= 4096) return launch_select<1024, true, 1, true>(a, f, g, prep != nullptr, st);
    if (p.seq_len <= kSelMaxChunk) return launch_select<1024, true>(a, f, g, prep != nullptr, st);
    return launch_select<1024, false>(a, f, g, prep != nullptr, st);
}

flowmm_status run_match_tc(const flowmm_params &p, const Layout &y, const void *k, const float *importance,
                           const uint8_t *mod, const int32_t *retained, const int32_t *evicted,
                           const int32_t *strategy, int32_t *match, float *match_sim, void *ws, cudaStream_t st,
                           int2 *tokmap, bool prepared) {
    const int UH = p.n_units * p.n_kv_heads, E = p.seq_len - p.n_keep;
    const MatchPrepArgs g = match_prep_args(p, y, k, importance, mod, retained, evicted, ws);
    if (!prepared) {                                 // (the fused call's selection launch has done it already)
        const int slices = (p.seq_len + kPrepSlice - 1) / kPrepSlice;
        launch(p.n_keep <= kPrepThreads ? match_prepare_kernel<1> : match_prepare_kernel<8>, dim3(UH, 1 + (slices < 64 ? slices : 64)), kPrepThreads, 0, st, g);
        FLOWMM_LAUNCHED("match_prepare");
    }
    if (!g.copy_here) {
        launch(match_gather_kernel, dim3(UH, (y.c_tot + 63) / 64), 256, 0, st, g);
        FLOWMM_LAUNCHED("match_gather");
    }

    CUtensorMap k_map, cand_map;
    const uint64_t kd[4] = {128, (uint64_t)p.seq_len, (uint64_t)p.n_kv_heads, (uint64_t)p.n_units};
    const uint64_t ks[3] = {(uint64_t)p.k_stride[2] * 2, (uint64_t)p.k_stride[1] * 2, (uint64_t)p.k_stride[0] * 2};
    const uint64_t cd[4] = {128, (uint64_t)y.c_tot, (uint64_t)UH, 1};
    const uint64_t cs[3] = {256, (uint64_t)y.c_tot * 256, (uint64_t)y.c_tot * 256 * (uint64_t)UH};
    if (y.c_tot <= mst::kMaxCols) {      // the whole candidate list of a head is one operand tile
        const uint32_t box_t[4] = {64, mst::kTile, 1, 1}, box_c[4] = {64, (uint32_t)y.c_tot, 1, 1};
        if (!tc::make_bf16_map(&k_map, k, 4, kd, ks, box_t) || !tc::make_bf16_map(&cand_map, g.cand_k, 4, cd, cs, box_c))
            return FLOWMM_ERR_CUDA;
        mst::Args a;
        a.cand_count = g.cand_count; a.cand_slot = g.cand_slot; a.rank = g.rank; a.strategy = strategy;
        a.cand_scale = g.cand_scale; a.modality = mod; a.match = match; a.match_sim = match_sim;
        a.tokmap = tokmap; a.merge_mode = p.merge_mode;
        a.status = at<int>(ws, y.status);
        a.Hkv = p.n_kv_heads; a.L = p.seq_len; a.E = E; a.Ctot = y.c_tot; a.n_heads = UH;
        const int tiles = (p.seq_len + mst::kTile - 1) / mst::kTile;
        a.by_nt = make_fastdiv((uint32_t)tiles); a.by_hkv = make_fastdiv((uint32_t)p.n_kv_heads);
        const int64_t n_tiles = (int64_t)UH * tiles;
        if (cudaFuncSetAttribute(mst::match_small_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)mst::kSmemBytes) != cudaSuccess)
            return FLOWMM_ERR_CUDA;
        launch(mst::match_small_tc_kernel, n_tiles < tc::sm_count() ? (int)n_tiles : tc::sm_count(), mst::kThreads, mst::kSmemBytes, st, k_map, cand_map, a);
        FLOWMM_LAUNCHED("match_small_tc");
        return FLOWMM_OK;
    }
    const uint32_t box_b[4] = {64, tcs::Big::kCols, 1, 1};
    if (!tc::make_bf16_map(&cand_map, g.cand_k, 4, cd, cs, box_b)) return FLOWMM_ERR_CUDA;
    MatchTcArgs a;
    a.cand_count = g.cand_count; a.cand_slot = g.cand_slot; a.evicted = evicted; a.strategy = strategy;
    a.cand_scale = g.cand_scale; a.evi_mod = g.evi_mod; a.tile_mod = g.tile_mod;
    a.match = match; a.match_sim = match_sim; a.status = at<int>(ws, y.status);
    a.Hkv = p.n_kv_heads; a.L = p.seq_len; a.E = E; a.Ctot = y.c_tot; a.n_rt = y.n_et; a.n_items = UH * y.n_et;
    a.k = static_cast<const __nv_bfloat16 *>(k);
    a.k_unit = p.k_stride[0]; a.k_head = p.k_stride[1]; a.row_bytes = (uint32_t)(p.k_stride[2] * 2);
    a.by_nrt = make_fastdiv((uint32_t)y.n_et); a.by_hkv = make_fastdiv((uint32_t)p.n_kv_heads);
    if (cudaFuncSetAttribute(match_tc_kernel<tcs::Big>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)tcs::Big::kSmemBytes) != cudaSuccess)
        return FLOWMM_ERR_CUDA;
    const int grid = a.n_items < tc::sm_count() ? a.n_items : tc::sm_count();
    launch(match_tc_kernel<tcs::Big>, grid, kMtThreads, tcs::Big::kSmemBytes, st, cand_map, a);
    FLOWMM_LAUNCHED("match_tc");
    return FLOWMM_OK;
}

// tokmap != nullptr (only with the short-list tensor-core kernel): also write the tensor-core merge's table
flowmm_status run_match(const flowmm_params &p, const Layout &y, const void *k, const float *importance,
                        const uint8_t *mod, const int32_t *retained, const int32_t *evicted, const int32_t *strategy,
                        int32_t *match, float *match_sim, void *ws, cudaStream_t st, int2 *tokmap = nullptr,
                        bool prepared = false) {
    const int E = p.seq_len - p.n_keep;
    if (E == 0) return FLOWMM_OK;
    if (use_tc(p)) return run_match_tc(p, y, k, importance, mod, retained, evicted, strategy, match, match_sim, ws, st, tokmap, prepared);
    MatchArgs a;
    a.k = k; a.importance = importance; a.modality = mod; a.retained = retained; a.evicted = evicted;
    a.strategy = strategy; a.match = match; a.match_sim = match_sim;
    a.Hkv = p.n_kv_heads; a.D = p.head_dim; a.L = p.seq_len; a.B = p.n_keep; a.E = E;
    a.tau_eff = tau_effective(p);
    for (int i = 0; i < 3; ++i) a.ks[i] = p.k_stride[i];
    // A row per thread where all blocks of 16 rows get an SM: a block's products then take a quarter of the time, but every block goes through
    // all pivots' rows.  fp32, head_dim 64, us, by 64 rows and by 16: 4 heads of 400 rows and 150 pivots 18.0, 12.3; 1 of 1200 and 300 24.9, 19.0;
    // with 1 to 1.3 blocks per SM 2 heads of 1200 and 150 15.9, 16.9, 4 of 600 and 300 28.8, 26.8; with 2 8 of 600 and 150 16.0, 21.8.
    const int UH = p.n_units * p.n_kv_heads;
    const bool one_row = (int64_t)UH * ((E + 15) / 16) <= tc::sm_count();
    const dim3 grid(UH, one_row ? (E + 15) / 16 : (E + kTile - 1) / kTile);
    auto kernel = p.dtype == FLOWMM_BF16 ? (one_row ? match_simt<__nv_bfloat16, 1> : match_simt<__nv_bfloat16, 4>)
                                         : (one_row ? match_simt<float, 1> : match_simt<float, 4>);
    launch(kernel, grid, kSimtThreads, 0, st, a);
    FLOWMM_LAUNCHED("match_simt");
    return FLOWMM_OK;
}

// Few slots per head: Eq. 5 as a product with the slot-by-token weight matrix on the tensor cores.
// (Below 65536 tokens a slot's fixed-point weight sum cannot overflow.)
bool merge_is_tc(const flowmm_params &p) {
    return p.seq_len > p.n_keep && p.dtype == FLOWMM_BF16 && p.head_dim == 128 && p.n_keep <= mtc::kMaxSlots &&
           p.seq_len < 65536 && p.path != FLOWMM_PATH_SIMT;
}

// map_ready: the (slot, weight) table of the tensor-core merge has been written already (by the matching kernel)
flowmm_status run_merge(const flowmm_params &p, const Layout &y, const void *k, const void *v,
                        const int32_t *retained, const int32_t *evicted, const int32_t *match, const float *match_sim,
                        void *k_out, void *v_out, void *ws, cudaStream_t st, bool map_ready = false) {
    const int E = p.seq_len - p.n_keep, UH = p.n_units * p.n_kv_heads;
    MergeArgs m;
    m.k = k; m.v = v; m.k_out = k_out; m.v_out = v_out; m.retained = retained;
    m.rows = nullptr; m.row_count = nullptr; m.first_slot = nullptr; m.pieces = nullptr; m.part_off = nullptr;
    m.partial = at<float>(ws, y.partial); m.ticket = nullptr; m.slot_done = nullptr;
    m.Hkv = p.n_kv_heads; m.D = p.head_dim; m.L = p.seq_len; m.B = p.n_keep; m.E = E;
    m.max_parts = y.max_parts; m.win = y.merge_win; m.n_win = y.n_win;
    for (int i = 0; i < 3; ++i) {
        m.ks[i] = p.k_stride[i]; m.vs[i] = p.v_stride[i]; m.kos[i] = p.ko_stride[i]; m.vos[i] = p.vo_stride[i];
    }
    // few slots per head: Eq. 5 as a product with the slot-by-token weight matrix on the tensor cores
    if (merge_is_tc(p)) {
        mtc::MapArgs ma;
        ma.retained = retained; ma.evicted = evicted; ma.match = match; ma.match_sim = match_sim;
        ma.tokmap = at<int2>(ws, y.tokmap); ma.L = p.seq_len; ma.B = p.n_keep; ma.E = E; ma.merge_mode = p.merge_mode;
        const int longest = E > p.n_keep ? E : p.n_keep;
        if (!map_ready) {
            launch(mtc::merge_map_kernel, dim3(UH, (longest + 255) / 256), 256, 0, st, ma);
            FLOWMM_LAUNCHED("merge_map");
        }
        CUtensorMap kmap, vmap;
        const uint64_t dims[4] = {128, (uint64_t)p.seq_len, (uint64_t)p.n_kv_heads, (uint64_t)p.n_units};
        const uint64_t ksb[3] = {(uint64_t)p.k_stride[2] * 2, (uint64_t)p.k_stride[1] * 2, (uint64_t)p.k_stride[0] * 2};
        const uint64_t vsb[3] = {(uint64_t)p.v_stride[2] * 2, (uint64_t)p.v_stride[1] * 2, (uint64_t)p.v_stride[0] * 2};
        const uint32_t box[4] = {64, mtc::kTile, 1, 1};
        if (!tc::make_bf16_map(&kmap, k, 4, dims, ksb, box) || !tc::make_bf16_map(&vmap, v, 4, dims, vsb, box))
            return FLOWMM_ERR_CUDA;
        mtc::Args a;
        a.tokmap = ma.tokmap; a.k_out = k_out; a.v_out = v_out; a.status = at<int>(ws, y.merge_status);
        a.Hkv = p.n_kv_heads; a.L = p.seq_len; a.B = p.n_keep; a.n_stages = p.n_keep <= 128 ? mtc::kMaxStages : 3;
        // few heads: K and V of a head on an SM each
        a.per_item = 2 * UH <= tc::sm_count() ? 1 : 2;
        a.n_items = a.per_item == 1 ? 2 * UH : UH;
        for (int i = 0; i < 3; ++i) { a.kos[i] = p.ko_stride[i]; a.vos[i] = p.vo_stride[i]; }
        const uint32_t smem = mtc::smem_bytes(p.n_keep, a.n_stages);
        if (!allow_smem(mtc::merge_tc_kernel)) return FLOWMM_ERR_CUDA;
        // ... and, while SMs are left, the steps of such an item on two or four (three steps each, or adding the parts up costs
        // what the split saves: 5 steps of 32 heads took 12 instead of 10 us; clusters of eight with this much shared memory start late)
        const int steps = (p.seq_len + mtc::kTile - 1) / mtc::kTile;
        a.ctas = 1;
        while (a.per_item == 1 && a.ctas < 4 && 2 * a.ctas * a.n_items <= tc::sm_count() && steps >= 6 * a.ctas) a.ctas *= 2;
        const int grid = a.ctas > 1 ? a.n_items * a.ctas : a.n_items < tc::sm_count() ? a.n_items : tc::sm_count();
        launch_cluster(dim3(a.ctas), mtc::merge_tc_kernel, grid, mtc::kThreads, smem, st, kmap, vmap, a);
        FLOWMM_LAUNCHED("merge_tc");
        return FLOWMM_OK;
    }
    // Short lists: straight from the matches.  Every block of slots reads its head's whole list, where the sorted way is two launches,
    // the first of them a block per head that walks all of the head's slots, and streams.  Up to 256 members the number of heads
    // decides, as that block's time grows with the slots of a head and the short way's with the slots of all heads; the second
    // launch counts while both are small.  Time of the short way over the sorted one, members spread evenly or 15 % of them in one slot,
    // 100 to 256 members, bf16 of 64 and 128 and fp32: 2 heads 0.09 to 0.14 at any number of slots, 8 heads 0.30 to 0.58, 24 heads
    // 0.70 to 0.95, 32 heads 0.72 to 1.04 up to 8000 blocks and 0.79 to 1.11 at 20 000 and 60 000, 40 heads 0.74 to 1.20 and 0.90 to
    // 1.27, 48 heads 0.85 to 1.23 and 1.06 to 1.56, 96 heads 0.97 to 1.24 at 3600 blocks and 0.99 to 1.58 beyond, 160 heads 1.03 to 1.39
    // and 1.15 to 1.84.  For up to 1000 members (500 0.6 to 1.6, 1000 1.0 to 2.3 with 15 % in one slot) 0.4 to 0.9 up to 2048 blocks.
    const int64_t slot_blocks = (int64_t)UH * ((p.n_keep + 7) / 8);
    // a slot per warp while the blocks fit the SMs together, else four, which share the block's copy of the list
    const int per = slot_blocks <= 4 * tc::sm_count() ? 1 : 4, grid_y = (p.n_keep + 8 * per - 1) / (8 * per);
    // (more slots than a grid has room for: the persistent kernels below take any number)
    if (E > 0 && grid_y <= 65535 && (E <= 256 ? UH <= 32 || slot_blocks <= 3600 : E <= kShortList && slot_blocks <= 2048)) {
        const dim3 grid(UH, grid_y);
        auto kernel = p.dtype == FLOWMM_BF16 ? (per == 1 ? merge_short_kernel<__nv_bfloat16, 1> : merge_short_kernel<__nv_bfloat16, 4>)
                                             : (per == 1 ? merge_short_kernel<float, 1> : merge_short_kernel<float, 4>);
        launch(kernel, grid, 256, 0, st, m, match, evicted, match_sim, p.merge_mode);
        FLOWMM_LAUNCHED("merge_short");
        return FLOWMM_OK;
    }
    if (E > 0) {
        CsrArgs c;
        c.match = match; c.evicted = evicted; c.match_sim = match_sim;
        c.sort_a = at<int>(ws, y.sort_a); c.sort_b = at<int>(ws, y.sort_b);
        c.retained = retained; c.rows = at<int2>(ws, y.rows); c.row_count = at<int2>(ws, y.row_count);
        c.off = at<int>(ws, y.off); c.first_slot = at<int>(ws, y.first_slot); c.part_off = at<int>(ws, y.part_off);
        c.pieces = at<int4>(ws, y.pieces); c.ticket = at<unsigned>(ws, y.ticket); c.slot_done = at<int>(ws, y.slot_done);
        c.B = p.n_keep; c.E = E; c.n_pass = y.csr_passes; c.max_parts = y.max_parts; c.merge_mode = p.merge_mode;
        c.win = y.merge_win; c.n_win = y.n_win;
        // Warps per head by the length of its list: 8 walk up to 4096 positions in 16 steps each, which ends before 32 warps
        // are through their barriers.  Sorted in shared memory when positions and counters fit, else through global memory.
        const bool long_list = E > 4096;
        int n_bits = 1;
        while ((p.n_keep >> n_bits) != 0) ++n_bits;
        // Few heads: a head's list is shared among 2, 4 or 8 CTAs, at least 1024 positions each, as long as every CTA has an
        // SM (with four per SM 128 heads of 33 792 tokens took 89 instead of 68 us: the scattered writes then set the pace) and
        // the counters fit it (16 heads of 33 000 positions, 3000 slots: 130 us by a CTA each, 35 by four; 5400 slots 168 and 43;
        // 74 heads by two 131 and 59, 170 and 65).  Counters of which an SM holds one set only leave clusters of four and eight
        // waiting for a place when they need nearly all SMs: 16 heads of 9000 by eight 28 us, by four 22, 37 heads by four 32, by
        // two 28.
        const size_t smem = csr_cluster_smem(p.n_keep);
        const int sms = tc::sm_count(), room = smem <= 112 * 1024 ? sms : sms * 5 / 6;
        int ctas = 8;
        while (ctas > 1 && (ctas * UH > (ctas > 2 ? room : sms) || E < 1024 * ctas)) ctas >>= 1;
        const size_t csr_smem = csr_count_smem(E, p.n_keep, long_list ? 32 : 8);
        if (ctas > 1 && E < 65536 && smem <= 224 * 1024) {
            if (!allow_smem(build_csr_cluster_kernel, 1024)) return FLOWMM_ERR_CUDA;
            launch_cluster(dim3(ctas), build_csr_cluster_kernel, UH * ctas, 32 * kCsrClusterWarps, smem, st, c, n_bits, ctas);
        } else if (E < 65536 && csr_smem <= 224 * 1024) {
            auto kernel = long_list ? build_csr_count_kernel<32> : build_csr_count_kernel<8>;
            if (!allow_smem(kernel, 1024)) return FLOWMM_ERR_CUDA;
            launch(kernel, UH, long_list ? 1024 : 256, csr_smem, st, c, n_bits);
        } else if (!long_list) launch(build_csr_kernel<8>, UH, 256, 0, st, c);
        else launch(build_csr_kernel<32>, UH, 1024, 0, st, c);
        FLOWMM_LAUNCHED("build_csr");
        m.rows = c.rows; m.row_count = c.row_count; m.first_slot = c.first_slot; m.pieces = c.pieces;
        m.part_off = c.part_off; m.ticket = c.ticket; m.slot_done = c.slot_done;
    }
    const int64_t items = (int64_t)UH * y.n_win;
    if ((int64_t)UH * p.seq_len < kManyRows) m.ticket = nullptr;
    if ((int64_t)UH * (E == 0 ? p.n_keep : (int64_t)p.n_keep + E / kPiece + 1) > 0xFFFF0000ll) return FLOWMM_ERR_SHAPE;   // (window numbers fit 32 bits long before)
    const int bytes = p.head_dim * (p.dtype == FLOWMM_BF16 ? 2 : 4) / 16;     // of a row per lane
    auto kernel = p.dtype == FLOWMM_BF16 ? (bytes == 16 ? mrow::merge_rows_kernel<__nv_bfloat16, 16> : mrow::merge_rows_kernel<__nv_bfloat16, 8>)
                                         : (bytes == 16 ? mrow::merge_rows_kernel<float, 16> : mrow::merge_rows_kernel<float, 32>);
    const size_t smem = mrow::kWarps * mrow::warp_bytes(bytes);
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return FLOWMM_ERR_CUDA;
    // Few windows: the pieces of long slots are items of their own behind them, on warps that would be idle (one head of 33 792
    // tokens 105 -> 99 us for the call); else they are spread over the windows, as most of a head's possible pieces are none (8 such
    // heads 237 us, as items of their own 245).
    const int64_t most = 3 * tc::sm_count(), apart = E > 0 && items + (int64_t)UH * y.max_parts <= 2 * mrow::kWarps * most ? (int64_t)UH * y.max_parts : 0;
    const int64_t blocks = (items + apart + mrow::kWarps - 1) / mrow::kWarps;
    launch(kernel, (int)(blocks < most ? blocks : most), mrow::kThreads, smem, st, m, (unsigned)items, (unsigned)apart, at<int>(ws, y.merge_status),
           make_fastdiv((uint32_t)y.n_win), make_fastdiv((uint32_t)UH), make_fastdiv((uint32_t)p.n_kv_heads));
    FLOWMM_LAUNCHED("merge_rows");
    return FLOWMM_OK;
}

// Whether the matching and the merge of a call go into one launch (match_merge_tc.cuh): heads that fill the GPU, few slots (see there).
// Up to a head per SM the line is half the SMs, whatever the length: K from memory twice costs the two launches as much as its heads' steps
// in a row cost the one.  The whole call, us, by two and by one, 64 slots: 76 heads of 300 tokens 24.2, 22.1, of 1280 46.8, 44.4, of 2000 57.6,
// 58.1, of 4000 89.7, 88.1, of 12 000 229, 212; 112 of 640 29.8, 27.2, of 2000 68.8, 66.0, of 12 000 309, 264; 144 of 4000 148, 130; but 72 of
// 640 25.9, 25.4, of 2000 49.5, 55.8, of 4000 79.9, 85.3, of 12 000 213, 207, and 48 of 640 24.8, 24.6, of 4000 63.6, 76.7.
// With several heads to an SM up to three steps a head are too few to hide its ends (1024 heads of 300 tokens 81.5 us by two launches, 82.9
// by one; of 384 the same), and a second round of few heads leaves SMs without any, where the matching alone spreads tiles (160 heads of
// 1200 tokens 85.0, 85.6; 256 of 640 42.9, 39.7).
bool use_match_merge(const flowmm_params &p) {
    const int UH = p.n_units * p.n_kv_heads, sms = tc::sm_count();
    if (!use_tc(p) || !merge_is_tc(p) || p.n_keep > mmt::kMaxSlots) return false;
    if (UH <= sms) return 2 * UH > sms;
    return p.seq_len > 3 * mmt::kTile && 5 * UH >= 6 * sms;
}

// Matching and merge behind a selection that has laid out the candidates.  match, match_sim: nullptr where nobody asks for them.
flowmm_status run_match_merge(const flowmm_params &p, const Layout &y, const void *k, const void *v, const uint8_t *mod,
                              const int32_t *strategy, int32_t *match, float *match_sim, void *k_out, void *v_out, void *ws, cudaStream_t st) {
    const int UH = p.n_units * p.n_kv_heads;
    CUtensorMap kmap, vmap, cand_map;
    const uint64_t dims[4] = {128, (uint64_t)p.seq_len, (uint64_t)p.n_kv_heads, (uint64_t)p.n_units};
    const uint64_t ksb[3] = {(uint64_t)p.k_stride[2] * 2, (uint64_t)p.k_stride[1] * 2, (uint64_t)p.k_stride[0] * 2};
    const uint64_t vsb[3] = {(uint64_t)p.v_stride[2] * 2, (uint64_t)p.v_stride[1] * 2, (uint64_t)p.v_stride[0] * 2};
    const uint64_t cd[4] = {128, (uint64_t)y.c_tot, (uint64_t)UH, 1};
    const uint64_t cs[3] = {256, (uint64_t)y.c_tot * 256, (uint64_t)y.c_tot * 256 * (uint64_t)UH};
    const uint32_t box[4] = {64, mmt::kTile, 1, 1}, box_c[4] = {64, (uint32_t)y.c_tot, 1, 1};
    if (!tc::make_bf16_map(&kmap, k, 4, dims, ksb, box) || !tc::make_bf16_map(&vmap, v, 4, dims, vsb, box) ||
        !tc::make_bf16_map(&cand_map, at<__nv_bfloat16>(ws, y.cand_k), 4, cd, cs, box_c))
        return FLOWMM_ERR_CUDA;
    mmt::Args a;
    a.cand_count = at<int>(ws, y.cand_count); a.cand_slot = at<int>(ws, y.cand_slot); a.cand_scale = at<float>(ws, y.cand_scale);
    a.rank = at<int>(ws, y.rank); a.strategy = strategy; a.modality = mod; a.match = match; a.match_sim = match_sim;
    a.k_out = k_out; a.v_out = v_out; a.status = at<int>(ws, y.status);
    a.Hkv = p.n_kv_heads; a.L = p.seq_len; a.E = p.seq_len - p.n_keep; a.B = p.n_keep; a.Ctot = y.c_tot; a.merge_mode = p.merge_mode;
    a.n_items = UH; a.at = mmt::smem_plan(p.n_keep, y.c_tot);
    for (int i = 0; i < 3; ++i) { a.kos[i] = p.ko_stride[i]; a.vos[i] = p.vo_stride[i]; }
    if (!allow_smem(mmt::match_merge_tc_kernel)) return FLOWMM_ERR_CUDA;
    launch(mmt::match_merge_tc_kernel, std::min(UH, tc::sm_count()), mmt::kThreads, a.at.total, st, kmap, vmap, cand_map, a);
    FLOWMM_LAUNCHED("match_merge_tc");
    return FLOWMM_OK;
}

}  // namespace

extern "C" {

flowmm_status flowmm_workspace_bytes(const flowmm_params *p, size_t *bytes) {
    if (!bytes) return FLOWMM_ERR_NULL;
    FLOWMM_TRY(validate(p));
    *bytes = make_layout(*p).total;
    return FLOWMM_OK;
}

flowmm_status flowmm_score(const flowmm_params *p, const void *q_win, const void *k, const uint8_t *modality,
                           float *importance, float *cross_mass, void *ws, size_t ws_bytes, void *cuda_stream) {
    profile_begin(static_cast<cudaStream_t>(cuda_stream));
    FLOWMM_TRY(validate(p));
    if (!q_win || !k || !modality || !importance || !cross_mass) return FLOWMM_ERR_NULL;
    if (!aligned16(q_win) || !aligned16(k) || !strides_ok(p->q_stride, p->head_dim) ||
        !strides_ok(p->k_stride, p->head_dim))
        return FLOWMM_ERR_ALIGN;
    Layout y;
    FLOWMM_TRY(check_ws(p, ws, ws_bytes, y));
    FLOWMM_TRY(check_device());
    return run_score(*p, y, q_win, k, modality, importance, cross_mass, ws, static_cast<cudaStream_t>(cuda_stream));
}

flowmm_status flowmm_layer_flow(const flowmm_params *p, const float *cross_mass, float *rho, int32_t *strategy,
                                void *cuda_stream) {
    profile_begin(static_cast<cudaStream_t>(cuda_stream));
    FLOWMM_TRY(validate(p));
    if (!cross_mass || !rho || !strategy) return FLOWMM_ERR_NULL;
    FLOWMM_TRY(check_device());
    return run_layer_flow(*p, cross_mass, rho, strategy, static_cast<cudaStream_t>(cuda_stream));
}

flowmm_status flowmm_select(const flowmm_params *p, const float *importance, int32_t *retained_idx,
                            int32_t *evicted_idx, void *ws, size_t ws_bytes, void *cuda_stream) {
    profile_begin(static_cast<cudaStream_t>(cuda_stream));
    FLOWMM_TRY(validate(p));
    if (!importance || !retained_idx || (!evicted_idx && p->n_keep < p->seq_len)) return FLOWMM_ERR_NULL;
    Layout y;
    FLOWMM_TRY(check_ws(p, ws, ws_bytes, y));
    FLOWMM_TRY(check_device());
    return run_select(*p, importance, retained_idx, evicted_idx, static_cast<cudaStream_t>(cuda_stream));
}

flowmm_status flowmm_match(const flowmm_params *p, const void *k, const float *importance, const uint8_t *modality,
                           const int32_t *retained_idx, const int32_t *evicted_idx, const int32_t *strategy,
                           int32_t *match, float *match_sim, void *ws, size_t ws_bytes, void *cuda_stream) {
    profile_begin(static_cast<cudaStream_t>(cuda_stream));
    FLOWMM_TRY(validate(p));
    const bool has_e = p->n_keep < p->seq_len;
    if (!k || !importance || !modality || !retained_idx || !strategy) return FLOWMM_ERR_NULL;
    if (has_e && (!evicted_idx || !match || !match_sim)) return FLOWMM_ERR_NULL;
    if (!aligned16(k) || !strides_ok(p->k_stride, p->head_dim)) return FLOWMM_ERR_ALIGN;
    Layout y;
    FLOWMM_TRY(check_ws(p, ws, ws_bytes, y));
    FLOWMM_TRY(check_device());
    FLOWMM_DEBUG_LISTS(*p, retained_idx, evicted_idx, nullptr, at<int>(ws, y.status), static_cast<cudaStream_t>(cuda_stream));
    return run_match(*p, y, k, importance, modality, retained_idx, evicted_idx, strategy, match, match_sim, ws,
                     static_cast<cudaStream_t>(cuda_stream));
}

flowmm_status flowmm_merge(const flowmm_params *p, const void *k, const void *v, const int32_t *retained_idx,
                           const int32_t *evicted_idx, const int32_t *match, const float *match_sim, void *k_out,
                           void *v_out, void *ws, size_t ws_bytes, void *cuda_stream) {
    profile_begin(static_cast<cudaStream_t>(cuda_stream));
    FLOWMM_TRY(validate(p));
    const bool has_e = p->n_keep < p->seq_len;
    if (!k || !v || !retained_idx || !k_out || !v_out) return FLOWMM_ERR_NULL;
    if (has_e && (!evicted_idx || !match || !match_sim)) return FLOWMM_ERR_NULL;
    if (!aligned16(k) || !aligned16(v) || !aligned16(k_out) || !aligned16(v_out) ||
        !strides_ok(p->k_stride, p->head_dim) || !strides_ok(p->v_stride, p->head_dim) ||
        !strides_ok(p->ko_stride, p->head_dim) || !strides_ok(p->vo_stride, p->head_dim))
        return FLOWMM_ERR_ALIGN;
    Layout y;
    FLOWMM_TRY(check_ws(p, ws, ws_bytes, y));
    FLOWMM_TRY(check_device());
    FLOWMM_DEBUG_LISTS(*p, retained_idx, evicted_idx, match, at<int>(ws, y.status), static_cast<cudaStream_t>(cuda_stream));
    return run_merge(*p, y, k, v, retained_idx, evicted_idx, match, match_sim, k_out, v_out, ws,
                     static_cast<cudaStream_t>(cuda_stream));
}

flowmm_status flowmm_compress_layer(const flowmm_params *p, const void *q_win, const void *k, const void *v,
                                    const uint8_t *modality, void *k_out, void *v_out, float *importance, float *rho,
                                    int32_t *strategy, int32_t *retained_idx, int32_t *evicted_idx, int32_t *match,
                                    float *match_sim, void *ws, size_t ws_bytes, void *cuda_stream) {
    profile_begin(static_cast<cudaStream_t>(cuda_stream));
    FLOWMM_TRY(validate(p));
    if (!q_win || !k || !v || !modality || !k_out || !v_out) return FLOWMM_ERR_NULL;
    if (!aligned16(q_win) || !aligned16(k) || !aligned16(v) || !aligned16(k_out) || !aligned16(v_out) ||
        !strides_ok(p->q_stride, p->head_dim) || !strides_ok(p->k_stride, p->head_dim) ||
        !strides_ok(p->v_stride, p->head_dim) || !strides_ok(p->ko_stride, p->head_dim) ||
        !strides_ok(p->vo_stride, p->head_dim))
        return FLOWMM_ERR_ALIGN;
    Layout y;
    FLOWMM_TRY(check_ws(p, ws, ws_bytes, y));
    FLOWMM_TRY(check_device());
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (!importance) importance = at<float>(ws, y.importance);
    if (!rho) rho = at<float>(ws, y.rho);
    if (!strategy) strategy = at<int32_t>(ws, y.strategy);
    if (!retained_idx) retained_idx = at<int32_t>(ws, y.retained);
    if (!evicted_idx) evicted_idx = at<int32_t>(ws, y.evicted);
    const bool matches_wanted = match || match_sim;
    if (!match) match = at<int32_t>(ws, y.match);
    if (!match_sim) match_sim = at<float>(ws, y.match_sim);
    float *cross_mass = at<float>(ws, y.cross_mass);
    int n_parts = 0;
    FLOWMM_TRY(run_score(*p, y, q_win, k, modality, importance, cross_mass, ws, st, &n_parts));
    // Eq. 6 and the theta rule ride along with the selection launch (which first adds up the partial masses, if any)
    // ... and so does the candidate layout of the tensor-core matching step
    const bool prep_in_select = p->seq_len > p->n_keep && use_tc(*p);
    const MatchPrepArgs prep = match_prep_args(*p, y, k, importance, modality, retained_idx, evicted_idx, ws);
    SelectFlow flow = {};
    flow.cross_part = n_parts > 0 ? at<float>(ws, y.cross_part) : nullptr; flow.n_parts = n_parts; flow.cross_mass = cross_mass;
    flow.rho = rho; flow.strategy = strategy; flow.n_units = p->n_units; flow.Hq = p->n_q_heads;
    flow.theta = p->theta; flow.flow_mode = p->flow_mode;
    FLOWMM_TRY(run_select(*p, importance, retained_idx, evicted_idx, st, &flow, prep_in_select ? &prep : nullptr));
    if (use_match_merge(*p))
        return run_match_merge(*p, y, k, v, modality, strategy, matches_wanted ? match : nullptr, match_sim, k_out, v_out, ws, st);
    // when both the short-list matching kernel and the tensor-core merge apply, the former writes the latter's table
    const bool map_in_match = p->seq_len > p->n_keep && use_tc(*p) && y.c_tot <= mst::kMaxCols && merge_is_tc(*p);
    FLOWMM_TRY(run_match(*p, y, k, importance, modality, retained_idx, evicted_idx, strategy, match, match_sim, ws, st,
                         map_in_match ? at<int2>(ws, y.tokmap) : nullptr, prep_in_select));
    FLOWMM_TRY(run_merge(*p, y, k, v, retained_idx, evicted_idx, match, match_sim, k_out, v_out, ws, st, map_in_match));
    return FLOWMM_OK;
}

flowmm_status flowmm_last_device_status(void *ws, void *cuda_stream) {
    if (!ws) return FLOWMM_ERR_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    int32_t word = 0;
    if (cudaMemcpyAsync(&word, ws, sizeof(word), cudaMemcpyDeviceToHost, st) != cudaSuccess) return FLOWMM_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return FLOWMM_ERR_CUDA;
    if (word != 0) {
        if (cudaMemsetAsync(ws, 0, sizeof(word), st) != cudaSuccess) return FLOWMM_ERR_CUDA;
        if (cudaStreamSynchronize(st) != cudaSuccess) return FLOWMM_ERR_CUDA;
    }
    return word >= 0 && word <= FLOWMM_ERR_INDEX ? static_cast<flowmm_status>(word) : FLOWMM_ERR_CUDA;
}

int32_t flowmm_last_launch_count(void) { return g_launches; }

int32_t flowmm_debug_build(void) {
#ifdef FLOWMM_DEBUG
    return 1;
#else
    return 0;
#endif
}

flowmm_status flowmm_profile_enable(int32_t on) {
    if (on && !g_prof.have_events) {
        for (int i = 0; i <= kMaxProfiled; ++i)
            if (cudaEventCreate(&g_prof.ev[i]) != cudaSuccess) return FLOWMM_ERR_CUDA;
        g_prof.have_events = true;
    }
    g_prof.on = on != 0;
    g_prof.n = 0;
    return FLOWMM_OK;
}

int32_t flowmm_profile_read(const char **names, float *ms, int32_t max_entries) {
    if (!g_prof.on || g_prof.n == 0) return 0;
    if (cudaEventSynchronize(g_prof.ev[g_prof.n]) != cudaSuccess) return -1;
    const int n = g_prof.n < max_entries ? g_prof.n : max_entries;
    for (int i = 0; i < n; ++i) {
        if (names) names[i] = g_prof.name[i];
        if (ms && cudaEventElapsedTime(&ms[i], g_prof.ev[i], g_prof.ev[i + 1]) != cudaSuccess) return -1;
    }
    return n;
}

const char *flowmm_status_string(flowmm_status s) {
    switch (s) {
        case FLOWMM_OK: return "ok";
        case FLOWMM_ERR_NULL: return "null pointer";
        case FLOWMM_ERR_SHAPE: return "inconsistent shape or parameter";
        case FLOWMM_ERR_BUDGET: return "retention budget out of range";
        case FLOWMM_ERR_DTYPE: return "unsupported dtype";
        case FLOWMM_ERR_WORKSPACE: return "workspace too small";
        case FLOWMM_ERR_ALIGN: return "pointer or stride not aligned";
        case FLOWMM_ERR_CUDA: return "CUDA error";
        case FLOWMM_ERR_TIMEOUT: return "device-side wait timed out";
        case FLOWMM_ERR_UNSUPPORTED_DEVICE: return "device is not compute capability 10.x";
        case FLOWMM_ERR_INDEX: return "index out of range (debug build)";
    }
    return "unknown status";
}

}  // extern "C"

// ---- full-prefill information flow ---------------------------------------------------------------
namespace {

constexpr int kFlowTile = 128;      // query rows per scoring call

// Query tile t of n: rows [lo, hi); the first tile takes the remainder so that all others are full.
void flow_tile(int L, int t, int &lo, int &hi) {
    const int rem = L % kFlowTile, n_full = L / kFlowTile;
    if (rem == 0) { lo = t * kFlowTile; hi = lo + kFlowTile; return; }
    if (t == 0) { lo = 0; hi = rem; return; }
    lo = rem + (t - 1) * kFlowTile; hi = lo + kFlowTile;
    (void)n_full;
}
int flow_tiles(int L) { return (L + kFlowTile - 1) / kFlowTile; }

// The scoring step's parameters for one query tile: the prompt cut after the tile's last row, the tile as window.
flowmm_params flow_tile_params(const flowmm_params &p, const int64_t qs[3], int lo, int hi) {
    flowmm_params t = p;
    t.seq_len = hi; t.window = hi - lo; t.n_keep = 1; t.keep_window = 0; t.tau = 0.f; t.tau_mode = FLOWMM_TAU_ABS;
    for (int i = 0; i < 3; ++i) t.q_stride[i] = qs[i];
    return t;
}

int flow_parts_tc(int L) { return (L + tcs::kItemRows - 1) / tcs::kItemRows * 8; }

struct FlowLayout { size_t std_bytes, mod, imp, parts, bits, total; };

// bf16 at head_dim 128: every query row in one launch (flow_tc.cuh).
flowmm_status run_flow_tc(const flowmm_params &p, const void *q, const int64_t q_stride[3], const void *k, const uint32_t *modbits,
                          int mod_words, float *parts, int *status, cudaStream_t st) {
    FlowTcArgs a = {};
    a.modbits = modbits; a.parts = parts; a.status = status;
    a.Hq = p.n_q_heads; a.Hkv = p.n_kv_heads; a.G = p.n_q_heads / p.n_kv_heads; a.L = p.seq_len;
    a.n_rp = (p.seq_len + tcs::kItemRows - 1) / tcs::kItemRows; a.n_heads = p.n_units * p.n_q_heads; a.mod_words = mod_words;
    a.n_items = a.n_heads * a.n_rp;
    const int sms = tc::sm_count(), grid = a.n_items < sms ? a.n_items : sms;
    a.by_grid = make_fastdiv((uint32_t)grid); a.n_rounds = (a.n_items + grid - 1) / grid;
    const float scale = p.softmax_scale != 0.f ? p.softmax_scale : 1.f / sqrtf((float)p.head_dim);
    a.scale_log2 = scale * kLog2e;
    // every block of rows reads its head's keys again: the keys of a group of heads take at most 48 MB of the 126 MB L2
    const int64_t head_bytes = (int64_t)p.seq_len * 256, fit = (48ll << 20) / head_bytes;
    const int n_uh = p.n_units * p.n_kv_heads, group = fit < 1 ? 1 : fit > n_uh ? n_uh : (int)fit;
    a.group_heads = group * a.G;
    a.by_group_items = make_fastdiv((uint32_t)(a.group_heads * a.n_rp)); a.by_group_heads = make_fastdiv((uint32_t)a.group_heads);
    a.by_last_heads = make_fastdiv((uint32_t)(n_uh % group ? n_uh % group * a.G : a.group_heads));
    a.by_g = make_fastdiv((uint32_t)a.G); a.by_hkv = make_fastdiv((uint32_t)p.n_kv_heads);
    CUtensorMap qa, k256;
    const uint64_t qd[4] = {128, (uint64_t)p.seq_len, (uint64_t)p.n_q_heads, (uint64_t)p.n_units};
    const uint64_t qs[3] = {(uint64_t)q_stride[2] * 2, (uint64_t)q_stride[1] * 2, (uint64_t)q_stride[0] * 2};
    const uint64_t kd[4] = {128, (uint64_t)p.seq_len, (uint64_t)p.n_kv_heads, (uint64_t)p.n_units};
    const uint64_t ks[3] = {(uint64_t)p.k_stride[2] * 2, (uint64_t)p.k_stride[1] * 2, (uint64_t)p.k_stride[0] * 2};
    const uint32_t bqa[4] = {64, tcs::kRows, 1, 1}, bk256[4] = {64, tcs::Big::kCols, 1, 1};
    if (!tc::make_bf16_map(&qa, q, 4, qd, qs, bqa) || !tc::make_bf16_map(&k256, k, 4, kd, ks, bk256)) return FLOWMM_ERR_CUDA;
    if (cudaFuncSetAttribute(flow_stats_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tcs::Big::kSmemBytes) != cudaSuccess)
        return FLOWMM_ERR_CUDA;
    launch(flow_stats_tc_kernel, grid, tcs::kThreads, tcs::Big::kSmemBytes, st, qa, k256, a);
    FLOWMM_LAUNCHED("flow_stats_tc");
    return FLOWMM_OK;
}

FlowLayout flow_layout(const flowmm_params &p, const int64_t qs[3]) {
    FlowLayout f = {};
    const int n = flow_tiles(p.seq_len);
    if (use_tc(p)) {
        f.std_bytes = 256;                                               // the status word
        f.parts = align256(f.std_bytes);
        f.bits = f.parts + align256((size_t)flow_parts_tc(p.seq_len) * p.n_units * p.n_q_heads * 4);
        f.total = f.bits + align256((size_t)p.n_units * ((p.seq_len + 31) / 32 + 8) * 4);
        return f;
    }
    for (int t = 0; t < n; ++t) {
        int lo, hi;
        flow_tile(p.seq_len, t, lo, hi);
        const size_t need = make_layout(flow_tile_params(p, qs, lo, hi)).total;
        if (need > f.std_bytes) f.std_bytes = need;
    }
    size_t o = align256(f.std_bytes);
    f.mod = o; o += align256((size_t)p.n_units * p.seq_len);
    f.imp = o; o += align256((size_t)p.n_units * p.n_kv_heads * p.seq_len * 4);
    f.parts = o; o += align256((size_t)n * p.n_units * p.n_q_heads * 4);
    f.total = o;
    return f;
}

flowmm_status validate_flow(const flowmm_params *p) {
    if (!p) return FLOWMM_ERR_NULL;
    flowmm_params t = *p;
    t.window = 1; t.n_keep = 1; t.keep_window = 0; t.tau = 0.f; t.tau_mode = FLOWMM_TAU_ABS;   // not used here
    return validate(&t);
}

}  // namespace

extern "C" flowmm_status flowmm_full_flow_workspace_bytes(const flowmm_params *p, size_t *bytes) {
    if (!bytes) return FLOWMM_ERR_NULL;
    FLOWMM_TRY(validate_flow(p));
    const int64_t dense[3] = {(int64_t)p->n_q_heads * p->seq_len * p->head_dim, (int64_t)p->seq_len * p->head_dim, p->head_dim};
    *bytes = flow_layout(*p, dense).total;
    return FLOWMM_OK;
}

extern "C" flowmm_status flowmm_full_flow(const flowmm_params *p, const void *q_full, const int64_t q_full_stride[3],
                                          const void *k, const uint8_t *modality, float *cross_mass, float *rho,
                                          int32_t *strategy, void *ws, size_t ws_bytes, void *cuda_stream) {
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    profile_begin(st);
    FLOWMM_TRY(validate_flow(p));
    if (!q_full || !q_full_stride || !k || !modality || !cross_mass || !strategy || !ws) return FLOWMM_ERR_NULL;
    if (!aligned16(q_full) || !aligned16(k) || !strides_ok(q_full_stride, p->head_dim) || !strides_ok(p->k_stride, p->head_dim) ||
        (reinterpret_cast<uintptr_t>(ws) & 255))
        return FLOWMM_ERR_ALIGN;
    const FlowLayout f = flow_layout(*p, q_full_stride);
    if (ws_bytes < f.total) return FLOWMM_ERR_WORKSPACE;
    FLOWMM_TRY(check_device());
    if (cudaMemsetAsync(ws, 0, 4, st) != cudaSuccess) return FLOWMM_ERR_CUDA;       // the status word
    int n_tiles = flow_tiles(p->seq_len);
    const int n = p->n_units * p->n_q_heads;
    float *parts = at<float>(ws, f.parts);
    if (use_tc(*p)) {
        const int mod_words = (p->seq_len + 31) / 32 + 8;              // + slack: whole 256-key tiles are indexed
        uint32_t *bits = at<uint32_t>(ws, f.bits);
        launch(pack_modality_kernel, dim3(p->n_units, (mod_words + 7) / 8), 256, 0, st, modality, p->seq_len, mod_words, bits);
        FLOWMM_LAUNCHED("pack_modality");
        FLOWMM_TRY(run_flow_tc(*p, q_full, q_full_stride, k, bits, mod_words, parts, static_cast<int *>(ws), st));
        n_tiles = flow_parts_tc(p->seq_len);
    } else {
        const size_t esize = p->dtype == FLOWMM_BF16 ? 2 : 4;
        uint8_t *mod = at<uint8_t>(ws, f.mod);
        float *imp = at<float>(ws, f.imp);
        for (int t = 0; t < n_tiles; ++t) {
            int lo, hi;
            flow_tile(p->seq_len, t, lo, hi);
            const flowmm_params tp = flow_tile_params(*p, q_full_stride, lo, hi);
            const Layout y = make_layout(tp);
            // the scoring kernels index the modality map with the cut prompt's length as the row pitch
            if (cudaMemcpy2DAsync(mod, (size_t)hi, modality, (size_t)p->seq_len, (size_t)hi, (size_t)p->n_units,
                                  cudaMemcpyDeviceToDevice, st) != cudaSuccess)
                return FLOWMM_ERR_CUDA;
            const char *q_tile = static_cast<const char *>(q_full) + (size_t)lo * (size_t)q_full_stride[2] * esize;
            FLOWMM_TRY(run_score(tp, y, q_tile, k, mod, imp, parts + (size_t)t * n, ws, st));
        }
    }
    launch(full_flow_reduce_kernel, p->n_units, 1024, 0, st, parts, n_tiles, n, p->n_q_heads, p->seq_len, p->theta, p->flow_mode,
                                                       cross_mass, rho, strategy);
    FLOWMM_LAUNCHED("full_flow_reduce");
    return FLOWMM_OK;
}

// ---- decode-step attention over a cache ---------------------------------------------------------
namespace {

flowmm_status validate_decode(const flowmm_decode_params *p) {
    if (!p) return FLOWMM_ERR_NULL;
    if (p->n_units < 1 || p->n_q_heads < 1 || p->n_kv_heads < 1 || p->n_keys < 1) return FLOWMM_ERR_SHAPE;
    if (p->n_q_heads % p->n_kv_heads != 0 || p->n_q_heads / p->n_kv_heads > 8) return FLOWMM_ERR_SHAPE;
    if (p->head_dim != 64 && p->head_dim != 128) return FLOWMM_ERR_SHAPE;
    if ((int64_t)p->n_units * p->n_kv_heads > kMaxHeadsPerCall) return FLOWMM_ERR_SHAPE;
    if (p->dtype != FLOWMM_F32 && p->dtype != FLOWMM_BF16) return FLOWMM_ERR_DTYPE;
    if (!(p->softmax_scale >= 0.f)) return FLOWMM_ERR_SHAPE;
    if (p->path != FLOWMM_PATH_AUTO && p->path != FLOWMM_PATH_SIMT) return FLOWMM_ERR_SHAPE;
    return FLOWMM_OK;
}

// How a call is cut into key ranges, and where its scratch lives:
// [status word, 256 bytes][partial records].
struct DecodePlan {
    bool tc;                 // tensor-core kernel (bf16, head_dim 128) or the SIMT one
    int n_split, per_split;  // ranges per (unit, KV head); keys (SIMT) or 128-key tiles (tensor core) per range
    size_t least;            // bytes of workspace below which the call is refused
};

constexpr size_t kDecodePartOff = 256;
constexpr int kMaxDecodeCluster = dtc::kMaxRanges;         // ranges of a head that are joined as one cluster (the portable cluster size)

// Partial records of the ranges of all heads: `fewest`, as many as the longest tensor-core ranges make, without which a call is refused, and
// `most`, that a workspace is asked to hold.  Both never fall when keys or heads are added, so that a workspace kept for the largest call serves
// the smaller ones.  Ranges that a cluster joins write none, so a plan needs room for more than eight ranges of a head alone: of these up to
// four per SM and one more per head (2560 heads of 1690 keys, 8 query heads each, 11 MB; eight records for every head were 85).  SIMT
// ranges, of 64 keys and more: four per SM in whole numbers per head.
struct DecodeRecords { int64_t fewest, most; };
DecodeRecords decode_records(bool tensor_cores, int uh, int keys) {
    constexpr int64_t few = 4 * kScoreCtas;
    if (!tensor_cores) return {0, std::min((int64_t)uh * ((keys + 63) / 64), few + uh - 1)};
    const int tiles = (keys + dtc::kTile - 1) / dtc::kTile;
    const int64_t fewest = (int64_t)uh * ((tiles + dtc::kMaxTiles - 1) / dtc::kMaxTiles);
    return {fewest, std::max(fewest, std::min((int64_t)uh * tiles, few + std::min<int64_t>(uh, few / kMaxDecodeCluster)))};
}
size_t decode_bytes(const flowmm_decode_params &p, int64_t records) {
    return kDecodePartOff + align256((size_t)records * (p.n_q_heads / p.n_kv_heads) * (p.head_dim + 2) * sizeof(float));
}

bool decode_use_tc(const flowmm_decode_params &p) { return p.dtype == FLOWMM_BF16 && p.head_dim == 128 && p.path != FLOWMM_PATH_SIMT; }

DecodePlan decode_plan(const flowmm_decode_params &p, size_t ws_bytes) {
    DecodePlan d;
    const int uh = p.n_units * p.n_kv_heads;
    d.tc = decode_use_tc(p);
    if (d.tc) {
        // Two CTAs share an SM.  Of the range lengths TMEM allows, the one whose call is the shortest by this account, in us: all tiles of K
        // and V at the memory's rate, or the one CTA's, 0.9 a tile, where that is longer; when the CTAs do not fit at once, 1 per further
        // round, and part of what the last ones take with the memory mostly idle; for joining the ranges 2 as a cluster, 3 as a launch of
        // its own.  Clusters find room for 0.88 of the CTAs (96 of three, 12 tiles each, ran two after the other: 47 us, by five of 7 tiles
        // 40).  Measured with every length on the 18 shapes the constants are from, 16 to 554 MB of 4 to 1024 heads: 1 % on average, 10 % at
        // most above the best length (4 and 18 % by rounds of CTAs times their tiles and a fixed cost each); on 31 others of 7 us and more, K
        // and V from memory, 2 and 13 % (9 and 54 %); one head alone of 24 306 keys 45 % (48 %).  Where 80 MB stay in L2 from the call before,
        // 56 heads of 2795 keys 12.2 us, 11.6 by rounds; from memory 16.4, 17.2.
        // (A smaller workspace than is asked for has room for fewer ranges.)
        const int tiles = (p.n_keys + dtc::kTile - 1) / dtc::kTile;
        const DecodeRecords records = decode_records(true, uh, p.n_keys);
        d.least = decode_bytes(p, records.fewest);
        const bool all_fit = ws_bytes >= decode_bytes(p, records.most);
        double best = 0.0;
        d.per_split = 0;
        for (int per = 1; per <= dtc::kMaxTiles && per <= tiles; ++per) {
            const int splits = (tiles + per - 1) / per;
            const bool cluster = splits > 1 && splits <= kMaxDecodeCluster;
            const int64_t n = (int64_t)uh * splits;
            if (splits > kMaxDecodeCluster && n != records.fewest && (n > records.most || (!all_fit && decode_bytes(p, n) > ws_bytes))) continue;
            const double slots = 2.0 * kScoreCtas * (cluster ? 0.88 : 1.0), ctas = (double)n, rounds = ctas / slots;
            const double tile_us = 0.00985, all = uh * (double)tiles * tile_us, lone = 0.9 * per;
            double cost = all > lone ? all : lone;
            if (rounds > 1.0) {
                const double last = ctas - floor(rounds) * slots, gap = lone + 3.0 - last * per * tile_us;
                cost = all + (last > 0.0 && gap > 0.0 ? gap * (cluster ? 0.5 : 0.1) : 0.0) + (rounds - 1.0);
            }
            cost += (splits == 1 ? 0.0 : cluster ? 2.0 : 3.0) + 0.15 * per;
            if (d.per_split == 0 || cost < best) { best = cost; d.per_split = per; }
        }
        d.n_split = (tiles + d.per_split - 1) / d.per_split;
    }
    if (!d.tc) {
        // enough CTAs for about four per SM, at least 64 keys each
        int want = (4 * kScoreCtas + uh - 1) / uh;
        const int max_split = (p.n_keys + 63) / 64;
        want = want < 1 ? 1 : (want > max_split ? max_split : want);
        d.per_split = (p.n_keys + want - 1) / want;
        d.n_split = (p.n_keys + d.per_split - 1) / d.per_split;
        d.least = decode_bytes(p, (int64_t)uh * d.n_split);
    }
    return d;
}

template <typename T, int D>
flowmm_status launch_decode(const DecodeArgs &a, int uh, int n_q, cudaStream_t st) {
    constexpr int groups = kDecThreads / (D / Elem<T>::kVec);
    const dim3 grid(uh, a.n_split);
    const int gp = a.G <= 1 ? 1 : a.G <= 2 ? 2 : a.G <= 4 ? 4 : 8;
    const size_t smem = (size_t)groups * gp * (D + 2) * sizeof(float);
    switch (gp) {
        case 1: launch(decode_partial_kernel<T, D, 1>, grid, kDecThreads, smem, st, a); break;
        case 2: launch(decode_partial_kernel<T, D, 2>, grid, kDecThreads, smem, st, a); break;
        case 4: launch(decode_partial_kernel<T, D, 4>, grid, kDecThreads, smem, st, a); break;
        default: launch(decode_partial_kernel<T, D, 8>, grid, kDecThreads, smem, st, a); break;
    }
    FLOWMM_LAUNCHED("decode_partial");
    launch(decode_combine_kernel<D>, n_q, kCombineParts * D, 0, st, a);
    FLOWMM_LAUNCHED("decode_combine");
    return FLOWMM_OK;
}

// Numbers of the calls that clear their own status word (status_word.cuh): consecutive calls differ, and none is a number
// that memory is likely to hold by itself (0, small integers).
uint32_t status_call_number() {
    static std::atomic<uint32_t> n{0};
    uint32_t call = 0;
    while (call == 0) call = (n.fetch_add(1, std::memory_order_relaxed) + 1) * 0x9E3779B1u;
    return call;
}

flowmm_status launch_decode_tc(const flowmm_decode_params &p, const DecodeArgs &a, int *status, int uh, cudaStream_t st) {
    CUtensorMap kmap, vmap;
    const uint64_t dims[4] = {128, (uint64_t)p.n_keys, (uint64_t)p.n_kv_heads, (uint64_t)p.n_units};
    const uint64_t ks[3] = {(uint64_t)p.k_stride[2] * 2, (uint64_t)p.k_stride[1] * 2, (uint64_t)p.k_stride[0] * 2};
    const uint64_t vs[3] = {(uint64_t)p.v_stride[2] * 2, (uint64_t)p.v_stride[1] * 2, (uint64_t)p.v_stride[0] * 2};
    const uint32_t box[4] = {64, dtc::kTile, 1, 1};
    if (!tc::make_bf16_map(&kmap, a.k, 4, dims, ks, box) || !tc::make_bf16_map(&vmap, a.v, 4, dims, vs, box))
        return FLOWMM_ERR_CUDA;
    // (function attributes belong to the current device: set on every call, like the other launchers)
    if (cudaFuncSetAttribute(dtc::decode_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)dtc::kSmemBytes) != cudaSuccess ||
        cudaFuncSetAttribute(dtc::decode_tc_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared) != cudaSuccess)
        return FLOWMM_ERR_CUDA;
    dtc::Args t;
    t.q = static_cast<const __nv_bfloat16 *>(a.q); t.part = a.part; t.out = a.out; t.status = status; t.call = status_call_number();
    t.Hq = a.Hq; t.Hkv = a.Hkv; t.G = a.G; t.N = a.N; t.n_split = a.n_split; t.tiles_per_split = a.keys_per_split;
    t.scale_log2 = a.scale_log2;
    t.clustered = a.n_split > 1 && a.n_split <= kMaxDecodeCluster;
    launch_cluster(dim3(1, t.clustered ? a.n_split : 1), dtc::decode_tc_kernel, dim3(uh, a.n_split), dtc::kThreads, dtc::kSmemBytes, st, kmap, vmap, t);
    FLOWMM_LAUNCHED("decode_tc");
    if (a.n_split <= kMaxDecodeCluster) return FLOWMM_OK;
    launch(decode_combine_kernel<128>, p.n_units * p.n_q_heads, kCombineParts * 128, 0, st, a);
    FLOWMM_LAUNCHED("decode_combine");
    return FLOWMM_OK;
}

}  // namespace

extern "C" flowmm_status flowmm_decode_workspace_bytes(const flowmm_decode_params *p, size_t *bytes) {
    if (!bytes) return FLOWMM_ERR_NULL;
    FLOWMM_TRY(validate_decode(p));
    *bytes = decode_bytes(*p, decode_records(decode_use_tc(*p), p->n_units * p->n_kv_heads, p->n_keys).most);
    return FLOWMM_OK;
}

extern "C" flowmm_status flowmm_decode_attention(const flowmm_decode_params *p, const void *q, const void *k,
                                                 const void *v, float *out, void *ws, size_t ws_bytes,
                                                 void *cuda_stream) {
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    profile_begin(st);
    FLOWMM_TRY(validate_decode(p));
    if (!q || !k || !v || !out || !ws) return FLOWMM_ERR_NULL;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !strides_ok(p->k_stride, p->head_dim) ||
        !strides_ok(p->v_stride, p->head_dim) || (reinterpret_cast<uintptr_t>(ws) & 255))
        return FLOWMM_ERR_ALIGN;
    const DecodePlan plan = decode_plan(*p, ws_bytes);
    if (ws_bytes < plan.least) return FLOWMM_ERR_WORKSPACE;
    FLOWMM_TRY(check_device());
    DecodeArgs a;
    a.status = static_cast<int *>(ws);                               // (cleared by the kernel)
    a.q = q; a.k = k; a.v = v; a.part = reinterpret_cast<float *>(static_cast<char *>(ws) + kDecodePartOff); a.out = out;
    a.Hq = p->n_q_heads; a.Hkv = p->n_kv_heads; a.G = p->n_q_heads / p->n_kv_heads; a.N = p->n_keys;
    a.n_split = plan.n_split; a.keys_per_split = plan.per_split;
    const float scale = p->softmax_scale != 0.f ? p->softmax_scale : 1.f / sqrtf((float)p->head_dim);
    a.scale_log2 = scale * kLog2e;
    for (int i = 0; i < 3; ++i) { a.ks[i] = p->k_stride[i]; a.vs[i] = p->v_stride[i]; }
    const int uh = p->n_units * p->n_kv_heads, n_q = p->n_units * p->n_q_heads;
    if (plan.tc) return launch_decode_tc(*p, a, static_cast<int *>(ws), uh, st);
    if (p->dtype == FLOWMM_BF16)
        return p->head_dim == 128 ? launch_decode<__nv_bfloat16, 128>(a, uh, n_q, st) : launch_decode<__nv_bfloat16, 64>(a, uh, n_q, st);
    return p->head_dim == 128 ? launch_decode<float, 128>(a, uh, n_q, st) : launch_decode<float, 64>(a, uh, n_q, st);
}

// ---- re-compression of a cache that grew during decoding ----------------------------------------
namespace {

// Every (unit, KV head) of the cache as a problem of its own: one KV head, its G query heads, its own row modalities.
// Needs the unit stride of every tensor to be heads x head stride (one stride then steps through units and heads).
bool per_head_params(const flowmm_params &p, flowmm_params &ph) {
    const int G = p.n_q_heads / p.n_kv_heads;
    if (p.q_stride[0] != (int64_t)p.n_q_heads * p.q_stride[1] || p.k_stride[0] != (int64_t)p.n_kv_heads * p.k_stride[1] ||
        p.v_stride[0] != (int64_t)p.n_kv_heads * p.v_stride[1] || p.ko_stride[0] != (int64_t)p.n_kv_heads * p.ko_stride[1] ||
        p.vo_stride[0] != (int64_t)p.n_kv_heads * p.vo_stride[1])
        return false;
    ph = p;
    ph.n_units = p.n_units * p.n_kv_heads; ph.n_q_heads = G; ph.n_kv_heads = 1;
    ph.q_stride[0] = (int64_t)G * p.q_stride[1];
    ph.k_stride[0] = p.k_stride[1]; ph.v_stride[0] = p.v_stride[1];
    ph.ko_stride[0] = p.ko_stride[1]; ph.vo_stride[0] = p.vo_stride[1];
    return true;
}

struct RecompressLayout { size_t strategy_h, total; };
RecompressLayout recompress_layout(const flowmm_params &ph) {
    RecompressLayout r;
    r.strategy_h = align256(make_layout(ph).total);
    r.total = r.strategy_h + align256((size_t)ph.n_units * 4);
    return r;
}

}  // namespace

extern "C" flowmm_status flowmm_recompress_workspace_bytes(const flowmm_params *p, size_t *bytes) {
    if (!bytes) return FLOWMM_ERR_NULL;
    FLOWMM_TRY(validate(p));
    flowmm_params ph;
    if (!per_head_params(*p, ph)) return FLOWMM_ERR_ALIGN;
    FLOWMM_TRY(validate(&ph));
    *bytes = recompress_layout(ph).total;
    return FLOWMM_OK;
}

extern "C" flowmm_status flowmm_recompress(const flowmm_params *p, const void *q_win, const void *k_cache,
                                           const void *v_cache, const uint8_t *row_modality, void *k_out, void *v_out,
                                           uint8_t *row_modality_out, float *importance, float *rho, int32_t *strategy,
                                           int32_t *retained_idx, int32_t *evicted_idx, int32_t *match, float *match_sim,
                                           void *ws, size_t ws_bytes, void *cuda_stream) {
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    profile_begin(st);
    FLOWMM_TRY(validate(p));
    if (!q_win || !k_cache || !v_cache || !row_modality || !k_out || !v_out || !row_modality_out) return FLOWMM_ERR_NULL;
    if (!aligned16(q_win) || !aligned16(k_cache) || !aligned16(v_cache) || !aligned16(k_out) || !aligned16(v_out) ||
        !strides_ok(p->q_stride, p->head_dim) || !strides_ok(p->k_stride, p->head_dim) ||
        !strides_ok(p->v_stride, p->head_dim) || !strides_ok(p->ko_stride, p->head_dim) ||
        !strides_ok(p->vo_stride, p->head_dim))
        return FLOWMM_ERR_ALIGN;
    flowmm_params ph;
    if (!per_head_params(*p, ph)) return FLOWMM_ERR_ALIGN;
    FLOWMM_TRY(validate(&ph));
    if (!ws) return FLOWMM_ERR_NULL;
    if (reinterpret_cast<uintptr_t>(ws) & 255) return FLOWMM_ERR_ALIGN;
    const Layout y = make_layout(ph);
    const RecompressLayout r = recompress_layout(ph);
    if (ws_bytes < r.total) return FLOWMM_ERR_WORKSPACE;
    FLOWMM_TRY(check_device());
    if (!importance) importance = at<float>(ws, y.importance);
    if (!rho) rho = at<float>(ws, y.rho);
    if (!strategy) strategy = at<int32_t>(ws, y.strategy);
    if (!retained_idx) retained_idx = at<int32_t>(ws, y.retained);
    if (!evicted_idx) evicted_idx = at<int32_t>(ws, y.evicted);
    const bool matches_wanted = match || match_sim;
    if (!match) match = at<int32_t>(ws, y.match);
    if (!match_sim) match_sim = at<float>(ws, y.match_sim);
    float *cross_mass = at<float>(ws, y.cross_mass);             // [U * Hkv, G] = [U, Hq]
    int32_t *strategy_h = at<int32_t>(ws, r.strategy_h);
    // scoring per (unit, KV head) against that head's own row modalities; Eq. 6 over all query heads of the layer rides along
    // with the selection, which hands the unit's strategy to each of its heads and notes the kept rows' modalities
    int n_parts = 0;
    FLOWMM_TRY(run_score(ph, y, q_win, k_cache, row_modality, importance, cross_mass, ws, st, &n_parts));
    const bool prep_in_select = p->seq_len > p->n_keep && use_tc(ph);
    const MatchPrepArgs prep = match_prep_args(ph, y, k_cache, importance, row_modality, retained_idx, evicted_idx, ws);
    SelectFlow flow = {};
    flow.cross_part = n_parts > 0 ? at<float>(ws, y.cross_part) : nullptr; flow.n_parts = n_parts; flow.cross_mass = cross_mass;
    flow.rho = rho; flow.strategy = strategy; flow.strategy_h = strategy_h; flow.n_units = p->n_units; flow.Hq = p->n_q_heads;
    flow.n_rep = p->n_kv_heads; flow.theta = p->theta; flow.flow_mode = p->flow_mode;
    FLOWMM_TRY(run_select(ph, importance, retained_idx, evicted_idx, st, &flow, prep_in_select ? &prep : nullptr, row_modality,
                          row_modality_out));
    if (use_match_merge(ph))
        return run_match_merge(ph, y, k_cache, v_cache, row_modality, strategy_h, matches_wanted ? match : nullptr, match_sim, k_out, v_out,
                               ws, st);
    const bool map_in_match = prep_in_select && y.c_tot <= mst::kMaxCols && merge_is_tc(ph);
    FLOWMM_TRY(run_match(ph, y, k_cache, importance, row_modality, retained_idx, evicted_idx, strategy_h, match, match_sim, ws, st,
                         map_in_match ? at<int2>(ws, y.tokmap) : nullptr, prep_in_select));
    return run_merge(ph, y, k_cache, v_cache, retained_idx, evicted_idx, match, match_sim, k_out, v_out, ws, st, map_in_match);
}

// ---- bounded-wait self-test ----------------------------------------------------------------------
namespace {
// One CTA waits on an mbarrier phase that nothing completes, with the same bounded waits the
// tensor-core kernels use, the first warp lane by lane and the second as a warp: after the limit the
// first waiter of each records FLOWMM_ERR_TIMEOUT, raises its warp's abort flag, and every thread returns.
__global__ void wait_timeout_selftest_kernel(int *status) {
    __shared__ __align__(8) unsigned long long bar;
    __shared__ int abort_flag[2];
    predecessor_done();
    if (threadIdx.x == 0) {
        abort_flag[0] = abort_flag[1] = 0;
        tc::mbar_init(tc::smem_u32(&bar), 1);
        tc::mbar_init_fence();
    }
    __syncthreads();
    if (threadIdx.x < 32) tc::mbar_wait(tc::smem_u32(&bar), 0, &abort_flag[0], status);
    else tc::mbar_wait_warp(tc::smem_u32(&bar), 0, &abort_flag[1], status);
}
}  // namespace

extern "C" flowmm_status flowmm_selftest_wait_timeout(void *ws, void *cuda_stream) {
    profile_begin(static_cast<cudaStream_t>(cuda_stream));
    if (!ws) return FLOWMM_ERR_NULL;
    FLOWMM_TRY(check_device());
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    launch(wait_timeout_selftest_kernel, 1, 64, 0, st, static_cast<int *>(ws));
    FLOWMM_LAUNCHED("wait_timeout_selftest");
    return FLOWMM_OK;
}

// ---- merge without caller scratch --------------------------------------------------------------
// Scratch of flowmm_merge_static: lives in the library image, one copy per GPU that loads it.
// (A little more than the size that callers know: merge_static_need.)
constexpr size_t kStaticScratch = FLOWMM_MERGE_STATIC_BYTES + FLOWMM_MERGE_STATIC_BYTES / 32;
static __device__ __align__(256) unsigned char g_merge_static_scratch[kStaticScratch];

namespace {

constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
void *g_static_ptr[kMaxDevices] = {};          // device address of the array, per device ordinal

// The array's name is only a handle in host code; the address a kernel can use comes from the
// runtime, once per device, with that device current.
flowmm_status merge_static_base(void **base) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return FLOWMM_ERR_CUDA;
    if (dev < 0 || dev >= kMaxDevices) return FLOWMM_ERR_UNSUPPORTED_DEVICE;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_ptr[dev]) {
        void *ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_merge_static_scratch) != cudaSuccess || !ptr) return FLOWMM_ERR_CUDA;
        g_static_ptr[dev] = ptr;
    }
    *base = g_static_ptr[dev];
    return FLOWMM_OK;
}

// The part of the workspace layout that the merge step touches, packed behind the array's status word
// (the first 256 bytes, where flowmm_merge_static_status finds it whatever the problem's shape).
Layout make_merge_layout(const flowmm_params &p) {
    Layout y = {};
    size_t o = 256;
    layout_merge(y, p, [&](size_t bytes) { const size_t at = o; o += align256(bytes); return at; });
    y.merge_status = 0;
    y.total = o;
    return y;
}

// The sum that decides whether a problem is small enough: 16 bytes and a table entry per member, which is what callers have been
// held to.  The layout above comes to less, or to 1 % more where slots are few.
size_t merge_static_need(const flowmm_params &p) {
    const size_t UH = (size_t)p.n_units * p.n_kv_heads, B = p.n_keep, E = (size_t)p.seq_len - B;
    return 256 + 4 * align256(UH * E * 4) + align256(UH * (B + E / kPiece + 1) * 16) + 3 * align256(UH * (B + 1) * 4) +
           align256(UH * (2 * (E / kPiece) + 2) * (2 * (size_t)p.head_dim + 4) * 4) + 256 + align256(UH * B * 4) + 256 +
           align256(UH * (size_t)p.seq_len * 8);
}

}  // namespace

extern "C" flowmm_status flowmm_merge_static(const flowmm_params *p, const void *k, const void *v,
                                             const int32_t *retained_idx, const int32_t *evicted_idx,
                                             const int32_t *match, const float *match_sim, void *k_out, void *v_out,
                                             void *cuda_stream) {
    profile_begin(static_cast<cudaStream_t>(cuda_stream));
    FLOWMM_TRY(validate(p));
    const bool has_e = p->n_keep < p->seq_len;
    if (!k || !v || !retained_idx || !k_out || !v_out) return FLOWMM_ERR_NULL;
    if (has_e && (!evicted_idx || !match || !match_sim)) return FLOWMM_ERR_NULL;
    if (!aligned16(k) || !aligned16(v) || !aligned16(k_out) || !aligned16(v_out) ||
        !strides_ok(p->k_stride, p->head_dim) || !strides_ok(p->v_stride, p->head_dim) ||
        !strides_ok(p->ko_stride, p->head_dim) || !strides_ok(p->vo_stride, p->head_dim))
        return FLOWMM_ERR_ALIGN;
    const Layout y = make_merge_layout(*p);
    if (merge_static_need(*p) > (size_t)FLOWMM_MERGE_STATIC_BYTES || y.total > kStaticScratch) return FLOWMM_ERR_WORKSPACE;   // problem too large for the array
    FLOWMM_TRY(check_device());
    void *base = nullptr;
    FLOWMM_TRY(merge_static_base(&base));
    FLOWMM_DEBUG_LISTS(*p, retained_idx, evicted_idx, match, static_cast<int *>(base), static_cast<cudaStream_t>(cuda_stream));
    // Nothing in this scratch has to start at zero: the rows, windows and pieces, the work counter and
    // the arrival counters are written (or cleared) by this call's first kernel before they are read, a
    // partial-sum record is only read for pieces that wrote it in the same call, and the status word is
    // sticky on purpose (the loader zero-fills the array; flowmm_merge_static_status clears the word).
    return run_merge(*p, y, k, v, retained_idx, evicted_idx, match, match_sim, k_out, v_out, base,
                     static_cast<cudaStream_t>(cuda_stream));
}

extern "C" flowmm_status flowmm_merge_static_status(void *cuda_stream) {
    FLOWMM_TRY(check_device());
    void *base = nullptr;
    FLOWMM_TRY(merge_static_base(&base));
    return flowmm_last_device_status(base, cuda_stream);
}

// Test hook of the reader above: stores `word` in the array's status word from the host, in stream order.
extern "C" flowmm_status flowmm_merge_static_poke_status(int32_t word, void *cuda_stream) {
    FLOWMM_TRY(check_device());
    void *base = nullptr;
    FLOWMM_TRY(merge_static_base(&base));
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (cudaMemcpyAsync(base, &word, sizeof(word), cudaMemcpyHostToDevice, st) != cudaSuccess) return FLOWMM_ERR_CUDA;
    return cudaStreamSynchronize(st) == cudaSuccess ? FLOWMM_OK : FLOWMM_ERR_CUDA;
}
