// libef21: C-ABI entry points (see include/ef21.h) and the host-side orchestration.
#include "../../include/ef21.h"

#include <cmath>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <set>
#include <utility>
#include <vector>

#include "apply.cuh"
#include "common.cuh"
#include "copy.cuh"
#include "ef.cuh"
#include "grad.cuh"
#include "persistent.cuh"
#include "wait_selftest.cuh"
#include "plus.cuh"
#include "topk.cuh"
#include "topk_cluster.cuh"
#include "topk_stream.cuh"

using namespace ef21;

#define CU(call)                                         \
    do {                                                 \
        cudaError_t e__ = (call);                        \
        if (e__ != cudaSuccess) return EF21_ERR_CUDA;    \
    } while (0)
#define EF(call)                                         \
    do {                                                 \
        ef21_status s__ = (call);                        \
        if (s__ != EF21_OK) return s__;                  \
    } while (0)


namespace {

constexpr size_t ALIGN = 256;
// Launch-path iterations up to this dimension are replayed as a CUDA graph.  Wider ones are launched one by one: a graph per iteration is
// a full stop between iterations, across which the gradient kernel could not fetch its first rows (20 x 300 x 5,001: 41.2 us an
// iteration without the graph, 43.1 with it; three launches take the host about 7 us).  EF21+, seven launches, 20 iterations one by one / replayed:
// 20 x 600 x 700 554 / 597, 4 x 60 x 3,000 494 / 527, 20 x 200 x 5,001 800 / 831; 4 x 50 x 600 398 / 389, 2 x 30 x 513 400 / 398.
constexpr i64 GRAPH_MAX_D = 512;
inline size_t align_up(size_t v) { return (v + ALIGN - 1) / ALIGN * ALIGN; }
inline i64 ceil_div(i64 a, i64 b) { return (a + b - 1) / b; }

// ---------------------------------------------------------------------------------------------
// Workspace layouts
// ---------------------------------------------------------------------------------------------

// Kernel launch as a programmatic dependent of whatever precedes it in the stream (see pdl_wait), with clusters of C blocks.
template <typename... Params, typename... Args>
cudaError_t launch(void (*kern)(Params...), dim3 grid, unsigned block, size_t smem, cudaStream_t st, unsigned C, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(block); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = C; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = C > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
}

// Opt-in of a kernel to more dynamic shared memory than the default 48 KB (and to clusters of more than eight blocks): an
// attribute per device, set once.
ef21_status allow_smem(const void* kern, size_t bytes, bool big_cluster = false) {
    static std::mutex mu;
    static std::set<std::pair<int, const void*>> done;
    int dev = -1;
    CU(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(mu);
    if (done.count({dev, kern})) return EF21_OK;
    CU(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    if (big_cluster) CU(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    done.insert({dev, kern});
    return EF21_OK;
}

struct TopkLayout {
    size_t state, hist, chunks, total;
    int nchunks;
    // one-pass path for long vectors (topk_stream.cuh); fast == false: sections absent
    bool fast;
    int nreg, nreg_pitch, region_log, cap;   // regions per vector (and rounded up to 8), log2 of their entries, candidate records per region
    i64 open_cap;                        // open entries per vector
    i64 samples;                         // per vector
    size_t ctl, open_hist, open_list, reg_cand, reg_base, slow_count, cand;
};

// From half of the entries on the bracket saves nothing: such messages take the multi-pass select.
bool fast_topk_eligible(i64 d, i64 k) { return d >= ST_MIN_D && 2 * k <= d; }

// Distance of the bracket's ends from the expected rank in the sample: 4.5 standard deviations of that rank.
double st_margin(double rank) { return 4.5 * std::sqrt(rank) + 4.0; }

// The three sections every Top-k call needs (selection state, histogram, per-chunk counts); the
// one-pass sections are absent.
TopkLayout topk_layout_general(i64 batch, i64 d, bool counted = false) {
    TopkLayout L{};
    L.nchunks = (int)ceil_div(d, TK_CHUNK);
    size_t o = 0;
    if (counted) { L.slow_count = o; o += align_up(4); }   // (in the same place for every batch: a handle's count runs on)
    L.state = o; o += align_up((size_t)batch * sizeof(TkState));
    L.hist = o; o += align_up((size_t)batch * TK_BINS * sizeof(unsigned));
    L.chunks = o; o += align_up((size_t)batch * (size_t)L.nchunks * sizeof(uint2));
    L.fast = false;
    L.total = o;
    return L;
}

TopkLayout topk_layout(i64 batch, i64 d, i64 k) {
    TopkLayout L = topk_layout_general(batch, d, fast_topk_eligible(d, k));
    size_t o = L.total;
    L.fast = fast_topk_eligible(d, k);
    if (L.fast) {
        L.region_log = batch * d >= ST_LARGE_TOTAL ? ST_REGION_LOG_LARGE : ST_REGION_LOG_SMALL;
        const i64 region = (i64)1 << L.region_log;
        L.nreg = (int)ceil_div(d, region);
        L.nreg_pitch = (L.nreg + 7) / 8 * 8;
        // Sample size: 512 sampled entries above the cut give a bracket of about +-20 %; at least 64 K, at most 256 K
        // entries, 4 M over the whole batch, a quarter of the vector.
        L.samples = std::max<i64>(512 * d / k, d / 64);
        L.samples = std::min<i64>(std::max<i64>(L.samples, 65536), std::max<i64>(65536, std::min<i64>(262144, 4194304 / batch)));
        L.samples = std::min<i64>(L.samples, d / 4);
        L.samples = L.samples >= 262144 ? 262144 : (L.samples >= 131072 ? 131072 : (L.samples >= 65536 ? 65536 : 32768));
        // Records per region: the expected candidates (the message plus the bracket's upper half) and six standard deviations
        // of a region's count; where more than a tenth of the entries are wanted a region is cheaper to read again.
        const double rank = (double)k * (double)L.samples / (double)d;
        const double expect = (double)region * (double)k / (double)d * (1.0 + st_margin(rank) / rank);
        const i64 cap = (i64)(expect + 6.0 * std::sqrt(expect)) + 16;
        L.cap = 10 * expect > (double)region ? 0 : (int)((cap + 7) / 8 * 8);
        L.open_cap = std::min<i64>(d, k <= 65536 ? 2 * k + 16384 : k / 2 + 131072);
        L.ctl = o; o += align_up((size_t)batch * sizeof(StCtl));
        L.open_hist = o; o += align_up((size_t)batch * ST_OPEN_BINS * 4);
        L.open_list = o; o += align_up((size_t)batch * L.open_cap * 8);
        L.reg_cand = o; o += align_up((size_t)batch * L.nreg_pitch * 4);
        L.reg_base = o; o += align_up((size_t)batch * L.nreg_pitch * 4);
        L.cand = o; o += align_up((size_t)batch * L.nreg * L.cap * sizeof(int4));
    }
    L.total = o;
    return L;
}

typedef void (*GradTileKernel)(const float*, const float*, const float*, const RowTile*, int, int, float*, double*,
                               const int*, int, const i64*, unsigned*, int);

// The gradient kernel for a row width: kernel, threads and shared memory per block; wide: a block works on whole rows and goes
// through a long tile, `resident` blocks per SM and `rows` rows at a time (0: short tiles, several per SM).
struct GradPlan { GradTileKernel kernel; unsigned threads; size_t smem; int resident, rows; };

template <int I>
constexpr GradTileKernel wide_kernel() {
    constexpr WideShape S = GRAD_WIDE_SHAPES[I];
    return grad_wide_kernel<S.columns, S.threads, S.groups, S.rows>;
}

GradPlan grad_plan(i64 ld) {
    const i64 slots = (ld / 4 + 31) / 32;
    if (slots <= 4) {
        // rows of up to 512 columns, a warp per batch of rows
        const GradTileKernel k = slots <= 1 ? grad_stream_kernel<1, 16>
                                            : (slots == 2 ? grad_stream_kernel<2, 8> : (slots == 3 ? grad_stream_kernel<3, 4> : grad_stream_kernel<4, 4>));
        return {k, GRAD_STREAM_BLOCK, (size_t)(GRAD_STREAM_BLOCK / 32) * ld * 4, 0, 0};
    }
    if (ld <= 8192) {
        static const GradTileKernel kernels[5] = {wide_kernel<0>(), wide_kernel<1>(), wide_kernel<2>(), wide_kernel<3>(), wide_kernel<4>()};
        const int at = grad_wide_shape((int)ld);
        const WideShape S = GRAD_WIDE_SHAPES[at];
        return {kernels[at], (unsigned)(S.threads * S.groups), (size_t)grad_wide_smem_bytes(S, (int)ld), 1, S.rows};
    }
    return {grad_tiles_kernel, GRAD_BLOCK, 0, 0, 0};
}

int grad_tile_rows(i64 N, i64 ld) {
    const GradPlan P = grad_plan(ld);
    // a wide tile: the rows of one resident block (the tiles of a load are cut when the shards are known, never shorter)
    if (P.resident) return (int)std::max<i64>(P.rows, ceil_div(N, 148 * P.resident));
    // two-sweep kernel: a tile's rows should stay in L1 for the second sweep; one-read kernel: any size
    i64 cap = P.kernel != grad_tiles_kernel ? GRAD_TILE_MAX_ROWS : 65536 / (ld * 4);
    if (cap < 1) cap = 1;
    if (cap > GRAD_TILE_MAX_ROWS) cap = GRAD_TILE_MAX_ROWS;
    i64 want = ceil_div(N, 4 * 148);
    if (want < 8) want = 8;
    return (int)(want < cap ? want : cap);
}

struct Layout {
    i64 ld;            // padded vector pitch (floats), multiple of 4
    int agg_tiles;     // tiles of AGG_TILE coordinates
    int tile_rows;     // rows per gradient tile
    i64 max_tiles;     // capacity of the gradient tile table
    size_t status, x, g, gi, msg_idx, msg_val, topk, agg_off, eval_out, slots;
    size_t msg2_idx, msg2_val, plus_cuts, plus_choice, plus_parts, plus_low, plus_nonzero, plus_cand;    // EF21+ (Algorithm 3)
    int plus_pitch;
    size_t A, y, row_off, tile_begin, tiles, partial, loss_partial, grad, mb_tile_begin, mb_tiles;
    size_t total;
    TopkLayout tk, tk2;                   // of n vectors; of the 2 n vectors of EF21+ (the same memory)
    bool pair;                            // EF21+ selects from 2 n vectors in one pass; else tk2 takes no part
};

bool fits_clusters(i64 batch, i64 d, i64 k);     // (tc_shape)

Layout make_layout(i64 n, i64 d, i64 k, i64 N) {
    Layout L;
    L.ld = (d + 3) / 4 * 4;
    L.agg_tiles = (int)ceil_div(d, AGG_TILE);
    L.tk = topk_layout(n, d, k);
    L.tk2 = topk_layout(2 * n, d, k);
    L.pair = L.tk2.fast && L.tk2.cap > 0 && 2 * n <= 65535 && !fits_clusters(n, d, k);          // (a batch of 2 n as one dimension of a grid)
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t at = o; o += align_up(bytes); return at; };
    L.status = take(256);
    L.x = take((size_t)L.ld * 4);
    L.g = take((size_t)L.ld * 4);
    L.gi = take((size_t)n * L.ld * 4);
    L.msg_idx = take((size_t)n * k * 4);
    L.msg_val = take((size_t)n * k * 4);
    L.topk = take(L.pair ? std::max(L.tk.total, L.tk2.total) : L.tk.total);
    L.agg_off = take((size_t)n * (L.agg_tiles + 1) * 4);
    L.eval_out = take(256);
    L.slots = take((size_t)2 * n * k * 8);
    L.msg2_idx = take((size_t)n * k * 4);
    L.msg2_val = take((size_t)n * k * 4);
    L.plus_cuts = take((size_t)2 * n * 8);
    L.plus_choice = take((size_t)n * 4);
    L.plus_parts = take((size_t)n * PLUS_MAX_PARTS * sizeof(double2));
    L.plus_pitch = (int)std::max<i64>(1, 148 * 4 / n);         // blocks per worker: four per SM in one wave
    L.plus_low = take(L.pair ? (size_t)n * L.plus_pitch * sizeof(double2) : 0);
    L.plus_nonzero = take(L.pair ? (size_t)n * L.plus_pitch * 4 : 0);
    L.plus_cand = take(L.pair ? (size_t)2 * n * ceil_div(L.tk2.nreg, 32) * 8 : 0);
    L.tile_rows = 0; L.max_tiles = 0;
    L.A = L.y = L.row_off = L.tile_begin = L.tiles = L.partial = L.loss_partial = L.grad = L.mb_tile_begin = L.mb_tiles = 0;
    if (N > 0) {
        L.tile_rows = grad_tile_rows(N, L.ld);
        // (the tiles of minibatch lists are shorter than those of the shards, but no more of them are made than fit the device)
        L.max_tiles = std::max<i64>(N / L.tile_rows, grad_plan(L.ld).resident * 148) + n;
        L.A = take((size_t)N * L.ld * 4);
        L.y = take((size_t)N * 4);
        L.row_off = take((size_t)(n + 1) * 8);
        L.tile_begin = take((size_t)(n + 1) * 4);
        L.tiles = take((size_t)L.max_tiles * sizeof(RowTile));
        L.partial = take((size_t)L.max_tiles * L.ld * 4);
        L.loss_partial = take((size_t)L.max_tiles * 8);
        L.grad = take((size_t)n * L.ld * 4);
        L.mb_tile_begin = take((size_t)(n + 1) * 4);
        L.mb_tiles = take((size_t)L.max_tiles * sizeof(RowTile));
    }
    L.total = o;
    return L;
}

bool valid_shape(i64 n, i64 d, i64 k, i64 N) {
    return n >= 1 && d >= 1 && k >= 1 && k <= d && d < ((i64)1 << 31) && N >= 0 && n <= 65535;
}

}  // namespace

// Launch plan of the persistent path (made by plan_persistent, kept in the handle until something it depends on changes).
struct PersistPlan {
    bool ok;
    bool roles;         // persistent_roles.inc (the last warp serves the block) instead of whole-block steps
    bool local;         // all workers in one cluster
    int C, rb, src, chunks, threads, extra, stages;
    size_t smem;
    PersistKernel kernel;
};

struct ef21_ctx {
    int n; i64 d; int k; float gamma, lambda; i64 N;
    cudaStream_t stream;
    int device;         // the device that was current at ef21_create
    char* ws;
    Layout L;
    bool shards_loaded, inited;
    int num_tiles, worker_tiles;        // gradient tiles: all, and the most that one worker has
    int path, last_path;
    bool agg_off_ready;                 // the last selection already wrote the aggregation's tile offsets
    int pk_cluster, pk_rb, pk_src, pk_threads;      // forced persistent-kernel shape (0 / -1 = automatic)
    int pk_used_cluster, pk_used_rb, pk_used_src, pk_used_threads;
    int pk_used_local, pk_used_stages;
    PersistPlan plan; bool plan_valid;  // cached plan of ef21_step's persistent launch
    PersistPlan mb_plan; bool mb_plan_valid; int mb_plan_tau;      // the same for the stochastic variant with mb_plan_tau rows
    unsigned pk_epoch, pk_par;          // epoch and slot half of the last persistent iteration (see PersistParams)
    int pk_body, pk_used_body;          // persistent kernel body: 0 automatic, 1 compute warps + service warp, 2 whole-block steps
    unsigned spin_limit;
    bool force_general_topk;
    int variant;                        // EF21_VARIANT_*
    int objective;                      // EF21_OBJECTIVE_*
    cudaStream_t aux_stream;            // created on first use: overlaps the next threshold estimate
    cudaEvent_t ev_fork, ev_join;
    cudaStream_t cap_stream;            // library-owned stream on which the iteration graph is captured
    cudaGraphExec_t iter_graph;         // one launch-path iteration of ef21_step, captured on first use
    int iter_graph_key;                 // what it was captured for (variant, objective)
    i64 iter_graph_launches;            // kernel launches inside it
    bool iter_graph_off;                // capture failed once: keep to plain launches
    i64 launches;
    std::vector<i64> row_off;
    std::vector<RowTile> tiles;
    std::vector<int> tile_begin;
    std::vector<RowTile> mb_tiles;      // tile table of the minibatch lists, rebuilt when tau changes
    std::vector<int> mb_tile_begin;
    int mb_tau;

    template <typename T> T* at(size_t off) const { return reinterpret_cast<T*>(ws + off); }
    float* x() const { return at<float>(L.x); }
    float* g() const { return at<float>(L.g); }
    float* gi() const { return at<float>(L.gi); }
    int* msg_idx() const { return at<int>(L.msg_idx); }
    float* msg_val() const { return at<float>(L.msg_val); }
    unsigned* status() const { return at<unsigned>(L.status); }
};

namespace {

// Several copies or clears as one launch; null destinations are left out, contiguous rows become one.
struct Copies {
    CopyArgs p;
    i64 blocks = 0;
    Copies() { p.count = 0; }
    void add(void* dst, i64 dpitch, const void* src, i64 spitch, i64 width, i64 rows) {
        if (!dst || width <= 0 || rows <= 0) return;
        if (dpitch == width && (!src || spitch == width)) { width *= rows; dpitch = spitch = width; rows = 1; }
        CopySeg& c = p.seg[p.count++];
        c.dst = static_cast<unsigned*>(dst); c.src = static_cast<const unsigned*>(src);
        c.dpitch = dpitch; c.spitch = spitch; c.width = width; c.rows = rows;
        c.units = rows * ceil_div(width, COPY_UNIT);
        blocks += c.units;
    }
    ef21_status run(cudaStream_t st, i64* launches) {
        if (blocks == 0) return EF21_OK;
        CU(launch(copy_segments_kernel, dim3((unsigned)blocks), COPY_THREADS, 0, st, 1, p));
        *launches += 1;
        return EF21_OK;
    }
};

struct TopkBuffers {
    TkState* state; unsigned* hist; uint2* chunks; int nchunks;
    TopkLayout L; char* base;            // sections of the one-pass path
};

TopkBuffers topk_buffers(char* base, const TopkLayout& L) {
    TopkBuffers B;
    B.state = reinterpret_cast<TkState*>(base + L.state);
    B.hist = reinterpret_cast<unsigned*>(base + L.hist);
    B.chunks = reinterpret_cast<uint2*>(base + L.chunks);
    B.nchunks = L.nchunks;
    B.L = L; B.base = base;
    return B;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// ---- Top-k by one cluster per vector (topk_cluster.cuh) ----
struct TcShape { int C, slice, threads; };

// Blocks per vector: as few as hold the vector in shared memory, then more while all clusters still run at once and a
// block keeps at least 8,192 entries (a shorter sweep per block; below that the two cluster barriers cost more than they
// save).  False where the vector is too long, or so long and the batch so large that the clusters would run in several
// waves of one-block-per-SM: the streaming kernels read such a batch at HBM speed (rounds with k = d / 100: 20 x 204,979 68 us in two waves,
// 48 streamed, 40 x 135,000 62 and 44, 100 x 131,072 122 and 74; k = d / 10 109 and 68, 95 and 63, 181 and 120).
// streamed: whether they would take it (fast_topk_eligible, and the caller has their scratch).  Where not, the limit is twice as long, and above it
// the multi-pass select follows (multi-pass / clusters in waves: 150 x 131,072 with 0.51 d 213 / 184 us, with 0.9 d 211 / 166; a round of
// 100 x 140,000 with 0.6 d 611 / 562).
bool tc_shape(i64 batch, i64 d, bool streamed, TcShape& S) {
    constexpr i64 SMS = 148;
    i64 C = 1;
    while (C <= TC_MAX_CLUSTER && ceil_div(d, C) > TC_MAX_SLICE) C *= 2;
    if (C > TC_MAX_CLUSTER || (d >= (streamed ? ST_MIN_D : 2 * ST_MIN_D) && batch * C > SMS)) return false;
    while (C < 8 && batch * C * 2 <= SMS && d / (2 * C) >= 8192) C *= 2;
    S.C = (int)C;
    S.slice = (int)((ceil_div(d, C) + 127) / 128 * 128);
    S.threads = C == 1 && d <= 2048 ? 256 : (C == 1 && d <= 8192 ? 512 : 1024);
    return true;
}

bool fits_clusters(i64 batch, i64 d, i64 k) { TcShape S; return tc_shape(batch, d, fast_topk_eligible(d, k), S); }

typedef void (*TcKernel)(const TcArgs);
template <int MODE>
TcKernel tc_lookup(const TcShape& S) {
    if (S.threads == 256) return tc_topk_kernel<MODE, 1, 256>;
    if (S.threads == 512) return tc_topk_kernel<MODE, 1, 512>;
    switch (S.C) {
        case 1: return tc_topk_kernel<MODE, 1, 1024>;
        case 2: return tc_topk_kernel<MODE, 2, 1024>;
        case 4: return tc_topk_kernel<MODE, 4, 1024>;
        case 8: return tc_topk_kernel<MODE, 8, 1024>;
        default: return tc_topk_kernel<MODE, 16, 1024>;
    }
}

// The same with the gradients formed on the way in.
template <int MODE>
TcKernel tc_grad_lookup(const TcShape& S) {
    if (S.threads == 256) return tc_topk_kernel<MODE, 1, 256, false, 1>;
    switch (S.C) {
        case 1: return tc_topk_kernel<MODE, 1, 512, false, 1>;
        case 2: return tc_topk_kernel<MODE, 1, 512, false, 2>;
        case 4: return tc_topk_kernel<MODE, 1, 512, false, 4>;
        default: return tc_topk_kernel<MODE, 1, 512, false, 8>;
    }
}

ef21_status enqueue_topk_cluster(cudaStream_t st, int mode, const TcShape& S, const float* a, i64 pitch_a, const float* b, i64 pitch_b,
                                 float gamma, int batch, i64 d, int k, int* idx_out, float* val_out, float* apply, i64 pitch_apply,
                                 i64* launches, unsigned* status, unsigned* slow_count = nullptr, unsigned long long* cut_out = nullptr) {
    const TcKernel kern = mode == TC_PLAIN ? tc_lookup<TC_PLAIN>(S) : (mode == TC_DIFF ? tc_lookup<TC_DIFF>(S) : tc_lookup<TC_EF>(S));
    const size_t smem = tc_smem_bytes(S.C, S.slice);
    EF(allow_smem(reinterpret_cast<const void*>(kern), tc_smem_bytes(S.C, S.C == 1 && S.threads < 1024 ? 8192 : TC_MAX_SLICE), S.C > 8));
    TcArgs p = {};
    p.a = a; p.pitch_a = pitch_a; p.b = const_cast<float*>(b); p.pitch_b = pitch_b;
    p.d = (int)d; p.k = k; p.slice = S.slice; p.gamma = gamma;
    p.idx_out = idx_out; p.val_out = val_out; p.apply = apply; p.pitch_apply = pitch_apply; p.status = status; p.slow_count = slow_count; p.cut_out = cut_out;
    CU(launch(kern, dim3((unsigned)batch * (unsigned)S.C), (unsigned)S.threads, smem, st, (unsigned)S.C, p));
    if (launches) *launches += 1;
    return EF21_OK;
}

// ---- Top-k of long vectors in one pass (topk_stream.cuh) ----
StArgs stream_args(const float* a, i64 pitch_a, const float* b, i64 pitch_b, float gamma, i64 d, int k, const TopkBuffers& B) {
    StArgs p;
    p.a = a; p.pitch_a = pitch_a; p.b = const_cast<float*>(b); p.pitch_b = pitch_b; p.d = d; p.k = k; p.pair = 0;
    p.nreg = B.L.nreg; p.nreg_pitch = B.L.nreg_pitch; p.region_log = B.L.region_log; p.cap = B.L.cap; p.open_cap = (unsigned)B.L.open_cap; p.gamma = gamma;
    p.ctl = reinterpret_cast<StCtl*>(B.base + B.L.ctl);
    p.open_hist = reinterpret_cast<unsigned*>(B.base + B.L.open_hist);
    p.open_list = reinterpret_cast<unsigned long long*>(B.base + B.L.open_list);
    p.reg_cand = reinterpret_cast<unsigned*>(B.base + B.L.reg_cand);
    p.reg_base = reinterpret_cast<unsigned*>(B.base + B.L.reg_base);
    p.cand = reinterpret_cast<int4*>(B.base + B.L.cand);
    p.slow_count = reinterpret_cast<unsigned*>(B.base + B.L.slow_count);
    return p;
}

// The bracket (first of the five kernels): clusters of eight blocks, of four or two when there are many vectors (two of these
// blocks fit on an SM).
template <int MODE>
ef21_status enqueue_stream_sample(cudaStream_t st, const StArgs& p, int batch, const TopkLayout& L, i64* launches) {
    const double rank = (double)p.k * (double)L.samples / (double)p.d;
    const int most = batch <= 37 ? 8 : (batch <= 74 ? 4 : 2);
    const int C = most == 8 && L.samples < 65536 ? 4 : most;         // (eight samples per thread at least)
    const i64 per_thread = L.samples / (ST_SAMPLE_THREADS * C);
    auto kern = C == 2 ? (per_thread >= 32 ? st_sample_kernel<MODE, 2, 32> : st_sample_kernel<MODE, 2, 16>)
                       : (C == 4 ? (per_thread >= 16 ? st_sample_kernel<MODE, 4, 16> : st_sample_kernel<MODE, 4, 8>)
                                 : (per_thread >= 32 ? st_sample_kernel<MODE, 8, 32>
                                                     : (per_thread >= 16 ? st_sample_kernel<MODE, 8, 16> : st_sample_kernel<MODE, 8, 8>)));
    CU(launch(kern, dim3((unsigned)(batch * C)), ST_SAMPLE_THREADS, 0, st, (unsigned)C, p, (float)rank, (float)st_margin(rank)));
    if (launches) *launches += 1;
    return EF21_OK;
}

template <int MODE>
ef21_status enqueue_topk_stream(cudaStream_t st, const float* a, i64 pitch_a, const float* b, i64 pitch_b, float gamma, int batch, i64 d,
                                int k, const StOut& out, const TopkBuffers& B, i64* launches, bool count_slow, bool sampled = false) {
    StArgs p = stream_args(a, pitch_a, b, pitch_b, gamma, d, k, B);
    if (!count_slow) p.slow_count = nullptr;
    if (!sampled) EF(enqueue_stream_sample<MODE>(st, p, batch, B.L, launches));
    const bool vec = aligned16(a) && (pitch_a % 4 == 0 || batch == 1) && (!b || (aligned16(b) && (pitch_b % 4 == 0 || batch == 1)));
    // open entries of a vector: twice the margin's share of the message (and the sampled range's steps, hence the 30 %)
    const double rank = (double)k * (double)B.L.samples / (double)d;
    const double open = 2.6 * st_margin(rank) / rank * (double)k;
    const i64 all_blocks = ceil_div(p.nreg, ST_WARPS);
    bool classify = vec && p.region_log == ST_REGION_LOG_LARGE && p.cap > 0;
    // blocks of the cut kernel's cluster: as few as hold the open entries where it classifies (16 x 4,194,304: 24 us with eight, 15 with
    // two), eight for the long lists of a few vectors
    int cut_blocks = classify || batch > 37 ? 2 : 8;
    while (classify && cut_blocks < 8 && open > 0.8 * cut_blocks * ST_OPEN_STAGE) cut_blocks *= 2;
    classify = classify && open <= 0.8 * cut_blocks * ST_OPEN_STAGE;
    if (!classify) cut_blocks = batch > 37 ? 2 : 8;
    if (classify) {
        CU(launch(st_collect_long_kernel<MODE>, dim3((unsigned)all_blocks, (unsigned)batch), ST_WARPS * 32, 0, st, 1, p));
    } else {
        auto collect = p.cap == 0 ? (vec ? st_collect_kernel<MODE, true, 4, false> : st_collect_kernel<MODE, false, 8, false>)
                                  : (vec ? st_collect_kernel<MODE, true, 4, true> : st_collect_kernel<MODE, false, 8, true>);
        // as many blocks as are resident, in turn; more where the open entries of one would not fit its buffer
        const i64 resident = std::max<i64>(1, 148 * 4 / batch), for_open = (i64)(1.5 * open / ST_BLOCK_OPEN);
        CU(launch(collect, dim3((unsigned)std::min(all_blocks, std::max(resident, for_open)), (unsigned)batch), ST_WARPS * 32, 0, st, 1, p));
    }
    typedef void (*CutKernel)(const StArgs);
    static const CutKernel cut_kernels[2][3] = {{st_cut_kernel<2, false>, st_cut_kernel<4, false>, st_cut_kernel<8, false>},
                                                {st_cut_kernel<2, true>, st_cut_kernel<4, true>, st_cut_kernel<8, true>}};
    const CutKernel cut = cut_kernels[classify ? 1 : 0][cut_blocks == 2 ? 0 : (cut_blocks == 4 ? 1 : 2)];
    EF(allow_smem(reinterpret_cast<const void*>(cut), st_cut_smem_bytes(classify)));
    CU(launch(cut, dim3((unsigned)(batch * cut_blocks)), 1024, st_cut_smem_bytes(classify), st, (unsigned)cut_blocks, p));
    if (p.cap > 0)
        CU(launch(st_compact_kernel<MODE>, dim3((unsigned)ceil_div(p.nreg, 32), (unsigned)batch), 256, 0, st, 1, p, out));
    else
        CU(launch(st_reread_kernel<MODE>, dim3((unsigned)ceil_div(p.nreg, 8), (unsigned)batch), 256, 0, st, 1, p, out));
    // vectors whose bracket missed: redone exactly (at once over where there is none)
    TcArgs t = {};
    t.a = a; t.pitch_a = pitch_a; t.b = const_cast<float*>(b); t.pitch_b = pitch_b; t.d = (int)d; t.k = k; t.batch = batch;
    t.idx_out = out.idx_out; t.val_out = out.val_out; t.apply = out.apply; t.pitch_apply = out.pitch_apply; t.status = out.status;
    t.flag = &p.ctl->slow; t.flag_pitch = sizeof(StCtl) / 4;
    t.tile_off = out.tile_off; t.ntiles = out.ntiles; t.tile = AGG_TILE; t.cut_out = out.cut_out;
    t.slice = (int)((ceil_div(d, 8) + 127) / 128 * 128);
    // in shared memory where they fit there (64 x 250,000 zeros, all redone: 244 us a call, from L2 340)
    constexpr int REDO = MODE == TC_EF ? TC_SENT : MODE;
    const bool fits = t.slice <= TC_MAX_SLICE;
    const TcKernel redo = fits ? tc_topk_kernel<REDO, 8, 1024, false, 0, true> : tc_topk_kernel<REDO, 8, 1024, true>;
    if (fits) EF(allow_smem(reinterpret_cast<const void*>(redo), tc_smem_bytes(8, TC_MAX_SLICE)));
    CU(launch(redo, dim3(8u * (unsigned)std::min(batch, 16)), 1024, tc_smem_bytes(8, fits ? t.slice : 0), st, 8, t));
    if (launches) *launches += 4;
    return EF21_OK;
}

// The handle's count of vectors that took the slow way (long vectors only; null where the layout keeps none).
unsigned* slow_counter(const TopkBuffers& B) { return B.L.fast ? reinterpret_cast<unsigned*>(B.base + B.L.slow_count) : nullptr; }

// Exact Top-k of v = a - b for `batch` vectors (b may be null): one cluster per vector where it fits, else the
// multi-pass radix select.
ef21_status enqueue_topk_general(cudaStream_t st, const float* a, i64 pitch_a, const float* b, i64 pitch_b,
                                 int batch, i64 d, int k, int* idx_out, float* val_out,
                                 const TopkBuffers& B, i64* launches, unsigned* status, float* apply_to = nullptr,
                                 i64 pitch_apply = 0, bool* applied = nullptr, unsigned long long* cut_out = nullptr) {
    if (applied) *applied = false;
    TcShape S;
    if (tc_shape(batch, d, false, S)) {
        // the whole selection in one launch (no scratch), which also adds the messages to apply_to if the caller asks for it
        if (applied) *applied = apply_to != nullptr;
        return enqueue_topk_cluster(st, b ? TC_DIFF : TC_PLAIN, S, a, pitch_a, b, pitch_b, 0.f, batch, d, k, idx_out, val_out, apply_to,
                                    pitch_apply, launches, status, status ? slow_counter(B) : nullptr, cut_out);
    }
    CU(launch(tk_reset_kernel, dim3(batch), 256, 0, st, 1, B.state, B.hist, batch, (unsigned)k));
    dim3 grid((unsigned)B.nchunks, (unsigned)batch);
    for (int level = 0; level < 3; ++level) {
        CU(launch(tk_hist_kernel, grid, TK_BLOCK, 0, st, 1, a, pitch_a, b, pitch_b, d, level, B.state, B.hist));
        CU(launch(tk_find_kernel, dim3(batch), 1024, 0, st, 1, B.state, B.hist, level));
    }
    CU(launch(tk_count_kernel, grid, TK_BLOCK, 0, st, 1, a, pitch_a, b, pitch_b, d, B.state, B.chunks, B.nchunks));
    CU(launch(tk_scan_kernel, dim3(batch), 1024, 0, st, 1, B.chunks, B.nchunks));
    CU(launch(tk_write_kernel, grid, TK_BLOCK, 0, st, 1, a, pitch_a, b, pitch_b, d, B.state, B.chunks, B.nchunks, k,
                                               idx_out, val_out, status, cut_out));
    if (launches) *launches += 10;
    CU(cudaGetLastError());
    return EF21_OK;
}

// Rows per tile for workers of m(i) rows: short tiles as the layout has them; wide ones as long as it takes for all tiles to be
// resident at once (a tile more than that would make a second wave of a few blocks).
template <typename Rows>
int cut_tile_rows(const ef21_ctx* c, Rows m) {
    const GradPlan P = grad_plan(c->L.ld);
    if (!P.resident) return c->L.tile_rows;
    i64 total = 0, longest = 1;
    for (int i = 0; i < c->n; ++i) { total += m(i); longest = std::max<i64>(longest, m(i)); }
    i64 R = std::max<i64>(P.rows, ceil_div(total, 148 * P.resident));
    for (; R < longest; R += std::max<i64>(1, R / 32)) {
        i64 tiles = 0;
        for (int i = 0; i < c->n; ++i) tiles += ceil_div(m(i), R);
        if (tiles <= 148 * P.resident) break;
    }
    return (int)R;
}

// What the gradients of a step are taken over: the shards' tiles, or those of the minibatch lists.
struct GradSource { int num_tiles, worker_tiles; size_t tiles, tile_begin; const int* batch_dev; int tau; };

GradSource full_source(const ef21_ctx* c) { return {c->num_tiles, c->worker_tiles, c->L.tiles, c->L.tile_begin, nullptr, 0}; }

ef21_status launch_grad_tiles(ef21_ctx* c, const GradSource& G, bool with_loss, bool early = false, bool stopped = false) {
    if (G.num_tiles == 0) return EF21_OK;
    const GradPlan P = grad_plan(c->L.ld);
    if (P.resident) EF(allow_smem(reinterpret_cast<const void*>(P.kernel), GRAD_WIDE_SMEM + GRAD_WIDE_SUMS));
    CU(launch(P.kernel, dim3((unsigned)G.num_tiles), P.threads, P.smem, c->stream, 1, c->at<float>(c->L.A), c->at<float>(c->L.y), c->x(),
              c->at<RowTile>(G.tiles), (int)c->L.ld, c->objective, c->at<float>(c->L.partial),
              with_loss ? c->at<double>(c->L.loss_partial) : nullptr, G.batch_dev, G.tau, c->at<i64>(c->L.row_off), c->status(), (early ? GRAD_WIDE_EARLY : 0) | (stopped ? GRAD_WIDE_STOPPED : 0)));
    c->launches += 1;
    return EF21_OK;
}

ef21_status launch_grad_finish(ef21_ctx* c, const GradSource& G) {
    dim3 grid((unsigned)ceil_div(c->L.ld, GRAD_FINISH_COLS), (unsigned)c->n);
    CU(launch(grad_finish_kernel, grid, GRAD_FINISH_COLS * GRAD_FINISH_LANES, 0, c->stream, 1, c->at<float>(c->L.partial),
              c->at<int>(G.tile_begin), c->at<i64>(c->L.row_off), c->x(), c->lambda, (int)c->d, (int)c->L.ld, c->at<float>(c->L.grad), G.tau));
    c->launches += 1;
    return EF21_OK;
}

// Whether the Top-k kernel can form the gradients from the tile partials itself, and in which shape: a thread then needs few dependent
// rounds of reading (eight tiles each), and a launch is saved.  Up to 512 columns and 32 tiles per worker one block per worker, two columns
// per thread.  Up to 8,192 columns and 40 tiles a cluster of up to eight blocks forms them, the first of which selects; no more blocks
// than SMs, since they are placed as the blocks of the gradient kernel end (20 x 5,001: 32.7 us an iteration with clusters of four, 35.0 of
// eight, 39.0 of two; 10 x 4,180: 16.1 with eight, 17.1 with four; two kernels 36.5 and 21.3).
bool select_can_form_grads(const ef21_ctx* c, const GradSource& G, TcShape& S) {
    if (c->d <= 512) return tc_shape(c->n, c->d, false, S) && S.threads == 256 && G.worker_tiles <= 4 * GRAD_FINISH_LANES;
    if (c->d > 8192 || G.worker_tiles > 5 * GRAD_FINISH_LANES) return false;
    i64 C = 1;
    while (C < 8 && c->n * C * 2 <= 148 && c->d / (2 * C) >= 128) C *= 2;
    S.C = (int)C; S.threads = 512;
    S.slice = (int)((c->d + 127) / 128 * 128);
    return ceil_div(c->d, C) <= 2048;
}

// Tile partials -> messages and worker states in one kernel (see select_can_form_grads).  mode: TC_DIFF, TC_EF, or TC_PLAIN for
// g_i = C(grad_i) from nothing.
ef21_status enqueue_grad_select(ef21_ctx* c, const GradSource& G, const TcShape& S, int mode) {
    const TcKernel kern = mode == TC_PLAIN ? tc_grad_lookup<TC_PLAIN>(S) : (mode == TC_DIFF ? tc_grad_lookup<TC_DIFF>(S) : tc_grad_lookup<TC_EF>(S));
    EF(allow_smem(reinterpret_cast<const void*>(kern), tc_smem_bytes(1, 8192)));
    TcArgs p = {};
    p.b = c->gi(); p.pitch_b = c->L.ld; p.d = (int)c->d; p.k = c->k; p.slice = S.slice; p.gamma = c->gamma;
    p.idx_out = c->msg_idx(); p.val_out = c->msg_val(); p.apply = c->gi(); p.pitch_apply = c->L.ld; p.status = c->status();
    p.partial = c->at<float>(c->L.partial); p.tile_begin = c->at<int>(G.tile_begin); p.row_off = c->at<i64>(c->L.row_off); p.x = c->x();
    p.lambda = c->lambda; p.ld = (int)c->L.ld; p.batch_rows = G.tau;
    CU(launch(kern, dim3((unsigned)c->n * (unsigned)S.C), (unsigned)S.threads, tc_smem_bytes(1, S.slice), c->stream, (unsigned)S.C, p));
    c->launches += 1;
    return EF21_OK;
}

ef21_status enqueue_grads(ef21_ctx* c, bool with_loss) {
    EF(launch_grad_tiles(c, full_source(c), with_loss));
    return launch_grad_finish(c, full_source(c));
}

// Minibatch gradients (Algorithm 5): worker i averages over the tau rows batch[i][0..tau) of its shard.
ef21_status minibatch_source(ef21_ctx* c, const int* batch_dev, int tau, GradSource& G) {
    if (c->mb_tau != tau) {            // (re)build the tile table of the batch lists
        const int R = cut_tile_rows(c, [&](int) { return (i64)tau; });
        c->mb_tiles.clear();
        c->mb_tile_begin.assign(c->n + 1, 0);
        for (int i = 0; i < c->n; ++i) {
            c->mb_tile_begin[i] = (int)c->mb_tiles.size();
            for (int r = 0; r < tau; r += R) {
                RowTile t; t.row0 = r; t.rows = std::min(R, tau - r); t.worker = i;
                c->mb_tiles.push_back(t);
            }
        }
        c->mb_tile_begin[c->n] = (int)c->mb_tiles.size();
        if ((i64)c->mb_tiles.size() > c->L.max_tiles) return EF21_ERR_WORKSPACE;
        CU(cudaMemcpyAsync(c->at<int>(c->L.mb_tile_begin), c->mb_tile_begin.data(), (size_t)(c->n + 1) * 4,
                           cudaMemcpyHostToDevice, c->stream));
        CU(cudaMemcpyAsync(c->at<RowTile>(c->L.mb_tiles), c->mb_tiles.data(), c->mb_tiles.size() * sizeof(RowTile),
                           cudaMemcpyHostToDevice, c->stream));
        CU(cudaStreamSynchronize(c->stream));      // the host vectors may be rebuilt by the next call
        c->mb_tau = tau;
    }
    int worker_tiles = 0;
    for (int i = 0; i < c->n; ++i) worker_tiles = std::max(worker_tiles, c->mb_tile_begin[i + 1] - c->mb_tile_begin[i]);
    G = {(int)c->mb_tiles.size(), worker_tiles, c->L.mb_tiles, c->L.mb_tile_begin, batch_dev, tau};
    return EF21_OK;
}

// Whether the handle's rounds take the one-pass Top-k of long vectors.
bool long_topk(const ef21_ctx* c) {
    TcShape S;
    return c->L.tk.fast && !c->force_general_topk && !tc_shape(c->n, c->d, true, S);
}

// Selection half of a message round: c_i = C(a_i - g_i) and g_i += c_i.  sampled: the threshold
// kernel of the one-pass Top-k has already run for these inputs.
ef21_status enqueue_round_select(ef21_ctx* c, const float* a, i64 pitch_a, bool sampled) {
    TopkBuffers B = topk_buffers(c->ws + c->L.topk, c->L.tk);
    if (long_topk(c)) {
        // the compaction also leaves the per-tile offsets of the messages for the aggregation
        const StOut out = {c->msg_idx(), c->msg_val(), c->gi(), c->L.ld, c->at<int>(c->L.agg_off), c->L.agg_tiles, c->status(), nullptr};
        EF(enqueue_topk_stream<TC_DIFF>(c->stream, a, pitch_a, c->gi(), c->L.ld, 0.f, c->n, c->d, c->k, out, B, &c->launches, true, sampled));
        c->agg_off_ready = true;
    } else {
        c->agg_off_ready = false;
        bool applied = false;
        EF(enqueue_topk_general(c->stream, a, pitch_a, c->gi(), c->L.ld, c->n, c->d, c->k, c->msg_idx(),
                                c->msg_val(), B, &c->launches, c->status(), c->gi(), c->L.ld, &applied));
        if (!applied) {
            const i64 total = (i64)c->n * c->k;
            CU(launch(apply_messages_kernel, dim3((unsigned)ceil_div(total, 256)), 256, 0, c->stream, 1, c->msg_idx(), c->msg_val(), total,
                                                                                        c->k, c->L.ld, c->gi()));
            c->launches += 1;
        }
    }
    CU(cudaGetLastError());
    return EF21_OK;
}

ef21_status enqueue_aggregate_into(ef21_ctx* c, float* target, float factor, int xmode);

// Aggregation half: g += (1/n) sum c_i (and, with xmode, an update of x in the same kernel).
ef21_status enqueue_round_aggregate(ef21_ctx* c, int xmode) {
    return enqueue_aggregate_into(c, c->g(), 1.0f / (float)c->n, xmode);
}

bool agg_by_table(const ef21_ctx* c) {
    return c->d <= AGG_TABLE_MAX_D && c->n <= AGG_TABLE_MAX_N && (i64)c->n * c->k <= AGG_TABLE_MAX_MESSAGES;
}

// target_j += factor * (sum over workers, ascending, of the values sent for coordinate j).
ef21_status enqueue_aggregate_into(ef21_ctx* c, float* target, float factor, int xmode) {
    if (agg_by_table(c)) {
        auto kern = xmode == AGG_X_KEEP ? aggregate_table_kernel<AGG_X_KEEP>
                    : xmode == AGG_INIT ? aggregate_table_kernel<AGG_INIT>
                                        : (xmode == AGG_X_BEFORE ? aggregate_table_kernel<AGG_X_BEFORE> : aggregate_table_kernel<AGG_X_AFTER>);
        const size_t smem = (size_t)c->n * AGG_TABLE_COLS * 4;
        EF(allow_smem(reinterpret_cast<const void*>(kern), (size_t)AGG_TABLE_MAX_N * AGG_TABLE_COLS * 4));
        CU(launch(kern, dim3((unsigned)ceil_div(c->d, AGG_TABLE_COLS)), AGG_BLOCK, smem, c->stream, 1, c->msg_idx(), c->msg_val(), c->n, c->k,
                  (int)c->d, factor, c->gamma, target, c->x()));
        c->launches += 1;
        return EF21_OK;
    }
    if (!c->agg_off_ready) {
        const i64 noff = (i64)c->n * (c->L.agg_tiles + 1);
        CU(launch(agg_offsets_kernel, dim3((unsigned)ceil_div(noff, 256)), 256, 0, c->stream, 1, c->msg_idx(), c->n, c->k,
                  c->L.agg_tiles, c->at<int>(c->L.agg_off)));
        c->launches += 1;
    }
    c->agg_off_ready = false;
    const dim3 tiles(c->L.agg_tiles);
    const int* off = c->at<int>(c->L.agg_off);
    if (c->n <= AGG_STAGE_MAX_N) {
        auto kern = xmode == AGG_X_KEEP ? aggregate_staged_kernel<AGG_X_KEEP>
                                        : (xmode == AGG_X_BEFORE ? aggregate_staged_kernel<AGG_X_BEFORE> : aggregate_staged_kernel<AGG_X_AFTER>);
        CU(launch(kern, tiles, AGG_BLOCK, 0, c->stream, 1, c->msg_idx(), c->msg_val(), off, c->n, c->k, c->L.agg_tiles, c->d, factor, c->gamma,
                  target, c->x(), long_topk(c) ? 1 : 0));
    } else {
        auto kern = xmode == AGG_X_KEEP ? aggregate_kernel<AGG_X_KEEP>
                                        : (xmode == AGG_X_BEFORE ? aggregate_kernel<AGG_X_BEFORE> : aggregate_kernel<AGG_X_AFTER>);
        CU(launch(kern, tiles, AGG_BLOCK, 0, c->stream, 1, c->msg_idx(), c->msg_val(), off, c->n, c->k, c->L.agg_tiles, c->d, factor, c->gamma,
                  target, c->x()));
    }
    c->launches += 1;
    return EF21_OK;
}

ef21_status enqueue_round(ef21_ctx* c, const float* a, i64 pitch_a, int xmode) {
    EF(enqueue_round_select(c, a, pitch_a, false));
    return enqueue_round_aggregate(c, xmode);
}

// Both selections of EF21+ on long vectors, as a batch of 2 n, and the distortions' sums (topk_stream.cuh): five launches.
ef21_status enqueue_plus_select(ef21_ctx* c, const float* a, i64 pitch_a, unsigned long long* cuts, PlusSums& sums) {
    const TopkBuffers B = topk_buffers(c->ws + c->L.topk, c->L.tk2);
    const int n = c->n;
    StArgs p = stream_args(a, pitch_a, c->gi(), c->L.ld, 0.f, c->d, c->k, B);
    p.pair = n;
    const unsigned groups = (unsigned)ceil_div(p.nreg, 32);
    sums.low = c->at<double2>(c->L.plus_low); sums.nonzero = c->at<int>(c->L.plus_nonzero); sums.low_pitch = c->L.plus_pitch;
    // as many blocks as are resident at most, every warp with the same number of regions
    const i64 rounds = ceil_div(ceil_div(p.nreg, ST_WARPS), c->L.plus_pitch);
    sums.low_parts = (int)ceil_div(ceil_div(p.nreg, ST_WARPS), rounds);
    sums.cand = c->at<double>(c->L.plus_cand); sums.groups = (int)groups; sums.ctl = p.ctl;
    EF(enqueue_stream_sample<TC_PAIR>(c->stream, p, 2 * n, B.L, &c->launches));
    EF(allow_smem(reinterpret_cast<const void*>(st_collect_pair_kernel), sizeof(StPairShared)));
    CU(launch(st_collect_pair_kernel, dim3((unsigned)sums.low_parts, (unsigned)n), ST_WARPS * 32, sizeof(StPairShared), c->stream, 1, p, sums));
    const int cut_blocks = 2 * n > 37 ? 2 : 8;
    auto cut = cut_blocks == 2 ? st_cut_kernel<2, false> : st_cut_kernel<8, false>;
    EF(allow_smem(reinterpret_cast<const void*>(cut), st_cut_smem_bytes(false)));
    CU(launch(cut, dim3((unsigned)(2 * n * cut_blocks)), 1024, st_cut_smem_bytes(false), c->stream, (unsigned)cut_blocks, p));
    int* idx_b = c->at<int>(c->L.msg2_idx);
    float* val_b = c->at<float>(c->L.msg2_val);
    CU(launch(st_compact_pair_kernel, dim3(groups, (unsigned)(2 * n)), 256, 0, c->stream, 1, p, sums, c->msg_idx(), c->msg_val(), idx_b, val_b, cuts,
              c->status()));
    TcArgs m = {};
    m.a = a; m.pitch_a = pitch_a; m.b = c->gi(); m.pitch_b = c->L.ld; m.d = (int)c->d; m.k = c->k; m.batch = n;
    m.idx_out = c->msg_idx(); m.val_out = c->msg_val(); m.status = c->status(); m.cut_out = cuts;
    m.flag = &p.ctl->slow; m.flag_pitch = sizeof(StCtl) / 4; m.slice = (int)((ceil_div(c->d, 8) + 127) / 128 * 128);
    TcArgs b = m;
    b.b = nullptr; b.pitch_b = 0; b.idx_out = idx_b; b.val_out = val_b; b.cut_out = cuts + n; b.flag = &p.ctl[n].slow;
    CU(launch(tc_pair_kernel<8, 1024>, dim3(8u * (unsigned)std::min(2 * n, 16)), 1024, tc_smem_bytes(8, 0), c->stream, 8, m, b));
    c->launches += 4;
    return EF21_OK;
}

// One round of EF21+ (Algorithm 3) on local gradients a: both compressed vectors, the choice by
// distortion, g_i <- chosen, g = (1/n) sum g_i.
ef21_status enqueue_plus_round(ef21_ctx* c, const float* a, i64 pitch_a, int xmode) {
    TopkBuffers B = topk_buffers(c->ws + c->L.topk, c->L.tk);
    int* idx_b = c->at<int>(c->L.msg2_idx);
    float* val_b = c->at<float>(c->L.msg2_val);
    unsigned long long* cuts = c->at<unsigned long long>(c->L.plus_cuts);       // [2][n]: Markov, plain
    PlusSums sums = {};
    if (long_topk(c) && c->L.pair) {
        EF(enqueue_plus_select(c, a, pitch_a, cuts, sums));
    } else if (long_topk(c)) {
        const StOut om = {c->msg_idx(), c->msg_val(), nullptr, 0, nullptr, 0, c->status(), cuts};
        const StOut ob = {idx_b, val_b, nullptr, 0, nullptr, 0, c->status(), cuts + c->n};
        EF(enqueue_topk_stream<TC_DIFF>(c->stream, a, pitch_a, c->gi(), c->L.ld, 0.f, c->n, c->d, c->k, om, B, &c->launches, true));
        EF(enqueue_topk_stream<TC_PLAIN>(c->stream, a, pitch_a, nullptr, 0, 0.f, c->n, c->d, c->k, ob, B, &c->launches, true));
    } else {
        EF(enqueue_topk_general(c->stream, a, pitch_a, c->gi(), c->L.ld, c->n, c->d, c->k, c->msg_idx(), c->msg_val(), B,
                                &c->launches, c->status(), nullptr, 0, nullptr, cuts));
        EF(enqueue_topk_general(c->stream, a, pitch_a, nullptr, 0, c->n, c->d, c->k, idx_b, val_b, B, &c->launches, c->status(), nullptr, 0,
                                nullptr, cuts + c->n));
    }
    // four blocks per SM over all workers, parts of at least 4,096 coordinates
    const i64 parts = std::max<i64>(1, std::min<i64>(std::min<i64>(PLUS_MAX_PARTS, 148 * 4 / c->n), c->d / 4096));
    double2* part = c->at<double2>(c->L.plus_parts);
    CU(launch(sums.low ? plus_distortion_kernel<true> : plus_distortion_kernel<false>, dim3((unsigned)parts, (unsigned)c->n), PLUS_BLOCK, 0, c->stream, 1, a, pitch_a, c->gi(), c->L.ld, c->d,
              ceil_div(c->d, parts), cuts, part, sums));
    CU(launch(sums.low ? plus_choose_kernel<true> : plus_choose_kernel<false>, dim3((unsigned)ceil_div(c->k, PLUS_BLOCK), (unsigned)c->n), PLUS_BLOCK, 0, c->stream, 1, part, (int)parts, c->gi(),
              c->L.ld, c->k, c->msg_idx(), c->msg_val(), idx_b, val_b, c->at<int>(c->L.plus_choice), sums));
    const unsigned blocks = (unsigned)std::min<i64>(ceil_div(c->d, 1024), 148 * 8);
    auto mean = xmode == AGG_X_KEEP ? plus_mean_kernel<AGG_X_KEEP>
                                    : (xmode == AGG_X_BEFORE ? plus_mean_kernel<AGG_X_BEFORE> : plus_mean_kernel<AGG_X_AFTER>);
    CU(launch(mean, dim3(blocks), 256, 0, c->stream, 1, a, pitch_a, cuts + c->n, c->at<int>(c->L.plus_choice), c->gi(), c->L.ld, c->n, c->d,
              1.0f / (float)c->n, c->gamma, c->g(), c->x()));
    c->launches += 3;
    return EF21_OK;
}

// One iteration of the original error feedback method (Algorithm 4) on local gradients a, from the
// state (x, e_i): e_i becomes p_i = e_i + gamma a_i, the messages are w_i = C(p_i), the master moves
// x by -(1/n) sum w_i, and e_i <- p_i - w_i.
ef21_status enqueue_ef_round(ef21_ctx* c, const float* a, i64 pitch_a) {
    TopkBuffers B = topk_buffers(c->ws + c->L.topk, c->L.tk);
    TcShape S;
    c->agg_off_ready = false;
    if (tc_shape(c->n, c->d, c->L.tk.fast && !c->force_general_topk, S)) {
        // the kernel that selects also forms p_i (kept as the new error) and clears the sent coordinates
        EF(enqueue_topk_cluster(c->stream, TC_EF, S, a, pitch_a, c->gi(), c->L.ld, c->gamma, c->n, c->d, c->k, c->msg_idx(), c->msg_val(),
                                c->gi(), c->L.ld, &c->launches, c->status(), slow_counter(B)));
    } else if (long_topk(c)) {
        const StOut out = {c->msg_idx(), c->msg_val(), c->gi(), c->L.ld, c->at<int>(c->L.agg_off), c->L.agg_tiles, c->status(), nullptr};
        EF(enqueue_topk_stream<TC_EF>(c->stream, a, pitch_a, c->gi(), c->L.ld, c->gamma, c->n, c->d, c->k, out, B, &c->launches, true));
        c->agg_off_ready = true;
    } else {
        const unsigned blocks = (unsigned)std::min<i64>(ceil_div((i64)c->n * c->d, 256), 148 * 16);
        CU(launch(ef_compose_kernel, dim3(blocks), 256, 0, c->stream, 1, a, pitch_a, c->gi(), c->L.ld, c->n, c->d, c->gamma));
        EF(enqueue_topk_general(c->stream, c->gi(), c->L.ld, nullptr, 0, c->n, c->d, c->k, c->msg_idx(), c->msg_val(), B,
                                &c->launches, c->status()));
        const i64 total = (i64)c->n * c->k;
        CU(launch(ef_subtract_sent_kernel, dim3((unsigned)ceil_div(total, 256)), 256, 0, c->stream, 1, c->msg_idx(), c->msg_val(), total, c->k,
                  c->L.ld, c->gi()));
        c->launches += 2;
    }
    return enqueue_aggregate_into(c, c->x(), -(1.0f / (float)c->n), AGG_X_KEEP);
}

ef21_status enqueue_x_update(ef21_ctx* c) {
    const unsigned blocks = (unsigned)std::min<i64>(ceil_div(c->d, 256), 148 * 8);
    CU(launch(x_update_kernel, dim3(blocks), 256, 0, c->stream, 1, c->g(), c->x(), c->d, c->gamma));
    c->launches += 1;
    CU(cudaGetLastError());
    return EF21_OK;
}

ef21_status zero_state(ef21_ctx* c) {
    Copies m;
    m.add(c->gi(), c->L.ld, nullptr, 0, c->L.ld, c->n);
    m.add(c->g(), c->L.ld, nullptr, 0, c->L.ld, 1);
    return m.run(c->stream, &c->launches);
}

ef21_status init_from(ef21_ctx* c, const float* V, i64 pitch, int mode) {
    EF(zero_state(c));
    if (mode == EF21_INIT_COMPRESSED) {
        EF(enqueue_round(c, V, pitch, AGG_X_KEEP));
    } else if (mode == EF21_INIT_GRADIENT) {
        const unsigned blocks = (unsigned)std::min<i64>(ceil_div(c->d, 256), 148 * 8);
        CU(launch(dense_init_kernel, dim3(blocks), 256, 0, c->stream, 1, V, pitch, c->n, c->d, c->L.ld, 1.0f / (float)c->n,
                                                        c->gi(), c->g()));
        c->launches += 1;
        CU(cudaGetLastError());
    }
    c->inited = true;
    return EF21_OK;
}

ef21_status finish_load(ef21_ctx* c, const i64* row_offsets_host) {
    // Validate and build the tile table.
    if (row_offsets_host[0] != 0 || row_offsets_host[c->n] != c->N) return EF21_ERR_INVALID_ARG;
    for (int i = 0; i < c->n; ++i)
        if (row_offsets_host[i + 1] < row_offsets_host[i]) return EF21_ERR_INVALID_ARG;
    c->row_off.assign(row_offsets_host, row_offsets_host + c->n + 1);
    c->tiles.clear();
    c->tile_begin.assign(c->n + 1, 0);
    const int R = cut_tile_rows(c, [&](int i) { return c->row_off[i + 1] - c->row_off[i]; });
    for (int i = 0; i < c->n; ++i) {
        c->tile_begin[i] = (int)c->tiles.size();
        for (i64 r = c->row_off[i]; r < c->row_off[i + 1]; r += R) {
            RowTile t;
            t.row0 = r;
            t.rows = (int)std::min<i64>(R, c->row_off[i + 1] - r);
            t.worker = i;
            c->tiles.push_back(t);
        }
    }
    c->tile_begin[c->n] = (int)c->tiles.size();
    c->num_tiles = (int)c->tiles.size();
    c->worker_tiles = 0;
    for (int i = 0; i < c->n; ++i) c->worker_tiles = std::max(c->worker_tiles, c->tile_begin[i + 1] - c->tile_begin[i]);
    if ((i64)c->num_tiles > c->L.max_tiles) return EF21_ERR_WORKSPACE;
    // a captured launch-path iteration has the old tile count baked into its grid
    if (c->iter_graph) { cudaGraphExecDestroy(c->iter_graph); c->iter_graph = nullptr; }
    c->plan_valid = false; c->mb_plan_valid = false;
    CU(cudaMemcpyAsync(c->at<i64>(c->L.row_off), c->row_off.data(), (size_t)(c->n + 1) * 8, cudaMemcpyHostToDevice, c->stream));
    CU(cudaMemcpyAsync(c->at<int>(c->L.tile_begin), c->tile_begin.data(), (size_t)(c->n + 1) * 4, cudaMemcpyHostToDevice, c->stream));
    if (c->num_tiles > 0)
        CU(cudaMemcpyAsync(c->at<RowTile>(c->L.tiles), c->tiles.data(), (size_t)c->num_tiles * sizeof(RowTile),
                           cudaMemcpyHostToDevice, c->stream));
    c->shards_loaded = true;
    return EF21_OK;
}


// ---------------------------------------------------------------------------------------------
// Persistent path
// ---------------------------------------------------------------------------------------------


// From two entries per worker on, the received messages are scattered into a [n][ld] table in shared
// memory (if that table is small): aggregation then costs n reads per coordinate instead of n*k.
constexpr int PK_STATIC_SMEM = 2048;                  // room for the kernels' static shared memory
constexpr i64 PK_RING_MAX_BYTES = (i64)110 << 20;      // shards that an L2 of 126 MB holds

bool pk_use_table(int n, int ld, int k) { return k >= 2 && (size_t)n * ld * 4 <= (size_t)PK_TABLE_MAX_BYTES; }

// RING source: barriers and stages of all warps.
size_t pk_ring_bytes(int ld, int threads, int rb, int stages) {
    return (size_t)(threads / 32) * (PK_RING_MAX_STAGES * 8 + (size_t)stages * rb * ld * 4);
}

size_t pk_smem_bytes(bool plus, int n, int k, int ld, int C, int nmsg, int src, i64 rows_cta, int threads) {
    size_t b = (size_t)(6 + threads / 32 + C) * ld * 4 + (size_t)((nmsg + 1) & ~1) * 8 + (size_t)((2 * ld + 15) & ~15);
    if (plus) b += (size_t)n * ld * 4 + (size_t)ld * 4 + (size_t)((ld + 15) & ~15) + (size_t)((n + 15) & ~15) + (size_t)2 * (threads / 32) * 8 + 16;   // replicas of all g_i, grad_i, second selection, branches, distortion partials
    else if (pk_use_table(n, ld, k)) b += (size_t)n * ld * 4;
    if (src == PK_SRC_SMEM) b += (size_t)rows_cta * ld * 4;
    return b;
}

// Shared memory of the kernel whose last warp serves the block (persistent_roles.inc): x, g, g_i, message
// sums, one partial per compute warp, the partials of the cluster's blocks, the message flags, the row slice.
size_t pk_roles_smem_bytes(int ld, int C, int src, i64 rows_cta, int threads) {
    size_t b = (size_t)(6 + threads / 32 + C) * ld * 4 + (size_t)((ld + 15) & ~15);
    if (src == PK_SRC_SMEM) b += (size_t)rows_cta * ld * 4;
    return b;
}

PersistPlan plan_persistent_body(ef21_ctx* c, bool roles, int tau = 0);

PersistKernel persistent_kernel_of(const ef21_ctx* c, bool roles, bool local, int chunks, int rb, int src, int threads, int extra) {
    const bool ef = c->variant == EF21_VARIANT_EF, plus = c->variant == EF21_VARIANT_EF21_PLUS;
    auto lookup = roles ? (ef ? (local ? pk_lookup_local_ef : pk_lookup_ef) : (local ? pk_lookup_local_ef21 : pk_lookup_ef21))
                  : ef  ? (local ? pk_lookup_local_wide_ef : pk_lookup_wide_ef)
                  : plus ? (local ? pk_lookup_local_plus : pk_lookup_plus)
                         : (local ? pk_lookup_local_wide_ef21 : pk_lookup_wide_ef21);
    return lookup(chunks, rb, src, threads, extra);
}

// Chooses the kernel body, cluster size, block size, rows per batch and the source of the shard rows; checks
// that all n clusters can be resident at once (the blocks wait on one another through global memory).
PersistPlan plan_persistent(ef21_ctx* c) {
    // Automatic choice: the serving-warp body for Top-1 (2.6 against 3.2 us per iteration on the mushrooms-shaped
    // workload, 3.4 against 4.0 on the a9a-shaped one, the same 10.4 on the w8a-shaped one, measured); with more
    // entries per message the three polling rounds of a single warp cost more than the whole block's table (a9a-shaped, Top-4:
    // 5.6 against 4.5 us).
    const bool roles_can = c->variant != EF21_VARIANT_EF21_PLUS && c->k <= PK_ROLES_MAX_K;
    const bool roles_first = c->pk_body == 1 || (c->pk_body == 0 && c->k == 1);
    if (roles_can && roles_first) {
        PersistPlan P = plan_persistent_body(c, true);
        if (P.ok || c->pk_body == 1) return P;
    }
    if (c->pk_body == 1) { PersistPlan P{}; return P; }
    return plan_persistent_body(c, false);
}

// tau > 0: plan for the stochastic variant (tau sampled rows per worker and iteration, read from global memory).
PersistPlan plan_persistent_body(ef21_ctx* c, bool roles, int tau) {
    PersistPlan P{}; P.roles = roles;
    const int ld = (int)c->L.ld;
    if (!c->shards_loaded || ld > 512 || c->k > PK_MAX_K || (i64)c->n * c->k > PK_MAX_MSGS) return P;
    const bool plus = c->variant == EF21_VARIANT_EF21_PLUS;
    if (plus && (size_t)c->n * ld * 4 > (size_t)PK_TABLE_MAX_BYTES) return P;      // every block keeps all g_i
    int dev = 0, sms = 0, max_smem = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return P;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const int chunk_slots = (ld / 4 + 31) / 32;
    const int max_rb256 = chunk_slots == 1 ? 32 : (chunk_slots == 2 ? 16 : 8);      // rb * chunk_slots <= 32
    const int max_rb512 = chunk_slots == 1 ? 16 : (chunk_slots == 2 ? 8 : 4);       // rb * chunk_slots <= 16
    i64 max_m = 0;
    for (int i = 0; i < c->n; ++i) max_m = std::max<i64>(max_m, c->row_off[i + 1] - c->row_off[i]);
    if (tau > 0) max_m = tau;
    const int nmsg = c->n * c->k;

    // One candidate shape for a cluster size: rows in registers with 8 warps if they fit, else with 16
    // warps, else staged in shared memory or streamed from L2 with 16 warps.
    int stages = 0;
    auto shape_for = [&](int C, int& rb, int& src, int& threads, int& extra) {
        const i64 rows_cta = ceil_div(std::max<i64>(max_m, 1), C);
        rb = 0; extra = 0;
        // (sampled rows: the serving warp gets none, the others fetch theirs ahead of time)
        for (int cand = 8; cand <= max_rb256 && !rb; cand *= 2)
            if (ceil_div(rows_cta, cand) <= (tau > 0 ? 7 : 8)) { rb = cand; src = PK_SRC_REG; threads = 256; }
        for (int cand = 4; cand <= max_rb512 && !rb; cand *= 2)
            if (ceil_div(rows_cta, cand) <= (tau > 0 ? 15 : 16)) { rb = cand; src = PK_SRC_REG; threads = 512; }
        // one row more than 16 per warp still fits the registers of 16 warps (one chunk slot)
        if (!rb && chunk_slots == 1 && ceil_div(rows_cta, 17) <= 16 && c->pk_threads == 0 && c->pk_rb == 0 && c->pk_src < 0) {
            rb = 16; extra = 1; src = PK_SRC_REG; threads = 512;
        }
        if (!rb) {
            rb = max_rb512; threads = 512;
            const size_t with_slice = roles ? pk_roles_smem_bytes(ld, C, PK_SRC_SMEM, rows_cta, threads)
                                            : pk_smem_bytes(plus, c->n, c->k, ld, C, nmsg, PK_SRC_SMEM, rows_cta, threads);
            src = with_slice <= (size_t)max_smem - PK_STATIC_SMEM ? PK_SRC_SMEM : PK_SRC_GMEM;
        }
        if (c->pk_threads > 0) {
            threads = c->pk_threads;
            const int cap = threads == 512 ? max_rb512 : max_rb256;
            if (rb > cap) rb = cap;
            if (src == PK_SRC_REG && ceil_div(rows_cta, rb) > threads / 32) src = PK_SRC_SMEM;
        }
        if (c->pk_rb > 0) {
            rb = c->pk_rb;
            if (src == PK_SRC_REG && ceil_div(rows_cta, rb) > threads / 32) src = PK_SRC_SMEM;
        }
        if (c->pk_src >= 0) src = c->pk_src;
        if (tau > 0) src = PK_SRC_SAMPLED;       // sampled rows change every iteration: read through the list
        stages = 0;
        if (src == PK_SRC_GMEM && c->pk_src < 0 && c->pk_rb == 0 && threads == 512 && c->N * (i64)ld * 4 <= PK_RING_MAX_BYTES) {
            // Rows that stay in L2 come through a ring in shared memory where batches of at least eight rows leave room for two
            // stages per warp (rows of up to 190 columns; 20 x 5,000 x 123: 8.8 against 10.6 us per iteration, 100 x 1,000 x 100:
            // 10.5 against 13.7).  With four rows per batch, and beyond L2, plain loads are as fast or faster (10.1 against
            // 10.5 us on 60 MB of 300 columns, 35 against 37 us on 200 MB of 123).
            const size_t rest = roles ? pk_roles_smem_bytes(ld, C, src, rows_cta, threads)
                                      : pk_smem_bytes(plus, c->n, c->k, ld, C, nmsg, src, rows_cta, threads);
            for (int cand = max_rb512; cand >= 8 && stages < 2; cand /= 2) {
                stages = 0;
                while (stages < PK_RING_MAX_STAGES && rest + pk_ring_bytes(ld, threads, cand, stages + 1) <= (size_t)max_smem - PK_STATIC_SMEM) ++stages;
                if (stages >= 2) { src = PK_SRC_RING; rb = cand; }
            }
            if (src != PK_SRC_RING) stages = 0;
        }
        return rows_cta;
    };

    // Order in which cluster sizes are tried: the smallest one that keeps a block's rows in registers
    // (fewer blocks = fewer senders and pollers), then the largest first.
    int order[9], norder = 0;
    if (c->pk_cluster > 0) {
        order[norder++] = c->pk_cluster;
    } else {
        int pref = 0;
        for (int C = 1; C <= 8 && !pref; ++C) {
            if ((i64)c->n * C > sms) break;
            int rb, src, threads, extra;
            shape_for(C, rb, src, threads, extra);
            if ((src == PK_SRC_REG || tau > 0) && threads == 256 && rb <= 16) pref = C;
        }
        if (pref) order[norder++] = pref;
        for (int C = 8; C >= 1; --C)
            if (C != pref) order[norder++] = C;
    }
    for (int oi = 0; oi < norder; ++oi) {
        const int C = order[oi];
        if ((i64)c->n * C > sms) continue;
        int rb = 0, src = PK_SRC_GMEM, threads = 256, extra = 0;
        const i64 rows_cta = shape_for(C, rb, src, threads, extra);
        if (c->pk_cluster == 0 && C > 1 && rows_cta < 8) continue;       // do not split below one batch
        if (src == PK_SRC_REG && ceil_div(rows_cta, rb + extra) > threads / 32) continue;
        const size_t smem = (roles ? pk_roles_smem_bytes(ld, C, src, rows_cta, threads)
                                   : pk_smem_bytes(plus, c->n, c->k, ld, C, nmsg, src, rows_cta, threads)) +
                            (src == PK_SRC_RING ? pk_ring_bytes(ld, threads, rb, stages) : 0);
        if (smem > (size_t)max_smem - PK_STATIC_SMEM) continue;
        // All workers in one cluster where it holds them and the kernel exists (rows in registers, or sampled), else a cluster per
        // worker.  A message then takes a store to shared memory instead of a trip through L2: 4 workers, d = 64, Top-4 2.55 ->
        // 2.17 us per iteration, 8 x 64 Top-2 2.45 -> 1.99, 10 x 112 Top-1 2.23 -> 2.00, 32 sampled rows 2.32 -> 2.00.  Vectors
        // of more than 128 coordinates with several entries per message stay with a cluster per worker (2 x 500, Top-8: 4.3 us
        // against 4.6: a thread then has several coordinates to look the words through for).
        for (const bool local : {true, false}) {
            if (local && ((i64)c->n * C > PK_LOCAL_BLOCKS || nmsg > PK_LOCAL_MSGS)) continue;
            PersistKernel kern = persistent_kernel_of(c, roles, local, chunk_slots, rb, src, threads, extra);
            if (!kern) continue;
            // the device's opt-in limit (less the kernel's static part), so that no other handle's plan for the same
            // kernel can lower it under this one's need
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem - PK_STATIC_SMEM) != cudaSuccess ||
                (local && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
                cudaGetLastError();
                continue;
            }
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)(c->n * C)); cfg.blockDim = dim3((unsigned)threads); cfg.dynamicSmemBytes = smem;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = (unsigned)(local ? c->n * C : C); attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr; cfg.numAttrs = 1;
            int active = 0;
            if (cudaOccupancyMaxActiveClusters(&active, kern, &cfg) != cudaSuccess) { cudaGetLastError(); continue; }
            if (active < (local ? 1 : c->n)) continue;
            P.ok = true; P.local = local; P.C = C; P.rb = rb; P.src = src; P.chunks = chunk_slots; P.threads = threads; P.extra = extra;
            P.smem = smem; P.stages = stages; P.kernel = kern;
            return P;
        }
    }
    return P;
}

// Persistent launches of different handles must not overlap on a device.  Each needs all of its clusters resident at
// once (they wait on one another through global memory); two launches that each got part of the SMs would wait for
// the other's until their bounded waits expire.  Launches on one stream are ordered by the stream.  A launch on another
// stream than the device's last persistent launch first waits (on the device, not on the host) for everything enqueued
// on that stream so far.
struct PersistGate {
    std::mutex mu;
    bool any = false;              // a persistent launch has been enqueued on this device
    bool detached = false;         // its handle is gone: `ev` stands for the work, the stream is not touched again
    cudaStream_t last_stream = nullptr;
    cudaEvent_t ev = nullptr;
};
constexpr int GATE_DEVICES = 64;
PersistGate g_gate[GATE_DEVICES];

PersistGate* gate_of_device(int dev) { return (dev >= 0 && dev < GATE_DEVICES) ? &g_gate[dev] : nullptr; }

ef21_status gate_order_after_last(PersistGate* G, cudaStream_t stream) {
    if (!G->any || (!G->detached && G->last_stream == stream)) return EF21_OK;
    if (!G->ev) CU(cudaEventCreateWithFlags(&G->ev, cudaEventDisableTiming));
    if (!G->detached) CU(cudaEventRecord(G->ev, G->last_stream));
    CU(cudaStreamWaitEvent(stream, G->ev, 0));
    return EF21_OK;
}

// Called when a handle goes away: its stream may be destroyed by the caller afterwards, so what it has enqueued is
// pinned to the event now.
void gate_forget_stream(int dev, cudaStream_t stream) {
    PersistGate* G = gate_of_device(dev);
    if (!G) return;
    std::lock_guard<std::mutex> lock(G->mu);
    if (!G->any || G->detached || G->last_stream != stream) return;
    if (!G->ev && cudaEventCreateWithFlags(&G->ev, cudaEventDisableTiming) != cudaSuccess) { cudaGetLastError(); G->any = false; return; }
    if (cudaEventRecord(G->ev, stream) != cudaSuccess) { cudaGetLastError(); G->any = false; return; }
    G->detached = true;
}

ef21_status run_persistent(ef21_ctx* c, const PersistPlan& P, int steps, const int* batch = nullptr, int tau = 0) {
    PersistGate* G = gate_of_device(c->device);
    std::unique_lock<std::mutex> gate_lock;
    if (G) {
        gate_lock = std::unique_lock<std::mutex>(G->mu);
        EF(gate_order_after_last(G, c->stream));
    }
    PersistParams p;
    p.batch = batch; p.tau = tau; p.ring_stages = P.stages;
    p.A = c->at<float>(c->L.A); p.y = c->at<float>(c->L.y); p.row_off = c->at<i64>(c->L.row_off);
    p.x = c->x(); p.g = c->g(); p.gi = c->gi(); p.msg_idx = c->msg_idx(); p.msg_val = c->msg_val();
    p.plus_choice = c->at<int>(c->L.plus_choice);
    p.slots = c->at<unsigned long long>(c->L.slots); p.status = c->status();
    p.n = c->n; p.d = (int)c->d; p.ld = (int)c->L.ld; p.k = c->k; p.C = P.C; p.steps = steps;
    p.objective = c->objective;
    p.slice_rows = 0; p.use_table = (!P.local && c->variant != EF21_VARIANT_EF21_PLUS && pk_use_table(c->n, (int)c->L.ld, c->k)) ? 1 : 0; p.gamma = c->gamma; p.lambda = c->lambda; p.inv_n = 1.0f / (float)c->n;
    // the epochs run on from launch to launch, so the slot array (cleared once, at creation) needs no clearing here
    p.spin_limit = c->spin_limit; p.epoch0 = c->pk_epoch; p.par0 = c->pk_par;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(c->n * P.C)); cfg.blockDim = dim3((unsigned)P.threads);
    cfg.dynamicSmemBytes = P.smem;
    cfg.stream = c->stream;
    // A plain cluster launch: that all n clusters fit on the device at once was checked with the
    // occupancy query when the plan was made.
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)(P.local ? c->n * P.C : P.C); attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, P.kernel, p);
    if (e != cudaSuccess) { cudaGetLastError(); return EF21_ERR_CUDA; }
    if (G) { G->any = true; G->detached = false; G->last_stream = c->stream; }
    c->launches += 1;
    if (!P.local) {           // (one cluster for all workers keeps its words in shared memory)
        c->pk_epoch = (unsigned)(((i64)c->pk_epoch + steps - 1) % 65535) + 1u;
        c->pk_par = (c->pk_par + (unsigned)steps) & 1u;
    }
    c->pk_used_cluster = P.C; c->pk_used_rb = P.rb; c->pk_used_src = P.src == PK_SRC_RING ? PK_SRC_GMEM : P.src; c->pk_used_threads = P.threads;
    c->pk_used_body = P.roles ? 1 : 2;
    c->pk_used_local = P.local ? 1 : 0; c->pk_used_stages = P.src == PK_SRC_RING ? P.stages : 0;
    return EF21_OK;
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------------------------

extern "C" {

const char* ef21_status_string(ef21_status s) {
    switch (s) {
        case EF21_OK: return "ok";
        case EF21_ERR_INVALID_ARG: return "invalid argument";
        case EF21_ERR_STATE: return "call order violated";
        case EF21_ERR_WORKSPACE: return "workspace too small or misaligned";
        case EF21_ERR_CUDA: return "CUDA runtime error";
        case EF21_ERR_TIMEOUT: return "bounded device wait expired";
        case EF21_ERR_NONFINITE: return "non-finite value";
        case EF21_ERR_UNSUPPORTED: return "shape not supported by the requested path";
    }
    return "unknown status";
}

size_t ef21_workspace_bytes(int32_t n, int64_t d, int32_t k, int64_t total_rows) {
    if (!valid_shape(n, d, k, total_rows)) return 0;
    return make_layout(n, d, k, total_rows).total;
}

ef21_status ef21_create(ef21_ctx** out, int32_t n, int64_t d, int32_t k, float gamma, float lambda,
                        int64_t total_rows, void* workspace_dev, size_t workspace_bytes, void* cuda_stream) {
    if (!out || !valid_shape(n, d, k, total_rows)) return EF21_ERR_INVALID_ARG;
    if (!(gamma > 0.f) || !std::isfinite(gamma) || !(lambda >= 0.f) || !std::isfinite(lambda)) return EF21_ERR_INVALID_ARG;
    if (!workspace_dev) return EF21_ERR_INVALID_ARG;
    Layout L = make_layout(n, d, k, total_rows);
    if (workspace_bytes < L.total || (reinterpret_cast<uintptr_t>(workspace_dev) % ALIGN) != 0) return EF21_ERR_WORKSPACE;
    ef21_ctx* c = new (std::nothrow) ef21_ctx();
    if (!c) return EF21_ERR_INVALID_ARG;
    c->n = n; c->d = d; c->k = k; c->gamma = gamma; c->lambda = lambda; c->N = total_rows;
    c->stream = reinterpret_cast<cudaStream_t>(cuda_stream);
    c->device = -1;
    if (cudaGetDevice(&c->device) != cudaSuccess) { cudaGetLastError(); c->device = -1; }
    c->ws = static_cast<char*>(workspace_dev);
    c->L = L;
    c->shards_loaded = false; c->inited = false; c->num_tiles = 0; c->worker_tiles = 0;
    c->path = EF21_PATH_AUTO; c->last_path = 0; c->launches = 0;
    c->pk_cluster = 0; c->pk_rb = 0; c->pk_src = -1; c->pk_threads = 0; c->agg_off_ready = false;
    c->pk_used_cluster = c->pk_used_rb = 0; c->pk_used_src = -1; c->pk_used_threads = 0;
    c->pk_used_local = c->pk_used_stages = 0;
    c->pk_body = 0; c->pk_used_body = 0; c->pk_epoch = 0u; c->pk_par = 0u; c->plan_valid = false; c->mb_plan_valid = false; c->mb_plan_tau = 0;
    c->spin_limit = 1u << 22;
    c->force_general_topk = false;
    c->variant = EF21_VARIANT_EF21;
    c->mb_tau = -1;
    c->objective = EF21_OBJECTIVE_LOGISTIC;
    c->aux_stream = nullptr; c->ev_fork = nullptr; c->ev_join = nullptr;
    // x, g, g_i and the messages lie one behind the other, the words that have to start at zero elsewhere are few
    Copies clear;
    clear.add(c->ws + L.status, 64, nullptr, 0, 64, 1);
    clear.add(c->ws + L.x, 1, nullptr, 0, 1, (i64)(L.topk - L.x) / 4);
    if (L.tk.fast) clear.add(c->ws + L.topk + L.tk.slow_count, 1, nullptr, 0, 1, 1);
    clear.add(c->ws + L.plus_choice, n, nullptr, 0, n, 1);
    clear.add(c->ws + L.slots, 1, nullptr, 0, 1, (i64)4 * n * k);
    const ef21_status e = clear.run(c->stream, &c->launches);
    if (e != EF21_OK) { delete c; return e; }
    *out = c;
    return EF21_OK;
}

void ef21_destroy(ef21_ctx* ctx) {
    if (!ctx) return;
    gate_forget_stream(ctx->device, ctx->stream);
    if (ctx->ev_fork) cudaEventDestroy(ctx->ev_fork);
    if (ctx->ev_join) cudaEventDestroy(ctx->ev_join);
    if (ctx->aux_stream) cudaStreamDestroy(ctx->aux_stream);
    if (ctx->iter_graph) cudaGraphExecDestroy(ctx->iter_graph);
    if (ctx->cap_stream) cudaStreamDestroy(ctx->cap_stream);
    delete ctx;
}

ef21_status ef21_load_shards(ef21_ctx* c, const float* A_dev, const float* y_dev, const int64_t* row_offsets_host) {
    if (!c || !row_offsets_host) return EF21_ERR_INVALID_ARG;
    if (c->N == 0) return EF21_ERR_STATE;
    if (!A_dev || !y_dev) return EF21_ERR_INVALID_ARG;
    const unsigned blocks = (unsigned)std::min<i64>(ceil_div(c->N * c->L.ld, 256), 148 * 16);
    CU(launch(pad_rows_kernel, dim3(blocks), 256, 0, c->stream, 1, A_dev, c->N, (int)c->d, (int)c->L.ld, c->at<float>(c->L.A)));
    c->launches += 1;
    CU(cudaGetLastError());
    CU(cudaMemcpyAsync(c->at<float>(c->L.y), y_dev, (size_t)c->N * 4, cudaMemcpyDeviceToDevice, c->stream));
    return finish_load(c, reinterpret_cast<const i64*>(row_offsets_host));
}

ef21_status ef21_load_shards_host(ef21_ctx* c, const float* A_host, const float* y_host, const int64_t* row_offsets_host) {
    if (!c || !row_offsets_host) return EF21_ERR_INVALID_ARG;
    if (c->N == 0) return EF21_ERR_STATE;
    if (!A_host || !y_host) return EF21_ERR_INVALID_ARG;
    // Host rows have pitch d; the device layout has pitch ld with zero padding.
    if (c->L.ld != c->d) CU(cudaMemsetAsync(c->at<float>(c->L.A), 0, (size_t)c->N * c->L.ld * 4, c->stream));
    CU(cudaMemcpy2DAsync(c->at<float>(c->L.A), (size_t)c->L.ld * 4, A_host, (size_t)c->d * 4, (size_t)c->d * 4,
                         (size_t)c->N, cudaMemcpyHostToDevice, c->stream));
    CU(cudaMemcpyAsync(c->at<float>(c->L.y), y_host, (size_t)c->N * 4, cudaMemcpyHostToDevice, c->stream));
    return finish_load(c, reinterpret_cast<const i64*>(row_offsets_host));
}

ef21_status ef21_set_x(ef21_ctx* c, const float* x0_dev) {
    if (!c || !x0_dev) return EF21_ERR_INVALID_ARG;
    Copies m;
    m.add(c->x(), c->d, x0_dev, c->d, c->d, 1);
    return m.run(c->stream, &c->launches);
}

ef21_status ef21_init(ef21_ctx* c, int32_t mode) {
    if (!c || mode < 0 || mode > 2) return EF21_ERR_INVALID_ARG;
    if (mode == EF21_INIT_ZERO) {
        EF(zero_state(c));
        c->inited = true;
        return EF21_OK;
    }
    if (!c->shards_loaded) return EF21_ERR_STATE;
    TcShape S;
    if (mode == EF21_INIT_COMPRESSED && agg_by_table(c) && select_can_form_grads(c, full_source(c), S)) {
        // three launches: the selection writes g_i whole, the aggregation g
        EF(launch_grad_tiles(c, full_source(c), false));
        EF(enqueue_grad_select(c, full_source(c), S, TC_PLAIN));
        EF(enqueue_round_aggregate(c, AGG_INIT));
        c->inited = true;
        return EF21_OK;
    }
    EF(enqueue_grads(c, false));
    return init_from(c, c->at<float>(c->L.grad), c->L.ld, mode);
}

ef21_status ef21_init_grads(ef21_ctx* c, const float* V_dev, int32_t mode) {
    if (!c || mode < 0 || mode > 2) return EF21_ERR_INVALID_ARG;
    if (mode != EF21_INIT_ZERO && !V_dev) return EF21_ERR_INVALID_ARG;
    return init_from(c, V_dev, c->d, mode);
}

// One iteration of ef21_step on the launch path, as plain kernel launches on the handle's stream.  The x update that opens the
// iteration has already been enqueued (or does not exist: Algorithm 4); xmode AGG_X_AFTER: the one of the next iteration is
// made by the kernel that updates g.  early: an iteration of the same call has been enqueued before (see grad_wide_kernel).
static ef21_status enqueue_launch_iteration(ef21_ctx* c, const GradSource& G, int xmode, bool early = false) {
    EF(launch_grad_tiles(c, G, false, early));
    TcShape S;
    if (c->variant != EF21_VARIANT_EF21_PLUS && select_can_form_grads(c, G, S)) {
        c->agg_off_ready = false;
        const bool ef = c->variant == EF21_VARIANT_EF;
        EF(enqueue_grad_select(c, G, S, ef ? TC_EF : TC_DIFF));
        return ef ? enqueue_aggregate_into(c, c->x(), -(1.0f / (float)c->n), AGG_X_KEEP) : enqueue_round_aggregate(c, xmode);
    }
    EF(launch_grad_finish(c, G));
    if (c->variant == EF21_VARIANT_EF) return enqueue_ef_round(c, c->at<float>(c->L.grad), c->L.ld);
    if (c->variant == EF21_VARIANT_EF21_PLUS) return enqueue_plus_round(c, c->at<float>(c->L.grad), c->L.ld, xmode);
    return enqueue_round(c, c->at<float>(c->L.grad), c->L.ld, xmode);
}

// `steps` launch-path iterations.  Short vectors make an iteration a fixed list of a few small kernels whose cost is their
// launches: the iterations before the last one are replayed as a CUDA graph captured once per handle and method.  Anything
// that stands in the way (the caller's stream is itself being captured, capture or instantiation fails) leaves the plain
// launches, which give the same results.
static ef21_status run_launch_iterations(ef21_ctx* c, int steps) {
    int done = 0;
    const bool graphable = c->d <= GRAPH_MAX_D && steps >= 3 && !c->iter_graph_off;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (c->variant != EF21_VARIANT_EF) EF(enqueue_x_update(c));
    if (graphable && cudaStreamIsCapturing(c->stream, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
        const int key = c->variant * 16 + c->objective;
        if (c->iter_graph && c->iter_graph_key != key) { cudaGraphExecDestroy(c->iter_graph); c->iter_graph = nullptr; }
        if (!c->iter_graph) {
            const i64 before = c->launches;
            cudaGraph_t graph = nullptr;
            // captured on a stream of the library's own (the caller's may be the legacy default stream, which
            // cannot be captured); the graph is then launched into the caller's stream
            bool ok = c->cap_stream || cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking) == cudaSuccess;
            ok = ok && cudaStreamBeginCapture(c->cap_stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
            if (ok) {
                cudaStream_t user_stream = c->stream;
                c->stream = c->cap_stream;
                const ef21_status st = enqueue_launch_iteration(c, full_source(c), AGG_X_AFTER);
                c->stream = user_stream;
                ok = cudaStreamEndCapture(c->cap_stream, &graph) == cudaSuccess && st == EF21_OK && graph != nullptr;
            }
            if (ok) ok = cudaGraphInstantiate(&c->iter_graph, graph, 0) == cudaSuccess;
            if (graph) cudaGraphDestroy(graph);
            c->iter_graph_launches = c->launches - before;
            c->launches = before;                         // the captured iteration has not run
            if (!ok) {
                cudaGetLastError();
                if (c->iter_graph) { cudaGraphExecDestroy(c->iter_graph); c->iter_graph = nullptr; }
                c->iter_graph_off = true;
            } else {
                c->iter_graph_key = key;
            }
        }
        if (c->iter_graph) {
            for (; done + 1 < steps; ++done) {
                CU(cudaGraphLaunch(c->iter_graph, c->stream));
                c->launches += c->iter_graph_launches;
            }
        }
    } else {
        cudaGetLastError();
    }
    for (; done < steps; ++done) EF(enqueue_launch_iteration(c, full_source(c), done + 1 < steps ? AGG_X_AFTER : AGG_X_KEEP, done > 0));
    c->last_path = EF21_PATH_LAUNCHES;
    return EF21_OK;
}

ef21_status ef21_step(ef21_ctx* c, int32_t steps) {
    if (!c || steps < 0) return EF21_ERR_INVALID_ARG;
    if (!c->shards_loaded || !c->inited) return EF21_ERR_STATE;
    if (steps == 0) return EF21_OK;
    if (c->path != EF21_PATH_LAUNCHES) {
        // planning asks the runtime several questions (attributes, occupancy of the cluster launch): once per
        // handle and setting, not once per call
        if (!c->plan_valid) { c->plan = plan_persistent(c); c->plan_valid = true; }
        const PersistPlan& P = c->plan;
        if (P.ok) {
            EF(run_persistent(c, P, steps));
            c->last_path = EF21_PATH_PERSISTENT;
            return EF21_OK;
        }
        if (c->path == EF21_PATH_PERSISTENT) return EF21_ERR_UNSUPPORTED;
    }
    return run_launch_iterations(c, steps);
}

ef21_status ef21_step_grads(ef21_ctx* c, const float* V_dev, int32_t steps) {
    if (!c || !V_dev || steps < 0) return EF21_ERR_INVALID_ARG;
    if (!c->inited) return EF21_ERR_STATE;
    if (c->variant == EF21_VARIANT_EF) {
        for (int t = 0; t < steps; ++t) EF(enqueue_ef_round(c, V_dev, c->d));
        c->last_path = EF21_PATH_LAUNCHES;
        return EF21_OK;
    }
    if (c->variant == EF21_VARIANT_EF21_PLUS) {
        for (int t = 0; t < steps; ++t) EF(enqueue_plus_round(c, V_dev, c->d, AGG_X_BEFORE));
        c->last_path = EF21_PATH_LAUNCHES;
        return EF21_OK;
    }
    const bool fast = long_topk(c);
    if (fast && steps > 1 && !c->aux_stream) {
        if (cudaStreamCreateWithFlags(&c->aux_stream, cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&c->ev_fork, cudaEventDisableTiming) != cudaSuccess ||
            cudaEventCreateWithFlags(&c->ev_join, cudaEventDisableTiming) != cudaSuccess) {
            cudaGetLastError();
            return EF21_ERR_CUDA;
        }
    }
    TopkBuffers B = topk_buffers(c->ws + c->L.topk, c->L.tk);
    if (!(fast && steps > 1)) {
        for (int t = 0; t < steps; ++t) {
            EF(enqueue_round(c, V_dev, c->d, AGG_X_BEFORE));
        }
        c->last_path = EF21_PATH_LAUNCHES;
        return EF21_OK;
    }
    // Same V at every step: the threshold estimate of round t+1 needs V and g_i^{t+1} only, so it runs beside the aggregation of
    // round t (g and x); the streaming pass of round t+1 waits for both.  The longer of the two follows the selection on
    // this stream, without an event in between: the aggregation where there are many message entries (64 x 4,194: 376.8 us a round
    // against 377.6, 24 x 40,000: 283 against 289), else the estimate (16 x 4,194: 125 against 135, 64 x 1,000: 121 against 125).
    cudaStream_t main_stream = c->stream;
    const bool agg_first = (i64)c->n * c->k > 131072;
    for (int t = 0; t < steps; ++t) {
        // (letting the streaming pass start while the aggregation still runs made the pass 15-20 % slower)
        if (t > 0) CU(cudaStreamWaitEvent(main_stream, c->ev_join, 0));
        EF(enqueue_round_select(c, V_dev, c->d, t > 0));
        if (t + 1 == steps) {
            EF(enqueue_round_aggregate(c, AGG_X_BEFORE));
            break;
        }
        CU(cudaEventRecord(c->ev_fork, main_stream));
        CU(cudaStreamWaitEvent(c->aux_stream, c->ev_fork, 0));
        const StArgs next = stream_args(V_dev, c->d, c->gi(), c->L.ld, 0.f, c->d, c->k, B);
        if (agg_first) {
            EF(enqueue_stream_sample<TC_DIFF>(c->aux_stream, next, c->n, B.L, &c->launches));
            EF(enqueue_round_aggregate(c, AGG_X_BEFORE));
        } else {
            c->stream = c->aux_stream;
            const ef21_status agg = enqueue_round_aggregate(c, AGG_X_BEFORE);
            c->stream = main_stream;
            EF(agg);
            EF(enqueue_stream_sample<TC_DIFF>(main_stream, next, c->n, B.L, &c->launches));
        }
        CU(cudaEventRecord(c->ev_join, c->aux_stream));
    }
    c->last_path = EF21_PATH_LAUNCHES;
    return EF21_OK;
}

ef21_status ef21_step_minibatches(ef21_ctx* c, const int32_t* batches_dev, int32_t tau, int32_t steps) {
    if (!c || !batches_dev || tau < 1 || steps < 0) return EF21_ERR_INVALID_ARG;
    if (!c->shards_loaded || !c->inited) return EF21_ERR_STATE;
    if (c->variant != EF21_VARIANT_EF21) return EF21_ERR_UNSUPPORTED;
    for (int i = 0; i < c->n; ++i)
        if (c->row_off[i + 1] - c->row_off[i] < tau) return EF21_ERR_INVALID_ARG;
    if (steps == 0) return EF21_OK;
    if (c->path != EF21_PATH_LAUNCHES && c->k <= PK_ROLES_MAX_K && c->pk_body != 2) {
        if (!c->mb_plan_valid || c->mb_plan_tau != tau) {
            c->mb_plan = plan_persistent_body(c, true, tau);
            c->mb_plan_tau = tau; c->mb_plan_valid = true;
        }
        if (c->mb_plan.ok) {
            EF(run_persistent(c, c->mb_plan, steps, batches_dev, tau));
            c->last_path = EF21_PATH_PERSISTENT;
            return EF21_OK;
        }
    }
    if (c->path == EF21_PATH_PERSISTENT) return EF21_ERR_UNSUPPORTED;
    EF(enqueue_x_update(c));
    for (int t = 0; t < steps; ++t) {
        GradSource G;
        EF(minibatch_source(c, batches_dev + (size_t)t * c->n * tau, tau, G));
        EF(enqueue_launch_iteration(c, G, t + 1 < steps ? AGG_X_AFTER : AGG_X_KEEP, t > 0));
    }
    c->last_path = EF21_PATH_LAUNCHES;
    return EF21_OK;
}

ef21_status ef21_step_minibatch(ef21_ctx* c, const int32_t* batch_dev, int32_t tau) {
    return ef21_step_minibatches(c, batch_dev, tau, 1);
}

ef21_status ef21_step_randk(ef21_ctx* c, const float* V_dev, const int32_t* sets_dev, int32_t steps) {
    if (!c || !sets_dev || steps < 0) return EF21_ERR_INVALID_ARG;
    if (!c->inited || (!V_dev && !c->shards_loaded)) return EF21_ERR_STATE;
    if (c->variant != EF21_VARIANT_EF21) return EF21_ERR_UNSUPPORTED;
    const i64 total = (i64)c->n * c->k;
    if (!V_dev && steps > 0) EF(enqueue_x_update(c));
    for (int t = 0; t < steps; ++t) {
        if (!V_dev) EF(enqueue_grads(c, false));
        const float* a = V_dev ? V_dev : c->at<float>(c->L.grad);
        const i64 pitch = V_dev ? c->d : c->L.ld;
        CU(launch(randk_select_kernel, dim3((unsigned)ceil_div(total, 256)), 256, 0, c->stream, 1,
            a, pitch, c->gi(), c->L.ld, sets_dev + (size_t)t * total, total, c->k, c->d, c->msg_idx(), c->msg_val(), c->status()));
        c->launches += 1;
        CU(cudaGetLastError());
        c->agg_off_ready = false;
        EF(enqueue_round_aggregate(c, V_dev ? AGG_X_BEFORE : (t + 1 < steps ? AGG_X_AFTER : AGG_X_KEEP)));
    }
    c->last_path = EF21_PATH_LAUNCHES;
    return EF21_OK;
}

ef21_status ef21_local_grads(ef21_ctx* c, float* grads_out_dev) {
    if (!c || !grads_out_dev) return EF21_ERR_INVALID_ARG;
    if (!c->shards_loaded) return EF21_ERR_STATE;
    EF(enqueue_grads(c, false));
    Copies m;
    m.add(grads_out_dev, c->d, c->at<float>(c->L.grad), c->L.ld, c->d, c->n);
    return m.run(c->stream, &c->launches);
}

size_t ef21_topk_workspace_bytes(int32_t batch, int64_t d, int32_t k) {
    if (batch < 1 || batch > 65535 || !valid_shape(1, d, k, 0)) return 0;
    TcShape S;
    if (tc_shape(batch, d, fast_topk_eligible(d, k), S)) return ALIGN;         // one launch, no scratch
    return topk_layout(batch, d, k).total;
}

ef21_status ef21_topk(const float* v_dev, int32_t batch, int64_t d, int32_t k, int32_t* idx_out_dev,
                      float* val_out_dev, void* workspace_dev, size_t workspace_bytes, void* cuda_stream) {
    if (!v_dev || !idx_out_dev || !val_out_dev || batch < 1 || batch > 65535 || !valid_shape(1, d, k, 0))
        return EF21_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
    TcShape S;
    const bool one_launch = tc_shape(batch, d, fast_topk_eligible(d, k), S);
    TopkLayout L{};
    if (one_launch) L.total = ALIGN; else L = topk_layout(batch, d, k);
    if (!workspace_dev || workspace_bytes < L.total || (reinterpret_cast<uintptr_t>(workspace_dev) % ALIGN) != 0)
        return EF21_ERR_WORKSPACE;
    if (one_launch)
        return enqueue_topk_cluster(st, TC_PLAIN, S, v_dev, d, nullptr, 0, 0.f, batch, d, k, idx_out_dev, val_out_dev, nullptr, 0, nullptr, nullptr);
    TopkBuffers B = topk_buffers(static_cast<char*>(workspace_dev), L);
    if (L.fast)
        return enqueue_topk_stream<TC_PLAIN>(st, v_dev, d, nullptr, 0, 0.f, batch, d, k,
                                             StOut{idx_out_dev, val_out_dev, nullptr, 0, nullptr, 0, nullptr, nullptr}, B, nullptr, false);
    return enqueue_topk_general(st, v_dev, d, nullptr, 0, batch, d, k, idx_out_dev, val_out_dev, B, nullptr, nullptr);
}

// ---------------------------------------------------------------------------------------------
// Top-k without any caller-provided or allocated scratch
// ---------------------------------------------------------------------------------------------
// Scratch of ef21_topk_static: lives in the library image, so every GPU that loads the library
// holds these bytes until the process exits.
constexpr size_t TOPK_STATIC_SCRATCH_BYTES = (size_t)1 << 20;
constexpr int TOPK_STATIC_MAX_BATCH = 64;
constexpr i64 TOPK_STATIC_MAX_CHUNKS = 16384;      // batch * ceil(d / 4096)
static __device__ __align__(256) unsigned char g_topk_static_scratch[TOPK_STATIC_SCRATCH_BYTES];

// Device address of the scratch array on the current device.  In host code the array's name is only
// a handle for the runtime, not an address a kernel could use, so the address is asked for once
// per device (with that device current) and cached.
static ef21_status topk_static_scratch(void** out) {
    constexpr int MAX_DEVICES = 64;
    static std::mutex mu;
    static void* addr[MAX_DEVICES] = {};
    int dev = -1;
    CU(cudaGetDevice(&dev));
    if (dev < 0 || dev >= MAX_DEVICES) return EF21_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void* p = nullptr;
        CU(cudaGetSymbolAddress(&p, g_topk_static_scratch));
        if (!p) return EF21_ERR_CUDA;
        addr[dev] = p;
    }
    *out = addr[dev];
    return EF21_OK;
}

ef21_status ef21_topk_static(const float* v_dev, int32_t batch, int64_t d, int32_t k, int32_t* idx_out_dev,
                             float* val_out_dev, void* cuda_stream) {
    if (!v_dev || !idx_out_dev || !val_out_dev || batch < 1 || !valid_shape(1, d, k, 0)) return EF21_ERR_INVALID_ARG;
    if (batch > TOPK_STATIC_MAX_BATCH || (i64)batch * ceil_div(d, TK_CHUNK) > TOPK_STATIC_MAX_CHUNKS)
        return EF21_ERR_UNSUPPORTED;                     // beyond the built-in scratch
    const TopkLayout L = topk_layout_general(batch, d);      // the same three sections ef21_topk lays out
    if (L.total > TOPK_STATIC_SCRATCH_BYTES) return EF21_ERR_UNSUPPORTED;
    void* scratch = nullptr;
    EF(topk_static_scratch(&scratch));
    TopkBuffers B = topk_buffers(static_cast<char*>(scratch), L);
    // tk_reset_kernel clears the selection state and the histograms of the vectors in use; the
    // per-chunk counts are fully rewritten before they are read.
    return enqueue_topk_general(reinterpret_cast<cudaStream_t>(cuda_stream), v_dev, d, nullptr, 0, batch, d, k,
                                idx_out_dev, val_out_dev, B, nullptr, nullptr);
}

ef21_status ef21_get_state(ef21_ctx* c, float* x_dev, float* g_dev, float* gi_dev, int32_t* last_idx_dev, float* last_val_dev) {
    if (!c) return EF21_ERR_INVALID_ARG;
    const i64 nk = (i64)c->n * c->k;
    Copies m;
    m.add(x_dev, c->d, c->x(), c->d, c->d, 1);
    m.add(g_dev, c->d, c->g(), c->d, c->d, 1);
    m.add(gi_dev, c->d, c->gi(), c->L.ld, c->d, c->n);
    m.add(last_idx_dev, nk, c->msg_idx(), nk, nk, 1);
    m.add(last_val_dev, nk, c->msg_val(), nk, nk, 1);
    return m.run(c->stream, &c->launches);
}

ef21_status ef21_get_state_host(ef21_ctx* c, float* x_host, float* g_host, float* gi_host, int32_t* last_idx_host, float* last_val_host) {
    if (!c) return EF21_ERR_INVALID_ARG;
    constexpr cudaMemcpyKind kind = cudaMemcpyDeviceToHost;
    if (x_host) CU(cudaMemcpyAsync(x_host, c->x(), (size_t)c->d * 4, kind, c->stream));
    if (g_host) CU(cudaMemcpyAsync(g_host, c->g(), (size_t)c->d * 4, kind, c->stream));
    if (gi_host) CU(cudaMemcpy2DAsync(gi_host, (size_t)c->d * 4, c->gi(), (size_t)c->L.ld * 4, (size_t)c->d * 4, (size_t)c->n, kind, c->stream));
    if (last_idx_host) CU(cudaMemcpyAsync(last_idx_host, c->msg_idx(), (size_t)c->n * c->k * 4, kind, c->stream));
    if (last_val_host) CU(cudaMemcpyAsync(last_val_host, c->msg_val(), (size_t)c->n * c->k * 4, kind, c->stream));
    CU(cudaStreamSynchronize(c->stream));
    return EF21_OK;
}

ef21_status ef21_set_state(ef21_ctx* c, const float* x_dev, const float* g_dev, const float* gi_dev) {
    if (!c) return EF21_ERR_INVALID_ARG;
    Copies m;
    if (x_dev) m.add(c->x(), c->d, x_dev, c->d, c->d, 1);
    if (g_dev) m.add(c->g(), c->d, g_dev, c->d, c->d, 1);
    if (gi_dev) m.add(c->gi(), c->L.ld, gi_dev, c->d, c->d, c->n);
    EF(m.run(c->stream, &c->launches));
    c->inited = true;
    return EF21_OK;
}

ef21_status ef21_eval(ef21_ctx* c, double* f, double* grad_norm2, double* G) {
    if (!c) return EF21_ERR_INVALID_ARG;
    if (!c->shards_loaded) return EF21_ERR_STATE;
    EF(enqueue_grads(c, true));
    CU(launch(eval_reduce_kernel, dim3(1), 1024, 0, c->stream, 1, c->at<double>(c->L.loss_partial), c->at<int>(c->L.tile_begin),
                                                  c->at<i64>(c->L.row_off), c->at<float>(c->L.grad), c->gi(), c->x(),
                                                  c->lambda, c->n, (int)c->d, (int)c->L.ld, c->at<double>(c->L.eval_out)));
    c->launches += 1;
    CU(cudaGetLastError());
    double out[3];
    CU(cudaMemcpyAsync(out, c->at<double>(c->L.eval_out), sizeof out, cudaMemcpyDeviceToHost, c->stream));
    CU(cudaStreamSynchronize(c->stream));
    if (f) *f = out[0];
    if (grad_norm2) *grad_norm2 = out[1];
    if (G) *G = out[2];
    if (!std::isfinite(out[0]) || !std::isfinite(out[1]) || !std::isfinite(out[2])) return EF21_ERR_NONFINITE;
    return EF21_OK;
}

ef21_status ef21_poll(ef21_ctx* c) {
    if (!c) return EF21_ERR_INVALID_ARG;
    unsigned word = 0;
    CU(cudaMemcpyAsync(&word, c->status(), 4, cudaMemcpyDeviceToHost, c->stream));
    CU(cudaStreamSynchronize(c->stream));
    if (word == 0) return EF21_OK;
    return word <= EF21_ERR_UNSUPPORTED ? (ef21_status)word : EF21_ERR_CUDA;
}

ef21_status ef21_set_path(ef21_ctx* c, int32_t path) {
    if (!c || path < EF21_PATH_AUTO || path > EF21_PATH_PERSISTENT) return EF21_ERR_INVALID_ARG;
    c->path = path;
    return EF21_OK;
}

ef21_status ef21_set_persistent_shape(ef21_ctx* c, int32_t cluster_blocks, int32_t rows_per_batch, int32_t row_source) {
    if (!c || cluster_blocks < 0 || cluster_blocks > 8) return EF21_ERR_INVALID_ARG;
    if (rows_per_batch != 0 && rows_per_batch != 4 && rows_per_batch != 8 && rows_per_batch != 16 && rows_per_batch != 32) return EF21_ERR_INVALID_ARG;
    if (row_source < -1 || row_source > 2) return EF21_ERR_INVALID_ARG;
    c->pk_cluster = cluster_blocks; c->pk_rb = rows_per_batch; c->pk_src = row_source;
    c->plan_valid = false; c->mb_plan_valid = false;
    return EF21_OK;
}

ef21_status ef21_set_persistent_threads(ef21_ctx* c, int32_t threads_per_block) {
    if (!c || (threads_per_block != 0 && threads_per_block != 256 && threads_per_block != 512)) return EF21_ERR_INVALID_ARG;
    c->pk_threads = threads_per_block;
    c->plan_valid = false; c->mb_plan_valid = false;
    return EF21_OK;
}

int32_t ef21_get_persistent_threads(const ef21_ctx* c) { return c ? c->pk_used_threads : 0; }

ef21_status ef21_set_persistent_body(ef21_ctx* c, int32_t body) {
    if (!c || body < 0 || body > 2) return EF21_ERR_INVALID_ARG;
    c->pk_body = body;
    c->plan_valid = false; c->mb_plan_valid = false;
    return EF21_OK;
}

int32_t ef21_get_persistent_body(const ef21_ctx* c) { return c ? c->pk_used_body : 0; }

ef21_status ef21_get_persistent_shape(const ef21_ctx* c, int32_t* cluster_blocks, int32_t* rows_per_batch, int32_t* row_source) {
    if (!c) return EF21_ERR_INVALID_ARG;
    if (cluster_blocks) *cluster_blocks = c->pk_used_cluster;
    if (rows_per_batch) *rows_per_batch = c->pk_used_rb;
    if (row_source) *row_source = c->pk_used_src;
    return EF21_OK;
}

ef21_status ef21_get_persistent_form(const ef21_ctx* c, int32_t* one_cluster, int32_t* ring_stages) {
    if (!c) return EF21_ERR_INVALID_ARG;
    if (one_cluster) *one_cluster = c->pk_used_local;
    if (ring_stages) *ring_stages = c->pk_used_stages;
    return EF21_OK;
}

ef21_status ef21_set_objective(ef21_ctx* c, int32_t objective) {
    if (!c || (objective != EF21_OBJECTIVE_LOGISTIC && objective != EF21_OBJECTIVE_LEAST_SQUARES)) return EF21_ERR_INVALID_ARG;
    c->objective = objective;
    return EF21_OK;
}

ef21_status ef21_set_variant(ef21_ctx* c, int32_t variant) {
    if (!c || variant < EF21_VARIANT_EF21 || variant > EF21_VARIANT_EF) return EF21_ERR_INVALID_ARG;
    c->variant = variant;
    c->plan_valid = false; c->mb_plan_valid = false;
    return EF21_OK;
}

ef21_status ef21_get_plus_choice(ef21_ctx* c, int32_t* choice_host) {
    if (!c || !choice_host) return EF21_ERR_INVALID_ARG;
    CU(cudaMemcpyAsync(choice_host, c->at<int>(c->L.plus_choice), (size_t)c->n * 4, cudaMemcpyDeviceToHost, c->stream));
    CU(cudaStreamSynchronize(c->stream));
    return EF21_OK;
}

ef21_status ef21_set_topk_algorithm(ef21_ctx* c, int32_t algorithm) {
    if (!c || algorithm < 0 || algorithm > 1) return EF21_ERR_INVALID_ARG;
    c->force_general_topk = algorithm == 1;
    return EF21_OK;
}

ef21_status ef21_fallback_count(ef21_ctx* c, int64_t* count) {
    if (!c || !count) return EF21_ERR_INVALID_ARG;
    unsigned v = 0;
    if (c->L.tk.fast) {
        CU(cudaMemcpyAsync(&v, c->ws + c->L.topk + c->L.tk.slow_count, 4, cudaMemcpyDeviceToHost, c->stream));
        CU(cudaStreamSynchronize(c->stream));
    }
    *count = (int64_t)v;
    return EF21_OK;
}

ef21_status ef21_clear_status(ef21_ctx* c) {
    if (!c) return EF21_ERR_INVALID_ARG;
    CU(cudaMemsetAsync(c->status(), 0, 256, c->stream));
    return EF21_OK;
}

ef21_status ef21_selftest_bounded_wait(ef21_ctx* c, uint32_t spin_limit) {
    if (!c || spin_limit == 0 || spin_limit > (1u << 24)) return EF21_ERR_INVALID_ARG;
    CU(cudaMemsetAsync(c->at<unsigned long long>(c->L.slots), 0, 8, c->stream));
    CU(launch(bounded_wait_selftest_kernel, dim3(1), 1, 0, c->stream, 1, c->at<unsigned long long>(c->L.slots), c->status(), spin_limit));
    c->launches += 1;
    // the gradient kernel of wide rows, as if its first wait had run out, with copies of rows under way (its partials are scratch)
    if (c->shards_loaded && grad_plan(c->L.ld).resident) EF(launch_grad_tiles(c, full_source(c), false, false, true));
    CU(cudaGetLastError());
    return EF21_OK;
}

ef21_status ef21_selftest_exchange_floor(ef21_ctx* c, int32_t steps) {
    if (!c || steps < 1) return EF21_ERR_INVALID_ARG;
    if (!c->shards_loaded || !c->inited) return EF21_ERR_STATE;
    if (c->variant != EF21_VARIANT_EF21) return EF21_ERR_UNSUPPORTED;
    // the shape ef21_step itself would launch, with the skeleton kernel of the same instantiation in its place
    PersistPlan P = plan_persistent(c);
    if (!P.ok) return EF21_ERR_UNSUPPORTED;
    const auto lookup = P.roles ? (P.local ? pk_lookup_local_floor : pk_lookup_floor) : (P.local ? pk_lookup_local_wide_floor : pk_lookup_wide_floor);
    P.kernel = lookup(P.chunks, P.rb, P.src, P.threads, P.extra);
    if (!P.kernel) return EF21_ERR_UNSUPPORTED;
    int dev = 0, max_smem = 0;
    CU(cudaGetDevice(&dev));
    CU(cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    CU(cudaFuncSetAttribute(P.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem - PK_STATIC_SMEM));
    if (P.local) CU(cudaFuncSetAttribute(P.kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    return run_persistent(c, P, steps);
}

int32_t ef21_last_path(const ef21_ctx* c) { return c ? c->last_path : 0; }
int64_t ef21_launch_count(const ef21_ctx* c) { return c ? c->launches : 0; }

}  // extern "C"
