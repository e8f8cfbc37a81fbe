// State updates of Algorithm 2 after the messages c_i = (idx, val)[k] are known:
//   g_i <- g_i + c_i                      (worker state, node loop)
//   g   <- g + (1/n) sum_i c_i            (master, last line of the loop)
//   x   <- x - gamma g                    (master, first line of the loop)
// The per-coordinate sum over workers runs in ascending worker index starting from 0, each
// operation a single rounded fp32 add / multiply, so the result does not depend on scheduling.
#pragma once
#include "common.cuh"

namespace ef21 {

constexpr int AGG_TILE = 2048;     // coordinates per block in the aggregation
constexpr int AGG_BLOCK = 256;

// g_i[idx] += val for all n*k message entries (indices within a worker are distinct).
__global__ void apply_messages_kernel(const int* __restrict__ idx, const float* __restrict__ val,
                                      i64 total, int k, i64 ld, float* __restrict__ gi) {
    pdl_trigger();
    pdl_wait(idx, val, gi);
    const i64 e = blockIdx.x * (i64)blockDim.x + threadIdx.x;
    if (e >= total) return;
    const i64 i = e / k;
    float* p = gi + i * ld + idx[e];
    *p = __fadd_rn(*p, val[e]);
}

// Scaled Rand-k (Appendix, Lemma 8 and Example 2: Rand-k times 1/(1 + omega) keeps the k sampled entries as they
// are): message entry t of worker i is (S, a[S] - g_i[S]) with S = sets[i][t], and g_i[S] takes the sum.  The sets are
// an input: k distinct indices in ascending order per worker.  An index outside [0, d), or one that does not exceed
// its predecessor, is reported through the status word and replaced by position t (never dereferenced as given).
__global__ void randk_select_kernel(const float* __restrict__ a, i64 pitch_a, float* __restrict__ gi, i64 ld,
                                    const int* __restrict__ sets, i64 total, int k, i64 d,
                                    int* __restrict__ idx_out, float* __restrict__ val_out, unsigned* status) {
    pdl_trigger();
    pdl_wait(a, gi, sets, idx_out, val_out, status);
    const i64 e = blockIdx.x * (i64)blockDim.x + threadIdx.x;
    if (e >= total) return;
    const i64 i = e / k;
    const int t = (int)(e - i * k);
    int j = sets[e];
    const bool bad = j < 0 || (i64)j >= d || (t > 0 && sets[e - 1] >= j);
    if (bad) { record_error(status, 1u /* EF21_ERR_INVALID_ARG */); j = t; }
    float* p = gi + i * ld + j;
    const float v = __fsub_rn(a[i * pitch_a + j], *p);
    idx_out[e] = j; val_out[e] = v;
    flag_nonfinite(status, v);
    *p = __fadd_rn(*p, v);
}

// off[i][b] = first position in worker i's ascending index list with idx >= b * AGG_TILE,
// for b = 0 .. ntiles (so tile b owns entries [off[i][b], off[i][b+1])).
__global__ void agg_offsets_kernel(const int* __restrict__ idx, int n, int k, int ntiles,
                                   int* __restrict__ off) {
    pdl_trigger();
    pdl_wait(idx, off);
    const i64 e = blockIdx.x * (i64)blockDim.x + threadIdx.x;
    const i64 total = (i64)n * (ntiles + 1);
    if (e >= total) return;
    const int i = (int)(e / (ntiles + 1));
    const int b = (int)(e - (i64)i * (ntiles + 1));
    const i64 bound = (i64)b * AGG_TILE;
    const int* __restrict__ ix = idx + (i64)i * k;
    int lo = 0, hi = k;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if ((i64)ix[mid] < bound) lo = mid + 1; else hi = mid;
    }
    off[e] = lo;
}

// What an aggregation does to x besides: nothing; x <- fma(-gamma, g^t, x) before g changes (Algorithm 2 updates x from g^t, then
// g^{t+1} from the messages); or the x update of the following iteration, from the new g.
// AGG_INIT (table kernel only): x stays, and g starts from zero.
enum { AGG_X_KEEP = 0, AGG_X_BEFORE = 1, AGG_X_AFTER = 2, AGG_INIT = 3 };

// One block per tile of AGG_TILE coordinates.
template <int XMODE>
__global__ void __launch_bounds__(AGG_BLOCK)
aggregate_kernel(const int* __restrict__ idx, const float* __restrict__ val, const int* __restrict__ off,
                 int n, int k, int ntiles, i64 d, float inv_n, float gamma,
                 float* __restrict__ g, float* __restrict__ x) {
    pdl_trigger();
    pdl_wait(idx, val, off, g, x);
    __shared__ float s[AGG_TILE];
    __shared__ unsigned char touched[AGG_TILE];
    const int b = blockIdx.x;
    const i64 j0 = (i64)b * AGG_TILE;
    for (int t = threadIdx.x; t < AGG_TILE; t += AGG_BLOCK) { s[t] = 0.f; touched[t] = 0; }
    __syncthreads();
    for (int i = 0; i < n; ++i) {
        const int lo = off[(i64)i * (ntiles + 1) + b], hi = off[(i64)i * (ntiles + 1) + b + 1];
        for (int e = lo + threadIdx.x; e < hi; e += AGG_BLOCK) {
            const int t = (int)((i64)idx[(i64)i * k + e] - j0);
            s[t] = __fadd_rn(s[t], val[(i64)i * k + e]);
            touched[t] = 1;
        }
        __syncthreads();
    }
    for (int t = threadIdx.x; t < AGG_TILE; t += AGG_BLOCK) {
        const i64 j = j0 + t;
        if (j >= d) break;
        if (XMODE == AGG_X_KEEP && !touched[t]) continue;
        const float old = g[j], now = touched[t] ? __fadd_rn(old, __fmul_rn(s[t], inv_n)) : old;
        if (XMODE != AGG_X_KEEP) x[j] = fmaf(-gamma, XMODE == AGG_X_BEFORE ? old : now, x[j]);
        if (touched[t]) g[j] = now;
    }
}

// The same aggregation with the tile's message entries first staged in shared memory (one
// parallel gather), so that the ordered pass over the workers touches shared memory only.
// Needs n <= AGG_STAGE_MAX_N; a tile with more than AGG_STAGE_CAP entries takes the direct loop.
// alone: nothing may be placed beside the blocks (no pdl_trigger), for handles whose rounds have a streaming pass.  A block takes 39 KB
// of shared memory, and an SM that never runs empty keeps that split: the streaming pass of the next round, two kernels further on, ran
// with an L1 too small for its loads in flight.  Calls of one round each, us a round, alone / not: 64 x 4,194,304 393 / 459,
// 64 x 1,000,000 121 / 158, 20 x 1,000,000 59 / 75, 1 x 25,000,000 141 / 161; with Algorithm 4 64 x 4,194,304 597 / 680.  Shorter vectors,
// whose selection is one kernel, lose the overlap: 20 x 200,000 62.2 / 61.3, 5 x 50,000 34.1 / 33.6.
constexpr int AGG_STAGE_MAX_N = 1024;
constexpr int AGG_STAGE_CAP = 3072;
constexpr int AGG_OWNER_SCAN_MAX = 512;   // tiles with at most this many entries skip the per-worker loop

template <int XMODE>
__global__ void __launch_bounds__(AGG_BLOCK)
aggregate_staged_kernel(const int* __restrict__ idx, const float* __restrict__ val, const int* __restrict__ off,
                        int n, int k, int ntiles, i64 d, float inv_n, float gamma,
                        float* __restrict__ g, float* __restrict__ x, int alone) {
    if (!alone) pdl_trigger();
    pdl_wait(idx, val, off, g, x);
    __shared__ float s[AGG_TILE];
    __shared__ __align__(4) unsigned short touched[AGG_TILE];   // staged entries per coordinate
    __shared__ int w_start[AGG_STAGE_MAX_N + 1];
    __shared__ int w_lo[AGG_STAGE_MAX_N];
    __shared__ unsigned short e_idx[AGG_STAGE_CAP];
    __shared__ float e_val[AGG_STAGE_CAP];
    __shared__ unsigned scratch[33];
    __shared__ unsigned short multi[AGG_OWNER_SCAN_MAX];
    __shared__ unsigned n_multi;
    const int b = blockIdx.x;
    const i64 j0 = (i64)b * AGG_TILE;
    for (int t = threadIdx.x; t < AGG_TILE; t += AGG_BLOCK) { s[t] = 0.f; touched[t] = 0; }
    if (threadIdx.x == 0) n_multi = 0u;
    unsigned base = 0u;
    for (int c0 = 0; c0 < n; c0 += AGG_BLOCK) {
        const int i = c0 + threadIdx.x;
        int lo = 0, hi = 0;
        if (i < n) { lo = off[(i64)i * (ntiles + 1) + b]; hi = off[(i64)i * (ntiles + 1) + b + 1]; }
        unsigned tot;
        const unsigned pre = block_excl_scan((unsigned)(hi - lo), scratch, tot);
        if (i < n) { w_start[i] = (int)(base + pre); w_lo[i] = lo; }
        base += tot;
    }
    if (threadIdx.x == 0) w_start[n] = (int)base;
    __syncthreads();
    const int total = (int)base;
    if (total <= AGG_STAGE_CAP) {
        for (int e = threadIdx.x; e < total; e += AGG_BLOCK) {
            int lo = 0, hi = n;                      // last worker i with w_start[i] <= e
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (w_start[mid] <= e) lo = mid; else hi = mid;
            }
            const i64 src = (i64)lo * k + w_lo[lo] + (e - w_start[lo]);
            e_idx[e] = (unsigned short)((i64)idx[src] - j0);
            e_val[e] = val[src];
        }
        __syncthreads();
        if (total <= AGG_OWNER_SCAN_MAX) {
            // Few entries: count the entries per coordinate (16-bit counters, two per word).
            unsigned* cnt32 = reinterpret_cast<unsigned*>(touched);
            for (int e = threadIdx.x; e < total; e += AGG_BLOCK) {
                const int t = e_idx[e];
                atomicAdd(&cnt32[t >> 1], (t & 1) ? 0x10000u : 1u);
            }
            __syncthreads();
            // coordinates hit once: the entry is the sum; entries of coordinates hit several times go
            // to a short list and are resolved by whole warps below, in staged (= worker) order
            for (int e = threadIdx.x; e < total; e += AGG_BLOCK) {
                const int t = e_idx[e];
                if (touched[t] == 1) s[t] = __fadd_rn(0.f, e_val[e]);
                else { const unsigned q = atomicAdd(&n_multi, 1u); multi[q] = (unsigned short)e; }
            }
            __syncthreads();
            const int nm = (int)n_multi;                 // <= total <= AGG_OWNER_SCAN_MAX
            const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
            // Many such entries and few workers: worker by worker instead, a barrier each.  (A look through the list costs a warp about 45
            // cycles per 32 entries, a worker about 70; 20 workers with 410 entries in a tile, 90 of them on shared coordinates:
            // 21.7 us for the kernel by looking, 9.8 worker by worker.)
            const bool by_worker = nm * total > 400 * n;
            if (by_worker) {
                for (int i = 0; i < n; ++i) {
                    for (int e = w_start[i] + threadIdx.x; e < w_start[i + 1]; e += AGG_BLOCK) {
                        const int t = e_idx[e];
                        if (touched[t] != 1) s[t] = __fadd_rn(s[t], e_val[e]);
                    }
                    __syncthreads();
                }
            }
            for (int q = by_worker ? nm : warp; q < nm; q += AGG_BLOCK / 32) {
                const int e = multi[q];
                const int t = e_idx[e];
                float acc = 0.f; bool owner = true, seen = false;
                for (int base2 = 0; base2 < total; base2 += 32) {
                    const int p = base2 + lane;
                    unsigned m = __ballot_sync(0xffffffffu, p < total && e_idx[p] == t);
                    if (m && !seen) { owner = (base2 + __ffs(m) - 1) == e; seen = true; }
                    if (!owner) break;                       // warp-uniform
                    while (m) { const int bit = __ffs(m) - 1; acc = __fadd_rn(acc, e_val[base2 + bit]); m &= m - 1; }
                }
                if (owner && lane == 0) s[t] = acc;
            }
            __syncthreads();
        } else
        for (int i = 0; i < n; ++i) {
            const int lo = w_start[i], hi = w_start[i + 1];
            if (lo == hi) continue;                  // uniform: read from shared memory
            for (int e = lo + threadIdx.x; e < hi; e += AGG_BLOCK) {
                const int t = e_idx[e];
                s[t] = __fadd_rn(s[t], e_val[e]);
                touched[t] = 1;
            }
            __syncthreads();
        }
    } else {
        for (int i = 0; i < n; ++i) {
            const int lo = w_lo[i], hi = lo + (w_start[i + 1] - w_start[i]);
            for (int e = lo + threadIdx.x; e < hi; e += AGG_BLOCK) {
                const int t = (int)((i64)idx[(i64)i * k + e] - j0);
                s[t] = __fadd_rn(s[t], val[(i64)i * k + e]);
                touched[t] = 1;
            }
            __syncthreads();
        }
    }
    // dense part of the tile: all loads first, then the updates
    constexpr int PER = AGG_TILE / AGG_BLOCK;
    float gv[PER], xv[PER];
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int t = u * AGG_BLOCK + threadIdx.x;
        const i64 j = j0 + t;
        gv[u] = 0.f; xv[u] = 0.f;
        if (j < d && (XMODE != AGG_X_KEEP || touched[t])) gv[u] = g[j];
        if (XMODE != AGG_X_KEEP && j < d) xv[u] = x[j];
    }
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int t = u * AGG_BLOCK + threadIdx.x;
        const i64 j = j0 + t;
        if (j >= d) continue;
        const float now = touched[t] ? __fadd_rn(gv[u], __fmul_rn(s[t], inv_n)) : gv[u];
        if (XMODE != AGG_X_KEEP) x[j] = fmaf(-gamma, XMODE == AGG_X_BEFORE ? gv[u] : now, xv[u]);
        if (touched[t]) g[j] = now;
    }
}

// Short vectors: a block of AGG_TABLE_COLS coordinates scatters the messages that fall on them into a table [n][columns] in shared
// memory and every thread adds up its column, workers ascending.  No tile offsets are needed, and the ordered sum is one
// read per worker (20 workers, d = 5,001, Top-50: 3 us against 4 + 19 us for the offsets and the staged kernel).  Every block
// goes through all n * k messages, hence only for few of them.
constexpr int AGG_TABLE_COLS = 128;
constexpr i64 AGG_TABLE_MAX_D = 16384, AGG_TABLE_MAX_MESSAGES = 65536;
constexpr int AGG_TABLE_MAX_N = 400;                       // 200 KB of shared memory
constexpr unsigned AGG_NO_ENTRY = 0xffffffffu;             // cell without a message (a NaN pattern no finite value has)

template <int XMODE>
__global__ void __launch_bounds__(AGG_BLOCK)
aggregate_table_kernel(const int* __restrict__ idx, const float* __restrict__ val, int n, int k, int d, float inv_n, float gamma,
                       float* __restrict__ g, float* __restrict__ x) {
    extern __shared__ __align__(16) unsigned agg_table[];                 // [n][AGG_TABLE_COLS]
    for (int e = threadIdx.x; e < n * (AGG_TABLE_COLS / 4); e += AGG_BLOCK)
        reinterpret_cast<uint4*>(agg_table)[e] = make_uint4(AGG_NO_ENTRY, AGG_NO_ENTRY, AGG_NO_ENTRY, AGG_NO_ENTRY);
    __syncthreads();
    pdl_trigger();
    pdl_wait(idx, val, g, x);
    const int j0 = blockIdx.x * AGG_TABLE_COLS, total = n * k;
    const unsigned magic = (unsigned)(((1ull << 32) + (unsigned)k - 1u) / (unsigned)k);      // e / k for e < 65,536: one high product
    constexpr int U = 4;
#pragma unroll 1
    for (int e0 = threadIdx.x; e0 < total; e0 += U * AGG_BLOCK) {
        int c[U];
#pragma unroll
        for (int u = 0; u < U; ++u) { const int e = e0 + u * AGG_BLOCK; c[u] = e < total ? idx[e] - j0 : -1; }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if ((unsigned)c[u] < (unsigned)AGG_TABLE_COLS) {
                const int e = e0 + u * AGG_BLOCK;
                const unsigned i = k == 1 ? (unsigned)e : __umulhi((unsigned)e, magic);
                agg_table[i * AGG_TABLE_COLS + c[u]] = __float_as_uint(val[e]);
            }
    }
    __syncthreads();
    const int t = threadIdx.x, j = j0 + t;
    if (t >= AGG_TABLE_COLS || j >= d) return;
    constexpr bool MOVE_X = XMODE == AGG_X_BEFORE || XMODE == AGG_X_AFTER;
    const float old = XMODE == AGG_INIT ? 0.f : g[j], xj = MOVE_X ? x[j] : 0.f;
    float s = 0.f; bool hit = false;
#pragma unroll 8
    for (int i = 0; i < n; ++i) {
        const unsigned w = agg_table[i * AGG_TABLE_COLS + t];
        const float sum = __fadd_rn(s, __uint_as_float(w));
        if (w != AGG_NO_ENTRY) { s = sum; hit = true; }
    }
    const float now = hit ? __fadd_rn(old, __fmul_rn(s, inv_n)) : old;
    if (MOVE_X) x[j] = fmaf(-gamma, XMODE == AGG_X_BEFORE ? old : now, xj);
    if (hit || XMODE == AGG_INIT) g[j] = now;
}

// x <- fma(-gamma, g, x), elementwise.
__global__ void x_update_kernel(const float* __restrict__ g, float* __restrict__ x, i64 d, float gamma) {
    pdl_trigger();
    pdl_wait(g, x);
    for (i64 j = blockIdx.x * (i64)blockDim.x + threadIdx.x; j < d; j += (i64)gridDim.x * blockDim.x)
        x[j] = fmaf(-gamma, g[j], x[j]);
}

// Dense initial state g_i^0 = V_i, g^0_j = ((0 + V_0j) + V_1j + ...) * (1/n): the k = d message
// round applied to zero state.
__global__ void dense_init_kernel(const float* __restrict__ V, i64 pitch_v, int n, i64 d, i64 ld,
                                  float inv_n, float* __restrict__ gi, float* __restrict__ g) {
    pdl_trigger();
    pdl_wait(V, gi, g);
    for (i64 j = blockIdx.x * (i64)blockDim.x + threadIdx.x; j < d; j += (i64)gridDim.x * blockDim.x) {
        float s = 0.f;
        for (int i = 0; i < n; ++i) {
            const float v = V[(i64)i * pitch_v + j];
            gi[(i64)i * ld + j] = __fadd_rn(0.f, v);
            s = __fadd_rn(s, v);
        }
        g[j] = __fadd_rn(0.f, __fmul_rn(s, inv_n));
    }
}

}  // namespace ef21
