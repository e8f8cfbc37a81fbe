// Exact Top-k of long vectors from ONE pass over HBM: v = a - b is formed on the fly and read once.
//
//   1. st_sample_kernel: a cluster per vector histograms a sample of the magnitude keys and brackets the k-th largest key:
//      about k - 4.5 sigma entries of the whole vector are expected above `hi` and k + 4.5 sigma above `lo`.
//   2. st_collect_kernel: the streaming pass.  A warp owns a region of 1,024 or 4,096 consecutive entries and lists those with
//      key >= lo in index order (ballot ranks); a record is (index, v, b + v), so the updated state value travels with the
//      candidate.  Entries with key >= hi are in the message for sure and only counted; those in between ("open" ones) also go
//      to a list of the vector and into a histogram of 2,048 steps of [lo, hi).  (Large batches: st_collect_long_kernel only
//      lists, and st_cut_kernel tells the sure entries from the open ones.)  st_cut_kernel, a cluster per vector, finds the
//      exact cut from that histogram and list -- a composite of key and index, so ties at the k-th key go to the lower
//      index -- and the position in the message at which every region's entries begin.
//   3. st_compact_kernel: eight lanes per region write the selected entries to their places, store b + v (Algorithm 4: zero)
//      on the selected coordinates and, on request, where each tile of coordinates begins in the message.  A region with more
//      candidates than its list holds is read again; where more than a tenth of the entries are wanted no lists are kept
//      (st_reread_kernel).
//   4. tc_topk_kernel<..., true> (topk_cluster.cuh) redoes, exactly and without any estimate, the vectors whose bracket missed
//      the k-th key or whose open list overflowed (masses of ties, fewer than k non-zeros); for the others it returns at once.
// The bracket only decides speed, never the result.
//
// What bounds it: HBM in step 2 (64 vectors of 4 million entries: 306 us, 7.0 TB/s of reading); steps 1 and 3 are a few
// microseconds each and take no part of a vector's length.
#pragma once
#include <cooperative_groups.h>

#include "common.cuh"
#include "topk_cluster.cuh"

namespace ef21 {

// Entries per region (one warp's share of the streaming pass): 4,096 for large batches, 1,024 below 2^26 entries in total,
// where longer regions would leave too few warps with loads in flight (1 x 4,194,304 entries: 24 us against 9).
constexpr int ST_REGION_LOG_LARGE = 12, ST_REGION_LOG_SMALL = 10;
constexpr i64 ST_LARGE_TOTAL = (i64)1 << 26;
constexpr int ST_WARPS = 8;             // regions per block of the streaming pass
constexpr int ST_SAMPLE_THREADS = 1024;
constexpr int ST_SAMPLE_STEPS = 1024;   // steps of the sampled range
constexpr int ST_OPEN_BINS = 2048;
constexpr int ST_OPEN_STAGE = 8192;     // open entries of the deciding step that are ranked in shared memory
constexpr int ST_BLOCK_OPEN = 2048;     // open entries a block of the streaming pass gathers before they go to the list
constexpr int ST_GATHER = 160;          // a warp's buffer for candidates: emptied from 32 on, after at most 128 more
constexpr i64 ST_MIN_D = 131072;        // shorter vectors go to a cluster each, however many there are

// Per vector: the bracket, the counters of the streaming pass, the exact cut.
struct StCtl {
    unsigned lo, hi, shift;             // open entries: lo <= key < hi; histogram step of 2^shift
    unsigned sure, open;                // entries >= hi, open entries
    unsigned slow;                      // 1: the exact kernel redoes this vector
    unsigned pad[2];
    unsigned long long cut;             // selected: (key << 32 | ~index) >= cut
    unsigned long long pad2[3];
};

struct StArgs {
    const float* a; i64 pitch_a;
    float* b; i64 pitch_b;
    i64 d; int k, nreg, nreg_pitch, region_log, cap;    // nreg_pitch: nreg rounded up to 8; cap: records per region (0: regions are always read again)
    unsigned open_cap;
    float gamma;
    int pair;                           // TC_PAIR: vectors in each half of the batch
    StCtl* ctl;                         // [batch]
    unsigned* open_hist;                // [batch][ST_OPEN_BINS]
    unsigned long long* open_list;      // [batch][open_cap]
    unsigned* reg_cand;                 // [batch][nreg_pitch] candidates of a region
    unsigned* reg_base;                 // [batch][nreg_pitch] selected entries, then their first position in the message
    int4* cand;                         // [batch][nreg][cap]
    unsigned* slow_count;               // may be null
};

__device__ __forceinline__ unsigned long long st_composite(unsigned key, unsigned idx) {
    return ((unsigned long long)key << 32) | (unsigned long long)(0xffffffffu - idx);
}

template <int MODE>
__device__ __forceinline__ float st_value(float a, float b, float gamma) {
    return MODE == TC_DIFF || MODE == TC_PAIR ? __fsub_rn(a, b) : (MODE == TC_EF ? __fadd_rn(b, __fmul_rn(gamma, a)) : a);
}

// ---- 1. bracket ---------------------------------------------------------------------------------
// One cluster of C blocks per vector; PT * 1024 * C samples in runs of 32 consecutive entries, all loads issued at once.
// The first eight samples of every thread give a floor under which nothing matters for the bracket (twice the rank and six
// standard deviations) and the largest magnitude; the range from floor to maximum is then counted in 1,024 even steps of the
// key, so that the bracket is placed to a few tenths of a percent whatever the distribution, and only the few samples above
// the floor go through shared-memory atomics.
template <int MODE, int C, int PT>
__global__ void __launch_bounds__(ST_SAMPLE_THREADS)
st_sample_kernel(const __grid_constant__ StArgs p, float rank, float margin) {
    namespace cg = cooperative_groups;
    __shared__ __align__(16) unsigned coarse[2048];
    __shared__ unsigned fine[ST_SAMPLE_STEPS];
    __shared__ unsigned scratch[33], floor_key, top_key, bounds[2];
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, rk = (int)cluster.block_rank(), vec = (int)(blockIdx.x / (unsigned)C);
    coarse[tid] = 0u; coarse[tid + 1024] = 0u; fine[tid] = 0u;
    if (tid == 0) { floor_key = 0x7f800000u; top_key = 0u; bounds[0] = 1u; bounds[1] = 0x80000000u; }
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");       // block 0's words are ready
    pdl_trigger();
    pdl_wait();
    const bool second = MODE == TC_PAIR && vec >= p.pair;
    const float* __restrict__ av = pdl_ptr(p.a + (i64)(second ? vec - p.pair : vec) * p.pitch_a);
    const float* __restrict__ bv = MODE == TC_PLAIN ? nullptr : pdl_ptr(p.b + (i64)(second ? 0 : vec) * p.pitch_b);
    const int warps = C * (ST_SAMPLE_THREADS / 32), w = rk * (ST_SAMPLE_THREADS / 32) + (tid >> 5);
    const i64 stride = p.d / ((i64)warps * PT);                     // >= 32: a quarter of the vector at most is sampled
    unsigned key[PT];
#pragma unroll
    for (int s = 0; s < PT; ++s) {
        const i64 j = ((i64)s * warps + w) * stride + lane;
        key[s] = mag_key(second ? av[j] : st_value<MODE>(av[j], MODE == TC_PLAIN ? 0.f : bv[j], p.gamma));
    }
    // open histogram of this vector, for the streaming pass
    for (int q = rk * ST_SAMPLE_THREADS + tid; q < ST_OPEN_BINS; q += C * ST_SAMPLE_THREADS) p.open_hist[(i64)vec * ST_OPEN_BINS + q] = 0u;
#pragma unroll
    for (int s = 0; s < 8; ++s) if (key[s] >> 20) atomicAdd(&coarse[key[s] >> 20], 1u);
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    {
        const float r8 = rank * 8.f / (float)(PT * C);
        const unsigned want = (unsigned)(2.f * r8 + 6.f * sqrtf(r8) + 32.f);
        const int b1 = 2047 - 2 * tid;                              // thread t owns the bins b1 and b1 - 1
        const unsigned c1 = coarse[b1], c0 = coarse[b1 - 1];
        unsigned total;
        const unsigned up = block_excl_scan(c1 + c0, scratch, total);
        if (c1 + c0 != 0u) {
            if (up == 0u) atomicMax(cluster.map_shared_rank(&top_key, 0), (unsigned)((c1 ? b1 : b1 - 1) + 1) << 20);
            if (up < want && want <= up + c1 + c0) atomicMin(cluster.map_shared_rank(&floor_key, 0), (unsigned)max(1, (b1 - 1) << 20));
        }
        if (tid == 0 && total < want) atomicMin(cluster.map_shared_rank(&floor_key, 0), 1u);
    }
    cluster.sync();
    const unsigned lowest = *cluster.map_shared_rank(&floor_key, 0), highest = max(*cluster.map_shared_rank(&top_key, 0), lowest + 1u);
    unsigned sh = 0u;
    while (((highest - 1u - lowest) >> sh) >= (unsigned)ST_SAMPLE_STEPS) ++sh;
#pragma unroll
    for (int s = 0; s < PT; ++s) if (key[s] >= lowest) atomicAdd(&fine[min((key[s] - lowest) >> sh, (unsigned)ST_SAMPLE_STEPS - 1u)], 1u);
    __syncthreads();
    if (rk != 0) {
        const unsigned c = fine[tid];
        if (c) atomicAdd(cluster.map_shared_rank(fine, 0) + tid, c);
    }
    cluster.sync();
    if (rk != 0) return;
    // lo: lower end of the step that holds the (rank + margin)-th largest sample; hi: upper end of that of the (rank - margin)-th
    const int step = ST_SAMPLE_STEPS - 1 - tid;
    const unsigned n = fine[step];
    unsigned total;
    const float up = (float)block_excl_scan(n, scratch, total), to = up + (float)n;
    if (up < rank + margin && rank + margin <= to) bounds[0] = lowest + ((unsigned)step << sh);
    if (rank - margin >= 1.f && up < rank - margin && rank - margin <= to && tid > 0) bounds[1] = lowest + ((unsigned)(step + 1) << sh);
    __syncthreads();
    if (tid == 0) {
        StCtl& ct = p.ctl[vec];
        const unsigned lo = max(bounds[0], 1u), hi = max(bounds[1], lo + 1u);
        const unsigned span = hi - lo;
        unsigned shift = 0u;
        while ((span >> shift) >= (unsigned)ST_OPEN_BINS) ++shift;
        ct.lo = lo; ct.hi = hi; ct.shift = shift; ct.sure = 0u; ct.open = 0u; ct.slow = 0u; ct.cut = 0ull;
    }
}

// ---- 2. streaming pass --------------------------------------------------------------------------
// The streaming pass for large batches of aligned rows, regions of 4,096 entries, one warp each; grid = (ceil(nreg / 8), batch).
// HBM bounds it.  The loop only lists candidates; four 16-byte loads per array are in flight per lane (64-68 registers, no spills,
// three or four blocks per SM).  64 x 4,194,304 entries, V and g_i: 306 us, 7.0 TB/s; one load per array and eight blocks of 32
// registers, which spilt, 331 us (a round 393 -> 379, of Algorithm 4 597 -> 564); two loads and five blocks 313.  (With the open
// entries counted on the way, or behind the loop, where a warp stops streaming, the pass takes longer; st_cut_kernel<C, true>
// counts them.)
constexpr int ST_LONG_LOADS = 4, ST_LONG_BLOCKS = 3;

template <int MODE>
__global__ void __launch_bounds__(ST_WARPS * 32, ST_LONG_BLOCKS)
st_collect_long_kernel(const __grid_constant__ StArgs p) {
    constexpr int U = ST_LONG_LOADS, REGION = 1 << ST_REGION_LOG_LARGE;
    pdl_trigger();
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int vec = blockIdx.y, region = blockIdx.x * ST_WARPS + (threadIdx.x >> 5);
    if (region >= p.nreg) return;
    const unsigned lo = p.ctl[vec].lo;
    const int first = region << ST_REGION_LOG_LARGE, end = (int)min((i64)REGION, p.d - first);    // positions below are relative to `first`
    const float* __restrict__ av = pdl_ptr(p.a + (i64)vec * p.pitch_a + first);
    float* bv = MODE == TC_PLAIN ? nullptr : pdl_ptr(p.b + (i64)vec * p.pitch_b + first);
    int4* out = p.cand + ((i64)vec * p.nreg + region) * p.cap;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    int cnt = 0;
    auto form = [&](float4 x, const float4& g) {
        x.x = st_value<MODE>(x.x, g.x, p.gamma); x.y = st_value<MODE>(x.y, g.y, p.gamma);
        x.z = st_value<MODE>(x.z, g.z, p.gamma); x.w = st_value<MODE>(x.w, g.w, p.gamma);
        return x;
    };
    // the candidates among 128 entries, four consecutive ones (from j0 on) per lane
    auto list = [&](int j0, const float4& x, const float4& g) {
        const float v[4] = {x.x, x.y, x.z, x.w}, old[4] = {g.x, g.y, g.z, g.w};
        bool pr[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) pr[e] = mag_key(v[e]) >= lo;       // lo >= 1: the zeros behind the end never are
        if (__any_sync(0xffffffffu, pr[0] | pr[1] | pr[2] | pr[3])) {
            const unsigned lt = (1u << lane) - 1u;
            int pos = cnt;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const unsigned bm = __ballot_sync(0xffffffffu, pr[e]);
                pos += __popc(bm & lt); cnt += __popc(bm);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (pr[e]) {
                    if (pos < p.cap) out[pos] = make_int4(first + j0 + e, __float_as_int(v[e]), __float_as_int(__fadd_rn(old[e], v[e])), 0);
                    ++pos;
                }
        }
    };
    if (end == REGION) {
#pragma unroll 1
        for (int j0 = 4 * lane; j0 < REGION; j0 += 128 * U) {
            float4 x[U], g[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                x[u] = __ldcs(reinterpret_cast<const float4*>(av + j0 + 128 * u));
                g[u] = MODE == TC_PLAIN ? zero : __ldcs(reinterpret_cast<const float4*>(bv + j0 + 128 * u));
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                x[u] = form(x[u], g[u]);
                if (MODE == TC_EF) __stcs(reinterpret_cast<float4*>(bv + j0 + 128 * u), x[u]);
                list(j0 + 128 * u, x[u], g[u]);
            }
        }
    } else {
        // the last region of a vector whose length is no multiple of 4,096
#pragma unroll 1
        for (int j0 = 4 * lane; j0 - 4 * lane < end; j0 += 128) {
            const int left = end - j0;
            float4 x = zero, g = zero;
            if (left > 0) { x.x = av[j0]; if (MODE != TC_PLAIN) g.x = bv[j0]; }
            if (left > 1) { x.y = av[j0 + 1]; if (MODE != TC_PLAIN) g.y = bv[j0 + 1]; }
            if (left > 2) { x.z = av[j0 + 2]; if (MODE != TC_PLAIN) g.z = bv[j0 + 2]; }
            if (left > 3) { x.w = av[j0 + 3]; if (MODE != TC_PLAIN) g.w = bv[j0 + 3]; }
            x = form(x, g);
            if (MODE == TC_EF) {
                if (left > 0) bv[j0] = x.x;
                if (left > 1) bv[j0 + 1] = x.y;
                if (left > 2) bv[j0 + 2] = x.z;
                if (left > 3) bv[j0 + 3] = x.w;
            }
            list(j0, x, g);
        }
    }
    if (lane == 0) p.reg_cand[(i64)vec * p.nreg_pitch + region] = (unsigned)cnt;
}

// The streaming pass for everything else: grid = (blocks per vector, batch), 256 threads, one warp per region, in turn.  VEC: both
// rows 16-byte aligned.  U loads per array are in flight per lane: short regions and 4-byte loads (rows of odd length) need
// more of them and leave room for four blocks per SM.
// LISTS: candidates are listed (else every region is read again, the sure entries are only counted and the open ones gathered).
// Short of HBM it is the number of instructions that bounds it, above all of those that few lanes take part in: candidates go to a
// buffer in shared memory, and whenever it holds 32 of them the lanes write and classify them side by side; whole batches of loads go
// without a bounds check.  Before, a lane wrote and classified its candidate alone: 20 x 2,642,533 with a tenth wanted 119 us, now 61;
// 16 x 1,000,003 (odd rows, one in a hundred) V and g_i 25.3 -> 22.7 us, V alone 23.3 -> 21.0; 4 x 1,461,252 14.7 -> 13.6.
template <int MODE, bool VEC, int U, bool LISTS>
__global__ void __launch_bounds__(ST_WARPS * 32, 4)
st_collect_kernel(const __grid_constant__ StArgs p) {
    __shared__ unsigned long long stage[ST_BLOCK_OPEN];
    __shared__ __align__(16) int4 gather_sh[ST_WARPS][ST_GATHER];
    __shared__ unsigned sure_sh, open_sh, open_at;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int vec = blockIdx.y;
    int4* gather = gather_sh[warp];
    if (tid == 0) { sure_sh = 0u; open_sh = 0u; }
    __syncthreads();
    pdl_trigger();
    pdl_wait();
#pragma unroll 1
    for (int region = blockIdx.x * ST_WARPS + warp; region < p.nreg; region += gridDim.x * ST_WARPS) {
        const unsigned lo = p.ctl[vec].lo, hi = LISTS ? 0u : p.ctl[vec].hi;
        const i64 base = (i64)region << p.region_log;
        const int end = (int)min((i64)1 << p.region_log, p.d - base);           // positions below are relative to the region
        const float* __restrict__ av = pdl_ptr(p.a + (i64)vec * p.pitch_a + base);
        float* bv = MODE == TC_PLAIN ? nullptr : pdl_ptr(p.b + (i64)vec * p.pitch_b + base);
        unsigned held = 0u, done = 0u, sure = 0u;                               // in the buffer, written before, sure entries (per lane)
        // the buffer's candidates: records to the region's list; an entry is sure, or open (gathered per block: one counter in
        // global memory for every one would serialise them)
        auto empty = [&]() {
            __syncwarp();
            const StCtl& ct = p.ctl[vec];
            int4* out = p.cand + ((i64)vec * p.nreg + region) * p.cap;
            for (unsigned e = lane; e < held; e += 32u) {
                const int4 w = gather[e];
                const unsigned key = (unsigned)w.y & 0x7fffffffu;
                if (LISTS) {
                    if (done + e < (unsigned)p.cap) out[done + e] = w;
                    if (key >= ct.hi) { ++sure; continue; }
                }
                atomicAdd(&p.open_hist[(i64)vec * ST_OPEN_BINS + ((key - ct.lo) >> ct.shift)], 1u);
                const unsigned long long x = st_composite(key, (unsigned)w.x);
                const unsigned at = atomicAdd(&open_sh, 1u);
                if (at < (unsigned)ST_BLOCK_OPEN) stage[at] = x;
                else {
                    const unsigned to = atomicAdd(&p.ctl[vec].open, 1u);
                    if (to < p.open_cap) p.open_list[(i64)vec * p.open_cap + to] = x;
                }
            }
            done += held; held = 0u;
            __syncwarp();
        };
        auto put = [&](unsigned at, int j, float v, float old) {
            gather[at] = make_int4((int)base + j, __float_as_int(v), __float_as_int(__fadd_rn(old, v)), 0);
        };
        // wanted: a candidate (no lists: an open entry)
        auto wanted = [&](float v) {
            const unsigned key = mag_key(v);
            if (LISTS) return key >= lo;
            if (key >= hi) ++sure;
            return key >= lo && key < hi;
        };
        // 128 entries, four consecutive ones per lane
        auto four = [&](int j0, const float4& x, const float4& g) {
            const float old[4] = {g.x, g.y, g.z, g.w};
            const float v[4] = {st_value<MODE>(x.x, old[0], p.gamma), st_value<MODE>(x.y, old[1], p.gamma),
                                st_value<MODE>(x.z, old[2], p.gamma), st_value<MODE>(x.w, old[3], p.gamma)};
            if (MODE == TC_EF) {
                if (j0 + 3 < end) __stcs(reinterpret_cast<float4*>(bv + j0), make_float4(v[0], v[1], v[2], v[3]));
                else { if (j0 < end) bv[j0] = v[0]; if (j0 + 1 < end) bv[j0 + 1] = v[1]; if (j0 + 2 < end) bv[j0 + 2] = v[2]; }
            }
            bool pr[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) pr[e] = wanted(v[e]);                      // lo >= 1: the zeros behind the end never are
            if (__any_sync(0xffffffffu, pr[0] | pr[1] | pr[2] | pr[3])) {
                const unsigned lt = (1u << lane) - 1u;
                unsigned pos = held;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const unsigned bm = __ballot_sync(0xffffffffu, pr[e]);
                    pos += (unsigned)__popc(bm & lt); held += (unsigned)__popc(bm);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (pr[e]) { put(pos, j0 + e, v[e], old[e]); ++pos; }
                if (held >= 32u) empty();
            }
        };
        // 32 * U entries, a lane's 32 apart
        auto apart = [&](int j0, float (&v)[U], const float (&old)[U], int left) {
            bool any = false;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                v[u] = st_value<MODE>(v[u], old[u], p.gamma);
                if (MODE == TC_EF && 32 * u < left) __stcs(bv + j0 + 32 * u, v[u]);
                any |= LISTS ? mag_key(v[u]) >= lo : wanted(v[u]);
            }
            if (__any_sync(0xffffffffu, any)) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const unsigned key = mag_key(v[u]);
                    const bool pr = key >= lo && (LISTS || key < hi);
                    const unsigned bm = __ballot_sync(0xffffffffu, pr);
                    if (pr) put(held + (unsigned)__popc(bm & ((1u << lane) - 1u)), j0 + 32 * u, v[u], old[u]);
                    held += (unsigned)__popc(bm);
                    if (u % 4 == 3 && held >= 32u) empty();
                }
            }
        };
        if (VEC) {
#pragma unroll 1
            for (int i0 = 0; i0 < end; i0 += 128 * U) {
                float4 x[U], g[U];
                if (i0 + 128 * U <= end) {
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int j0 = i0 + 128 * u + 4 * lane;
                        x[u] = __ldcs(reinterpret_cast<const float4*>(av + j0));
                        g[u] = MODE == TC_PLAIN ? make_float4(0.f, 0.f, 0.f, 0.f) : __ldcs(reinterpret_cast<const float4*>(bv + j0));
                    }
                } else {
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int j0 = i0 + 128 * u + 4 * lane, left = end - j0;
                        x[u] = g[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (left > 0) { x[u].x = av[j0]; if (MODE != TC_PLAIN) g[u].x = bv[j0]; }
                        if (left > 1) { x[u].y = av[j0 + 1]; if (MODE != TC_PLAIN) g[u].y = bv[j0 + 1]; }
                        if (left > 2) { x[u].z = av[j0 + 2]; if (MODE != TC_PLAIN) g[u].z = bv[j0 + 2]; }
                        if (left > 3) { x[u].w = av[j0 + 3]; if (MODE != TC_PLAIN) g[u].w = bv[j0 + 3]; }
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) four(i0 + 128 * u + 4 * lane, x[u], g[u]);
            }
        } else {
#pragma unroll 1
            for (int i0 = 0; i0 < end; i0 += 32 * U) {
                const int j0 = i0 + lane, left = end - j0;
                float v[U], old[U];
                if (i0 + 32 * U <= end) {
#pragma unroll
                    for (int u = 0; u < U; ++u) { v[u] = __ldcs(av + j0 + 32 * u); old[u] = MODE == TC_PLAIN ? 0.f : __ldcs(bv + j0 + 32 * u); }
                    apart(j0, v, old, 32 * U);
                } else {
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        v[u] = 32 * u < left ? __ldcs(av + j0 + 32 * u) : 0.f;
                        old[u] = MODE != TC_PLAIN && 32 * u < left ? __ldcs(bv + j0 + 32 * u) : 0.f;
                    }
                    apart(j0, v, old, left);
                }
            }
        }
        empty();
        sure = __reduce_add_sync(0xffffffffu, sure);
        if (lane == 0) {
            if (LISTS) p.reg_cand[(i64)vec * p.nreg_pitch + region] = done;
            p.reg_base[(i64)vec * p.nreg_pitch + region] = sure;
            if (sure) atomicAdd(&sure_sh, sure);
        }
    }
    __syncthreads();
    const unsigned mine = min(open_sh, (unsigned)ST_BLOCK_OPEN);
    if (tid == 0) {
        open_at = mine ? atomicAdd(&p.ctl[vec].open, mine) : 0u;
        if (sure_sh) atomicAdd(&p.ctl[vec].sure, sure_sh);
    }
    __syncthreads();
    for (unsigned e = tid; e < mine; e += ST_WARPS * 32)
        if (open_at + e < p.open_cap) p.open_list[(i64)vec * p.open_cap + open_at + e] = stage[e];
}

// ---- EF21+: both selections and the distortions from one pass -------------------------------------
// Worker i compresses a_i - g_i (vector i of the batch) and a_i (vector n + i).  One pass over a_i and g_i lists the candidates of both
// and adds up the distortions' terms of the entries below each bracket, which are not in that message for sure; those of the candidates
// are added by st_compact_pair_kernel, which knows the cuts.  The terms of a region are squared and added in 32 bits, the regions in 64:
// these sums only tell apart distortions that differ by more than their rounding can be, the others are decided by the ordered 64-bit
// sums as ever (plus_decision).  (All in 64 bits the pass took 65 us for 16 x 1,000,003, conversions and all.)
struct PlusSums {
    double2* low; int* nonzero;         // [n][low_pitch]: (M, B) of the entries below the brackets, per block of the pass; whether g_i has a non-zero there
    int low_pitch, low_parts;
    double* cand; int groups;           // [2 n][groups]: M, then B, of the candidates
    const StCtl* ctl;                   // [2 n]
};

constexpr int ST_PAIR_LOADS = 8, ST_PAIR_OPEN = 1024, ST_PAIR_GATHER = 32 + 32 * ST_PAIR_LOADS;      // (emptied from 32 on)

// A warp's buffer of candidates, and the block's open entries.
struct StPairShared {
    float a[2][ST_WARPS][ST_PAIR_GATHER], g[ST_WARPS][ST_PAIR_GATHER];
    unsigned short at[2][ST_WARPS][ST_PAIR_GATHER];
    unsigned long long open[2][ST_PAIR_OPEN];
};

// grid = (blocks per worker, n), 256 threads, one warp per region, in turn, all blocks resident and every warp with the same number of
// regions (a few blocks more than fit made a second wave: 61 us).  Bound by instructions, about fifty per 32 entries: 16 x 1,000,003,
// one in a hundred, 44 us against 24 + 21 + 32 for two passes and the distortions' own (65 with a call of the emptying code in every
// quarter of a batch, which is more code than the instruction cache takes well; the next batch fetched ahead costs the fourth
// block per SM: 45).
__global__ void __launch_bounds__(ST_WARPS * 32, 4)
st_collect_pair_kernel(const __grid_constant__ StArgs p, const __grid_constant__ PlusSums sums) {
    constexpr int U = ST_PAIR_LOADS;
    extern __shared__ __align__(16) unsigned char st_pair_smem[];
    StPairShared& sh = *reinterpret_cast<StPairShared*>(st_pair_smem);
    __shared__ unsigned sure_sh[2], open_sh[2], open_at[2];
    __shared__ double low_sh[2][ST_WARPS];
    __shared__ int nonzero_sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, worker = blockIdx.y;
    if (tid < 2) { sure_sh[tid] = 0u; open_sh[tid] = 0u; }
    if (tid == 0) nonzero_sh = 0;
    __syncthreads();
    pdl_trigger();
    pdl_wait();
    double low[2] = {0.0, 0.0};
    unsigned bits = 0u;                                              // of g_i, without the signs
    const int vecs[2] = {worker, p.pair + worker};
    const int first = blockIdx.x * ST_WARPS + warp, step = gridDim.x * ST_WARPS;
    const float* __restrict__ av = pdl_ptr(p.a + (i64)worker * p.pitch_a);
    const float* __restrict__ bv = pdl_ptr(p.b + (i64)worker * p.pitch_b);
    // the entries i0 + lane, 32 apart, of a region; zeros behind the end of the vector
    float a_next[U], g_next[U];
    auto fetch = [&](int region, int i0) {
        const i64 j = ((i64)region << p.region_log) + i0 + lane, left = p.d - j;
        if (left + lane >= 32 * U) {
#pragma unroll
            for (int u = 0; u < U; ++u) { a_next[u] = av[j + 32 * u]; g_next[u] = bv[j + 32 * u]; }
        } else {
#pragma unroll
            for (int u = 0; u < U; ++u) { a_next[u] = 32 * u < left ? av[j + 32 * u] : 0.f; g_next[u] = 32 * u < left ? bv[j + 32 * u] : 0.f; }
        }
    };
#pragma unroll 1
    for (int region = first; region < p.nreg; region += step) {
        const unsigned lo[2] = {p.ctl[vecs[0]].lo, p.ctl[vecs[1]].lo};
        const i64 base = (i64)region << p.region_log;
        const int end = (int)min((i64)1 << p.region_log, p.d - base);           // positions below are relative to the region
        unsigned held[2] = {0u, 0u}, done[2] = {0u, 0u}, sure[2] = {0u, 0u};
        float below[2] = {0.f, 0.f};                                            // this region's terms, 32 or 128 per lane
        // a buffer's candidates: records to the region's list; an entry is sure, or open
        auto empty = [&](int s) {
            __syncwarp();
            const StCtl& ct = p.ctl[vecs[s]];
            int4* out = p.cand + ((i64)vecs[s] * p.nreg + region) * p.cap;
#pragma unroll 1
            for (unsigned e = lane; e < held[s]; e += 32u) {
                const float a = sh.a[s][warp][e], g = s == 0 ? sh.g[warp][e] : 0.f;
                const float v = s == 0 ? __fsub_rn(a, g) : a;                   // (a - 0 would change the bits, and so the order, of a NaN)
                const int j = (int)base + sh.at[s][warp][e];
                const unsigned key = mag_key(v);
                if (done[s] + e < (unsigned)p.cap) out[done[s] + e] = make_int4(j, __float_as_int(v), __float_as_int(g), __float_as_int(a));
                if (key >= ct.hi) { ++sure[s]; continue; }
                atomicAdd(&p.open_hist[(i64)vecs[s] * ST_OPEN_BINS + ((key - ct.lo) >> ct.shift)], 1u);
                const unsigned long long x = st_composite(key, (unsigned)j);
                const unsigned at = atomicAdd(&open_sh[s], 1u);
                if (at < (unsigned)ST_PAIR_OPEN) sh.open[s][at] = x;
                else {
                    const unsigned to = atomicAdd(&p.ctl[vecs[s]].open, 1u);
                    if (to < p.open_cap) p.open_list[(i64)vecs[s] * p.open_cap + to] = x;
                }
            }
            done[s] += held[s]; held[s] = 0u;
            __syncwarp();
        };
#pragma unroll 1
        for (int i0 = 0; i0 < end; i0 += 32 * U) {
            const int j0 = i0 + lane;
            const bool last = i0 + 32 * U >= end;
            fetch(region, i0);
            float (&a)[U] = a_next, (&g)[U] = g_next;
#pragma unroll
            for (int u = 0; u < U; ++u) {                                       // entries behind the end are zeros
                const float v = __fsub_rn(a[u], g[u]);
                const bool pr[2] = {mag_key(v) >= lo[0], mag_key(a[u]) >= lo[1]};
                if (!pr[0]) below[0] = fmaf(v, v, below[0]);
                if (!pr[1]) below[1] = fmaf(a[u], a[u], below[1]);
                bits |= __float_as_uint(g[u]);
#pragma unroll
                for (int s = 0; s < 2; ++s) {
                    const unsigned bm = __ballot_sync(0xffffffffu, pr[s]);
                    if (bm == 0u) continue;
                    if (pr[s]) {
                        const unsigned to = held[s] + (unsigned)__popc(bm & ((1u << lane) - 1u));
                        sh.a[s][warp][to] = a[u];
                        if (s == 0) sh.g[warp][to] = g[u];
                        sh.at[s][warp][to] = (unsigned short)(j0 + 32 * u);
                    }
                    held[s] += (unsigned)__popc(bm);
                }
            }
#pragma unroll
            for (int s = 0; s < 2; ++s)
                if (held[s] >= 32u || last) empty(s);
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            low[s] += (double)below[s];
            const unsigned all = __reduce_add_sync(0xffffffffu, sure[s]);
            if (lane == 0) {
                p.reg_cand[(i64)vecs[s] * p.nreg_pitch + region] = done[s];
                p.reg_base[(i64)vecs[s] * p.nreg_pitch + region] = all;
                if (all) atomicAdd(&sure_sh[s], all);
            }
        }
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        low[s] = warp_sum(low[s]);
        if (lane == 0) low_sh[s][warp] = low[s];
    }
    if (__any_sync(0xffffffffu, (bits << 1) != 0u) && lane == 0) nonzero_sh = 1;
    __syncthreads();
    if (tid == 0) {
        double2 sum = make_double2(0.0, 0.0);
        for (int w = 0; w < ST_WARPS; ++w) { sum.x += low_sh[0][w]; sum.y += low_sh[1][w]; }
        sums.low[(i64)worker * sums.low_pitch + blockIdx.x] = sum;
        sums.nonzero[(i64)worker * sums.low_pitch + blockIdx.x] = nonzero_sh;
    }
    if (tid < 2) {
        const unsigned n = min(open_sh[tid], (unsigned)ST_PAIR_OPEN);
        open_at[tid] = n ? atomicAdd(&p.ctl[vecs[tid]].open, n) : 0u;
        if (sure_sh[tid]) atomicAdd(&p.ctl[vecs[tid]].sure, sure_sh[tid]);
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < 2; ++s)
        for (unsigned e = tid; e < min(open_sh[s], (unsigned)ST_PAIR_OPEN); e += ST_WARPS * 32)
            if (open_at[s] + e < p.open_cap) p.open_list[(i64)vecs[s] * p.open_cap + open_at[s] + e] = sh.open[s][e];
}

// ---- exact cut and the regions' first positions ---------------------------------------------------
// One cluster of C blocks of 1,024 threads per vector; dynamic shared memory for ST_OPEN_STAGE composites.  CLASSIFY: the streaming
// pass has only listed the candidates; they are divided into sure and open ones here, the open ones of a block stay in its
// shared memory (another ST_OPEN_STAGE composites and the histogram).
__host__ __device__ constexpr size_t st_cut_smem_bytes(bool classify) {
    return (size_t)ST_OPEN_STAGE * 8 + (classify ? (size_t)ST_OPEN_STAGE * 8 + (size_t)ST_OPEN_BINS * 4 : 0);
}

template <int C, bool CLASSIFY>
__global__ void __launch_bounds__(1024)
st_cut_kernel(const __grid_constant__ StArgs p) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char st_cut_smem[];
    unsigned long long* stage = reinterpret_cast<unsigned long long*>(st_cut_smem);      // block 0: open entries of the deciding step
    unsigned long long* mine_open = stage + ST_OPEN_STAGE;                               // CLASSIFY: this block's open entries
    unsigned* hist = reinterpret_cast<unsigned*>(mine_open + ST_OPEN_STAGE);             // CLASSIFY: their histogram
    __shared__ unsigned scratch[33], scratch_b[32], found[3], stage_n, sure_sh, open_sh, over_sh;
    __shared__ unsigned long long cut_sh, differ_sh;
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, rk = (int)cluster.block_rank(), vec = (int)(blockIdx.x / (unsigned)C);
    if (tid == 0) { stage_n = 0u; sure_sh = 0u; open_sh = 0u; over_sh = 0u; differ_sh = 0ull; }
    if (CLASSIFY) { hist[tid] = 0u; hist[tid + 1024] = 0u; }
    __syncthreads();
    if (!CLASSIFY) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); // block 0's counter is ready
    pdl_trigger();
    pdl_wait();
    StCtl& ct = p.ctl[vec];
    const unsigned k = (unsigned)p.k, lo = ct.lo, hi = ct.hi, shift = ct.shift;
    unsigned* base = p.reg_base + (i64)vec * p.nreg_pitch;
    const unsigned long long* list = CLASSIFY ? mine_open : p.open_list + (i64)vec * p.open_cap;
    const unsigned e0 = CLASSIFY ? (unsigned)tid : (unsigned)(rk * 1024 + tid), e_step = CLASSIFY ? 1024u : C * 1024u;
    unsigned long long x0 = 0ull;
    uint2 c;
    unsigned sure, open, my_open;                                    // of the vector; open entries this block goes through
    bool slow;
    if (CLASSIFY) {
        // 2^group lanes per region, as many as there are threads for; neighbouring regions go to different blocks, so that every
        // block has its share of the open entries (a lane per region and block 0 taking the first 1,024 of them: 64 x 1,024
        // regions 20 us, 16 x 1,024 35 us, and more open entries than one block holds from k = d / 400 on)
        int group = 0;
        while (group < 5 && (p.nreg << (group + 1)) <= C * 1024) ++group;
        const unsigned lanes = 1u << group, sub = (unsigned)tid & (lanes - 1u);
        unsigned sure_mine = 0u;
        bool over = false;
        for (int r0 = 0; r0 < p.nreg; r0 += (C * 1024) >> group) {
            const int r = r0 + (tid >> group) * C + rk;
            const unsigned n = r < p.nreg ? p.reg_cand[(i64)vec * p.nreg_pitch + r] : 0u;
            const int2* rec = reinterpret_cast<const int2*>(p.cand + ((i64)vec * p.nreg + r) * p.cap);
            unsigned s = 0u;
            over |= n > (unsigned)p.cap;
#pragma unroll 4
            for (unsigned e = sub; e < min(n, (unsigned)p.cap); e += lanes) {
                const int2 w = rec[2 * e];
                const unsigned key = (unsigned)w.y & 0x7fffffffu;
                if (key >= hi) ++s;
                else {
                    atomicAdd(&hist[(key - lo) >> shift], 1u);
                    const unsigned at = atomicAdd(&open_sh, 1u);
                    if (at < (unsigned)ST_OPEN_STAGE) mine_open[at] = st_composite(key, (unsigned)w.x);
                }
            }
            sure_mine += s;
            __syncwarp();
            for (unsigned off = 1u; off < lanes; off <<= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            if (r < p.nreg && sub == 0u) base[r] = s;
        }
        sure_mine = __reduce_add_sync(0xffffffffu, sure_mine);
        if ((tid & 31) == 0 && sure_mine) atomicAdd(&sure_sh, sure_mine);
        if (over) over_sh = 1u;
        __syncthreads();
        if (tid == 0 && open_sh > (unsigned)ST_OPEN_STAGE) over_sh = 1u;
        __threadfence();
        cluster.sync();
        sure = open = 0u; slow = false;
        c = make_uint2(0u, 0u);
#pragma unroll
        for (int r = 0; r < C; ++r) {
            sure += *cluster.map_shared_rank(&sure_sh, r); open += *cluster.map_shared_rank(&open_sh, r);
            slow |= *cluster.map_shared_rank(&over_sh, r) != 0u;
            const uint2 o = reinterpret_cast<const uint2*>(cluster.map_shared_rank(hist, r))[1023 - tid];
            c.x += o.x; c.y += o.y;
        }
        my_open = open_sh;
        slow |= sure > k || sure + open < k;
    } else {
        x0 = e0 < p.open_cap ? list[e0] : 0ull;                      // on its way while the counters and the histogram arrive
        c = reinterpret_cast<const uint2*>(p.open_hist + (i64)vec * ST_OPEN_BINS)[1023 - tid];
        sure = ct.sure; open = ct.open;
        my_open = open;
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        slow = sure > k || sure + open < k || open > p.open_cap;     // the same in all blocks
    }
    unsigned need = slow ? 0u : k - sure;
    unsigned step = 0u, pop = 0u;
    if (need > 0u) {
        // step of [lo, hi) that holds the need-th largest open entry: thread t owns two steps, the higher one first
        unsigned total;
        const unsigned up = block_excl_scan(c.x + c.y, scratch, total);
        if (up < need && need <= up + c.y) { found[0] = (unsigned)(2047 - 2 * tid); found[1] = up; found[2] = c.y; }
        else if (up + c.y < need && need <= up + c.y + c.x) { found[0] = (unsigned)(2046 - 2 * tid); found[1] = up + c.y; found[2] = c.x; }
        __syncthreads();
        step = found[0]; pop = found[2];
        need -= found[1];
        slow = pop > (unsigned)ST_OPEN_STAGE;
    }
    if (slow) {
        if (CLASSIFY) cluster.sync();                                // (the others may still read this block's counters)
        if (rk == 0 && tid == 0) { ct.slow = 1u; if (p.slow_count) atomicAdd(p.slow_count, 1u); }
        return;
    }
    unsigned long long cut = st_composite(hi, 0xffffffffu);       // need == 0: the sure entries are the message
    if (need > 0u) {
        unsigned long long* stage0 = cluster.map_shared_rank(stage, 0);
        unsigned* stage_n0 = cluster.map_shared_rank(&stage_n, 0);
        // entries of higher steps are in the message: count them into their regions; those of the step go to block 0
#pragma unroll 4
        for (unsigned e = e0; e < my_open; e += e_step) {
            const unsigned long long x = !CLASSIFY && e == e0 ? x0 : list[e];
            const unsigned s = ((unsigned)(x >> 32) - lo) >> shift;
            if (s > step) atomicAdd(&base[(0xffffffffu - (unsigned)x) >> p.region_log], 1u);
            else if (s == step) stage0[atomicAdd(stage_n0, 1u)] = x;
        }
        __threadfence();
        cluster.sync();
        if (rk != 0) return;
        if (pop <= 256u) {
            // one entry per thread, ranked by counting (the composites are distinct)
            const bool have = tid < (int)pop;
            const unsigned long long mine = have ? stage[tid] : 0ull;
            unsigned gt = 0u;
            if (have)
#pragma unroll 4
                for (unsigned o = 0; o < pop; ++o) gt += stage[o] > mine ? 1u : 0u;
            if (have && gt + 1u == need) cut_sh = mine;
            __syncthreads();
            cut = cut_sh;
        } else {
            // Largest cut with at least `need` entries at or above it.  Bits that all of them share are the cut's; the others are
            // found two at a time.  (All bits of the step, one at a time: rounds on 64 x 4,194,304 values of bf16, whose groups of
            // equal keys share all but the index, 395 us instead of 388.)
            const unsigned long long any = stage[0];
            unsigned long long differ = 0ull;
            for (unsigned e = tid; e < pop; e += 1024u) differ |= stage[e] ^ any;
            const unsigned dh = __reduce_or_sync(0xffffffffu, (unsigned)(differ >> 32)), dl = __reduce_or_sync(0xffffffffu, (unsigned)differ);
            if ((tid & 31) == 0) atomicOr(&differ_sh, ((unsigned long long)dh << 32) | dl);
            __syncthreads();
            differ = differ_sh;
            cut = any & ~differ;
#pragma unroll 1
            while (differ != 0ull) {
                const unsigned long long b1 = 1ull << (63 - __clzll((long long)differ));
                differ ^= b1;
                const unsigned long long b0 = differ != 0ull ? 1ull << (63 - __clzll((long long)differ)) : 0ull;
                differ ^= b0;
                unsigned two = 0u, one = 0u;                         // at or above cut + b1 + b0 (low half) and cut + b1; cut + b0
                for (unsigned e = tid; e < pop; e += 1024u) {
                    const unsigned long long x = stage[e];
                    two += (x >= (cut | b1 | b0) ? 1u : 0u) + (x >= (cut | b1) ? 0x10000u : 0u);
                    one += x >= (cut | b0) ? 1u : 0u;
                }
                two = __reduce_add_sync(0xffffffffu, two); one = __reduce_add_sync(0xffffffffu, one);
                if ((tid & 31) == 0) { scratch[tid >> 5] = two; scratch_b[tid >> 5] = one; }
                __syncthreads();
                two = __reduce_add_sync(0xffffffffu, scratch[tid & 31]); one = __reduce_add_sync(0xffffffffu, scratch_b[tid & 31]);
                __syncthreads();
                if ((two & 0xffffu) >= need) cut |= b1 | b0;
                else if ((two >> 16) >= need) cut |= b1;
                else if (one >= need) cut |= b0;
            }
        }
        for (unsigned e = tid; e < pop; e += 1024u) {
            const unsigned long long x = stage[e];
            if (x >= cut) atomicAdd(&base[(0xffffffffu - (unsigned)x) >> p.region_log], 1u);
        }
        __threadfence();
        __syncthreads();
    } else {
        if (CLASSIFY) cluster.sync();
        if (rk != 0) return;
    }
    if (tid == 0) ct.cut = cut;
    // counts -> first positions (the counts were changed by atomics: read them from L2, behind the barrier)
    base = pdl_ptr(base);
    unsigned before = 0u;
    for (int r0 = 0; r0 < p.nreg; r0 += 8192) {
        const int r = r0 + 8 * tid;                                  // the padding behind the last region is added up and ignored
        const bool in = r < p.nreg;
        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
        const uint4 lo4 = in ? __ldcg(reinterpret_cast<const uint4*>(base + r)) : z, hi4 = in ? __ldcg(reinterpret_cast<const uint4*>(base + r) + 1) : z;
        unsigned total;
        const unsigned sum = lo4.x + lo4.y + lo4.z + lo4.w + hi4.x + hi4.y + hi4.z + hi4.w;
        uint4 a, b;
        a.x = before + block_excl_scan(sum, scratch, total);
        a.y = a.x + lo4.x; a.z = a.y + lo4.y; a.w = a.z + lo4.z;
        b.x = a.w + lo4.w; b.y = b.x + hi4.x; b.z = b.y + hi4.y; b.w = b.z + hi4.z;
        if (in) { reinterpret_cast<uint4*>(base + r)[0] = a; reinterpret_cast<uint4*>(base + r)[1] = b; }
        before += total;
    }
}

// ---- 3. ordered compaction ----------------------------------------------------------------------
struct StOut {
    int* idx_out; float* val_out;       // [batch][k]
    float* apply; i64 pitch_apply;      // receives b + v on the selected coordinates (TC_EF: zero); may be null
    int* tile_off; int ntiles;          // [batch][ntiles + 1] first message position of every 2,048 coordinates; may be null
    unsigned* status;
    unsigned long long* cut_out;        // [batch] the cut of every vector; may be null
};

// grid = (ceil(nreg / 32), batch), 256 threads: eight lanes per region (four in one wave instead of two: no faster).
template <int MODE>
__global__ void __launch_bounds__(256)
st_compact_kernel(const __grid_constant__ StArgs p, const StOut o) {
    pdl_trigger();
    pdl_wait();
    const int vec = blockIdx.y, lane = threadIdx.x & 31, sub = lane & 7, group = lane & ~7;
    const int region = blockIdx.x * 32 + (threadIdx.x >> 3);
    const StCtl& ct = p.ctl[vec];
    if (ct.slow) return;
    const unsigned long long cut = ct.cut;
    if (o.cut_out && blockIdx.x == 0 && threadIdx.x == 0) o.cut_out[vec] = cut;
    const bool have = region < p.nreg;
    const unsigned n = have ? p.reg_cand[(i64)vec * p.nreg_pitch + region] : 0u;
    unsigned pos = have ? p.reg_base[(i64)vec * p.nreg_pitch + region] : 0u;
    const unsigned first = pos;
    int* io = o.idx_out + (i64)vec * p.k;
    float* vo = o.val_out + (i64)vec * p.k;
    float* app = o.apply ? o.apply + (i64)vec * o.pitch_apply : nullptr;
    const i64 base = (i64)region << p.region_log;
    unsigned front = 0u;                                            // selected entries in the first 2,048 coordinates of the region
    const bool two_tiles = o.tile_off && p.region_log == 12;
    auto emit = [&](bool sel, int j, float v, float nw) {
        const unsigned bal = (__ballot_sync(0xffffffffu, sel) >> group) & 0xffu;
        if (sel) {
            const unsigned at = pos + (unsigned)__popc(bal & ((1u << sub) - 1u));
            io[at] = j; vo[at] = v;
            flag_nonfinite(o.status, v);
            if (app) app[j] = MODE == TC_EF ? __fsub_rn(v, v) : nw;
        }
        if (two_tiles) front += (unsigned)__popc((__ballot_sync(0xffffffffu, sel && j < base + 2048) >> group) & 0xffu);
        pos += (unsigned)__popc(bal);
    };
    const bool listed = n <= (unsigned)p.cap;
    const unsigned steps = __reduce_max_sync(0xffffffffu, listed ? (n + 7u) / 8u : 0u);
    const int4* in = p.cand + ((i64)vec * p.nreg + (have ? region : 0)) * p.cap;
    for (unsigned s = 0; s < steps; ++s) {
        const unsigned e = 8u * s + (unsigned)sub;
        const bool mine = listed && e < n;
        const int4 w = mine ? in[e] : make_int4(0, 0, 0, 0);
        const float v = __int_as_float(w.y);
        emit(mine && st_composite(mag_key(v), (unsigned)w.x) >= cut, w.x, v, __int_as_float(w.z));
    }
    // regions whose list overflowed (or that keep none): all four groups of the warp stay together, each reads its own
    if (__any_sync(0xffffffffu, !listed)) {
        const float* __restrict__ av = pdl_ptr(p.a + (i64)vec * p.pitch_a);
        const float* bv = MODE == TC_PLAIN ? nullptr : p.b + (i64)vec * p.pitch_b;
        for (int s = 0; s < 1 << (p.region_log - 3); s += 4) {
            float v[4], nw[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const i64 j = base + 8 * (s + u) + sub;
                const bool in_range = !listed && j < p.d;
                const float b = (MODE != TC_PLAIN && in_range) ? bv[j] : 0.f;        // TC_EF: v itself by now
                v[u] = !in_range ? 0.f : (MODE == TC_EF ? b : st_value<MODE>(av[j], b, p.gamma));
                nw[u] = __fadd_rn(b, v[u]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const i64 j = base + 8 * (s + u) + sub;
                emit(!listed && j < p.d && st_composite(mag_key(v[u]), (unsigned)j) >= cut, (int)j, v[u], nw[u]);
            }
        }
    }
    if (o.tile_off && have && sub == 0) {
        int* off = o.tile_off + (i64)vec * (o.ntiles + 1);
        if (two_tiles) {
            off[2 * region] = (int)first;
            if (2 * region + 1 < o.ntiles) off[2 * region + 1] = (int)(first + front);
        } else if ((region & 1) == 0) {
            off[region >> 1] = (int)first;                          // two regions of 1,024 make a tile
        }
        if (region == p.nreg - 1) off[o.ntiles] = p.k;
    }
}

// The messages of EF21+ and the candidates' terms of the distortions; grid = (ceil(nreg / 32), 2 n), 256 threads, eight lanes per region.
// A Markov record is (index, v, g, a), a plain one (index, a, 0, a).
__global__ void __launch_bounds__(256)
st_compact_pair_kernel(const __grid_constant__ StArgs p, const __grid_constant__ PlusSums sums, int* idx_m, float* val_m, int* idx_b, float* val_b,
                       unsigned long long* cut_out, unsigned* status) {
    pdl_trigger();
    pdl_wait(idx_m, val_m, idx_b, val_b, cut_out, status);
    __shared__ double sum_sh[8];
    const int vec = blockIdx.y, lane = threadIdx.x & 31, sub = lane & 7, group = lane & ~7;
    const bool plain = vec >= p.pair;
    const int worker = plain ? vec - p.pair : vec;
    const int region = blockIdx.x * 32 + (threadIdx.x >> 3);
    const StCtl& ct = p.ctl[vec];
    if (ct.slow) return;
    const unsigned long long cut = ct.cut;
    const unsigned lo = ct.lo;
    if (blockIdx.x == 0 && threadIdx.x == 0) cut_out[vec] = cut;
    const bool have = region < p.nreg;
    const unsigned n = have ? p.reg_cand[(i64)vec * p.nreg_pitch + region] : 0u;
    unsigned pos = have ? p.reg_base[(i64)vec * p.nreg_pitch + region] : 0u;
    int* io = (plain ? idx_b : idx_m) + (i64)worker * p.k;
    float* vo = (plain ? val_b : val_m) + (i64)worker * p.k;
    const i64 base = (i64)region << p.region_log;
    double sum = 0.0;
    auto emit = [&](bool mine, int j, float v, float g, float a) {
        const bool sel = mine && st_composite(mag_key(v), (unsigned)j) >= cut;
        const unsigned bal = (__ballot_sync(0xffffffffu, sel) >> group) & 0xffu;
        if (sel) {
            const unsigned at = pos + (unsigned)__popc(bal & ((1u << sub) - 1u));
            io[at] = j; vo[at] = v;
            flag_nonfinite(status, v);
        }
        if (mine) {
            const double e = plain ? (sel ? 0.0 : (double)a) : (double)(sel ? __fadd_rn(g, v) : g) - (double)a;
            sum = fma(e, e, sum);
        }
        pos += (unsigned)__popc(bal);
    };
    const bool listed = n <= (unsigned)p.cap;
    const unsigned steps = __reduce_max_sync(0xffffffffu, listed ? (n + 7u) / 8u : 0u);
    const int4* in = p.cand + ((i64)vec * p.nreg + (have ? region : 0)) * p.cap;
    for (unsigned s = 0; s < steps; ++s) {
        const unsigned e = 8u * s + (unsigned)sub;
        const bool mine = listed && e < n;
        const int4 w = mine ? in[e] : make_int4(0, 0, 0, 0);
        emit(mine, w.x, __int_as_float(w.y), __int_as_float(w.z), __int_as_float(w.w));
    }
    // regions whose list overflowed: all four groups of the warp stay together, each reads its own
    if (__any_sync(0xffffffffu, !listed)) {
        const float* __restrict__ av = pdl_ptr(p.a + (i64)worker * p.pitch_a);
        const float* __restrict__ bv = pdl_ptr(p.b + (i64)worker * p.pitch_b);
        for (int s = 0; s < 1 << (p.region_log - 3); ++s) {
            const i64 j = base + 8 * s + sub;
            const bool in_range = !listed && j < p.d;
            const float a = in_range ? av[j] : 0.f, g = in_range ? bv[j] : 0.f, v = plain ? a : __fsub_rn(a, g);
            emit(in_range && mag_key(v) >= lo, (int)j, v, g, a);
        }
    }
    sum = warp_sum(sum);
    if (lane == 0) sum_sh[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        double all = 0.0;
        for (int w = 0; w < 8; ++w) all += sum_sh[w];
        sums.cand[(i64)vec * sums.groups + blockIdx.x] = all;
    }
}

// The compaction where no lists are kept (more than a tenth of the entries are wanted): one warp per region reads it again, and gathers
// the selected ones of 256 entries in shared memory before they are written side by side.  Bound by instructions (20 x 2,642,533, a
// tenth wanted: 83 us with a store per lane and entry, now 73).
// grid = (ceil(nreg / 8), batch), 256 threads.
constexpr int ST_REREAD_LOADS = 8;

template <int MODE>
__global__ void __launch_bounds__(256)
st_reread_kernel(const __grid_constant__ StArgs p, const StOut o) {
    __shared__ int2 gather_sh[8][32 * ST_REREAD_LOADS];
    pdl_trigger();
    pdl_wait();
    const int vec = blockIdx.y, lane = threadIdx.x & 31;
    const int region = blockIdx.x * 8 + (threadIdx.x >> 5);
    const StCtl& ct = p.ctl[vec];
    if (ct.slow || region >= p.nreg) return;
    const unsigned long long cut = ct.cut;
    if (o.cut_out && blockIdx.x == 0 && threadIdx.x == 0) o.cut_out[vec] = cut;
    const unsigned cut_key = (unsigned)(cut >> 32), cut_idx = 0xffffffffu - (unsigned)cut;
    const unsigned first = p.reg_base[(i64)vec * p.nreg_pitch + region];
    unsigned pos = first;
    const i64 base = (i64)region << p.region_log;
    const int end = (int)min((i64)1 << p.region_log, p.d - base);
    const float* __restrict__ av = pdl_ptr(p.a + (i64)vec * p.pitch_a + base);
    const float* bv = MODE == TC_PLAIN ? nullptr : p.b + (i64)vec * p.pitch_b + base;
    int* io = o.idx_out + (i64)vec * p.k;
    float* vo = o.val_out + (i64)vec * p.k;
    float* app = o.apply ? o.apply + (i64)vec * o.pitch_apply + base : nullptr;
    constexpr int U = ST_REREAD_LOADS;
    int2* gather = gather_sh[threadIdx.x >> 5];
    const i64 tie = (i64)cut_idx - base;                            // an entry at the cut's key is in the message up to here
#pragma unroll 1
    for (int i0 = 0; i0 < end; i0 += 32 * U) {
        const int j0 = i0 + lane;
        const int left = i0 + 32 * U <= end ? 32 * U : end - j0;
        if (o.tile_off && j0 == 2048) o.tile_off[(i64)vec * (o.ntiles + 1) + 2 * region + 1] = (int)pos;
        float v[U], b[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            b[u] = MODE != TC_PLAIN && 32 * u < left ? bv[j0 + 32 * u] : 0.f;        // TC_EF: v itself by now
            v[u] = MODE != TC_EF && 32 * u < left ? av[j0 + 32 * u] : 0.f;
        }
        unsigned n = 0u;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            v[u] = MODE == TC_EF ? b[u] : st_value<MODE>(v[u], b[u], p.gamma);
            const bool sel = 32 * u < left && mag_key(v[u]) >= cut_key + (j0 + 32 * u > tie ? 1u : 0u);
            const unsigned bal = __ballot_sync(0xffffffffu, sel);
            if (sel) {
                gather[n + (unsigned)__popc(bal & ((1u << lane) - 1u))] = make_int2((int)base + j0 + 32 * u, __float_as_int(v[u]));
                if (app) app[j0 + 32 * u] = MODE == TC_EF ? __fsub_rn(v[u], v[u]) : __fadd_rn(b[u], v[u]);
            }
            n += (unsigned)__popc(bal);
        }
        __syncwarp();
        for (unsigned e = lane; e < n; e += 32u) {
            const int2 w = gather[e];
            io[pos + e] = w.x; vo[pos + e] = __int_as_float(w.y);
            flag_nonfinite(o.status, __int_as_float(w.y));
        }
        pos += n;
        __syncwarp();
    }
    if (o.tile_off && lane == 0) {
        int* off = o.tile_off + (i64)vec * (o.ntiles + 1);
        if (p.region_log == 12) off[2 * region] = (int)first;
        else if ((region & 1) == 0) off[region >> 1] = (int)first;
        if (region == p.nreg - 1) off[o.ntiles] = p.k;
    }
}

}  // namespace ef21
