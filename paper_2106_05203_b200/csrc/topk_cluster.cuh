// Exact Top-k of vectors that fit into the shared memory of one thread-block cluster: the whole selection in ONE
// launch, one cluster of C blocks per vector.
//
//   1. block r holds the coordinates [r * slice, (r + 1) * slice) of v in shared memory (v is formed once, on the way in;
//      kept as its bits rotated left by one, so that an unsigned compare orders magnitudes) and counts the leading 11 bits
//      of the magnitude keys in a shared-memory histogram;
//   2. the non-empty bins are added up in the block that owns the bin (distributed shared memory, 2048 / C bins per block),
//      every block reads the sums and finds the bin that holds the k-th largest key (redundantly: the barrier that handing
//      the result around would need costs more than the reading);
//   3. every block lists its own keys of that bin; every block then reads all C lists and finds the k-th largest key T by
//      counting (up to TC_RANKED keys) or by two more histograms over the list.  More than TC_LIST keys in the bin (ties,
//      narrow ranges): the two histograms run over the vector instead;
//   4. ordered compaction: the lists also tell how many entries above T (and equal to T) the warps and blocks before this
//      one hold; ties at T are taken in index order.
// The same kernel, with the vector left in global memory, is the exact fallback of the streaming path (topk_stream.cuh).
//
// What bounds it: latencies and issue slots, not bandwidth.  A block executes each piece of code once, a cluster barrier
// takes about 1,000 cycles (measured; __syncthreads 40), and what all 32 warps of a block execute redundantly costs eight
// times what eight of them would pay.  Hence two cluster barriers on the path, few and short code paths, searches by eight
// warps.
#pragma once
#include <cooperative_groups.h>

#include "bisect.cuh"
#include "common.cuh"
#include "grad.cuh"

namespace ef21 {

constexpr int TC_BITS = 11, TC_BINS = 1 << TC_BITS;      // digits of 11 + 11 + 9 bits
constexpr int TC_LIST = 2048;               // keys of the deciding bin that are handled as a list
constexpr int TC_RANKED = 256;              // up to this many of them are ranked by counting (two more histograms: +1.2 us)
constexpr int TC_MAX_CLUSTER = 16;          // 16 needs the non-portable cluster size; used only where 8 blocks cannot hold the vector
constexpr int TC_MAX_SLICE = 47104;         // floats per block (184 KB)

// How v is formed: TC_PLAIN v = a; TC_DIFF v = a - b; TC_EF v = b + gamma * a, and b takes v (Algorithm 4: the error vector
// becomes the vector to be compressed); TC_SENT v = b, which a TC_EF pass has already formed; TC_PAIR (long vectors of EF21+): the
// first half of the batch is a - b, the second half the same a once more.
enum { TC_PLAIN = 0, TC_DIFF = 1, TC_EF = 2, TC_SENT = 3, TC_PAIR = 4 };

// What a sweep does with an entry beside keeping it: count it, take the thread's largest, nothing.
enum { TC_COUNT = 0, TC_LARGEST = 1, TC_KEEP = 2 };
template <int V> struct TcUse { static constexpr int value = V; };

struct TcArgs {
    const float* a; i64 pitch_a;
    float* b; i64 pitch_b;                  // TC_EF: updated in place
    int d, k, slice;
    float gamma;
    int* idx_out; float* val_out;
    float* apply; i64 pitch_apply;          // TC_DIFF: receives b + v on the selected coordinates; TC_EF, TC_SENT: v - v there; TC_PLAIN: v there and 0 elsewhere; may be null
    unsigned* status;
    unsigned long long* cut_out;            // [batch]: an entry is selected if and only if (key << 32 | ~index) >= cut; may be null
    unsigned* slow_count;                   // counts the vectors with more than TC_LIST entries equal to T; may be null
    // GRAD only: a is the mean of worker i's tile partials plus the regulariser term at x (the sums of grad_finish_kernel)
    const float* partial; const int* tile_begin; const i64* row_off; const float* x;
    float lambda; int ld, batch_rows;
    // REDO only: vectors whose flag (one word every flag_pitch words) is zero are left alone; tile_off (may be null):
    // [batch][ntiles + 1] first message position of every `tile` coordinates
    const unsigned* flag; int flag_pitch, batch;
    int* tile_off; int ntiles, tile;
};

__host__ __device__ constexpr size_t tc_smem_bytes(int C, int slice) {
    return (size_t)slice * 4 + (size_t)TC_LIST * 5 + (size_t)TC_BINS * 4 + (C > 1 ? (size_t)(TC_LIST + TC_BINS) * 4 : 0);
}

// Bin of the histogram (bin 0 not counted in it) that holds the need-th largest of `population` entries: found[] = bin,
// entries in higher bins, entries in the bin.  All threads call it; the first 256 search, eight bins each.
__device__ __noinline__ void tc_find_bin(const unsigned* hist, unsigned need, unsigned population, unsigned* wsum, unsigned* found) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (warp < 8) {
        // thread t owns the bins [2040 - 8 t, 2048 - 8 t), highest first
        const uint4 hi = reinterpret_cast<const uint4*>(hist)[2 * (255 - tid) + 1], lo = reinterpret_cast<const uint4*>(hist)[2 * (255 - tid)];
        const unsigned c[8] = {hi.w, hi.z, hi.y, hi.x, lo.w, lo.z, lo.y, lo.x};
        unsigned sum = 0u;
#pragma unroll
        for (int q = 0; q < 8; ++q) sum += c[q];
        const unsigned wtot = __reduce_add_sync(0xffffffffu, sum);
        if (lane == 0) wsum[warp] = wtot;
        asm volatile("bar.sync 1, 256;" ::: "memory");
        unsigned before = 0u, total = 0u;
#pragma unroll
        for (int w = 0; w < 8; ++w) { const unsigned t = wsum[w]; if (w < warp) before += t; total += t; }
        if (before < need && need <= before + wtot) {                // one warp
            unsigned up = before + warp_incl_scan(sum) - sum;
            if (up < need && need <= up + sum) {                     // one lane
                bool open = true;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    if (open && need <= up + c[q]) { found[0] = (unsigned)(2047 - (8 * tid + q)); found[1] = up; found[2] = c[q]; open = false; }
                    up += c[q];
                }
            }
        } else if (need > total && tid == 0) {
            found[0] = 0u; found[1] = total; found[2] = population - total;
        }
    }
    __syncthreads();
}

// Few entries (few_limit: a quarter of the threads at most) of a vector that one block holds, NV per thread: at least k threads have an entry at or above the k-th
// largest of the threads' largest ones.  A floor with k to 5/4 k + 4 of these above it is found by bisection (a barrier that counts per
// step, six to eight steps between the smallest and the greatest of them); the message is among the entries from the floor on, about 5/4 k
// again as a rule, which are ranked one against the other, two to eight lanes per entry.  No histogram, no sweep for the compaction.
// 16 x 5,829, Top-58: 8.8 us with the histogram, now 7.7; selection behind the gradients of 20 x 5,001, Top-50: 10.4 -> 5.2 thousand cycles.
// list_n is zero and ws complete on entry; false (for all threads): more candidates than are ranked, nothing is written.
__host__ __device__ constexpr int tc_few_values(int threads) { return threads == 256 ? 8 : 16; }

template <int MODE, int THREADS>
__device__ __forceinline__ bool tc_few(const TcArgs& p, int vec, const unsigned* ws, unsigned* hist, unsigned* list, unsigned* wmin, unsigned* wmax,
                                       unsigned& list_n) {
    constexpr int NV = tc_few_values(THREADS), WARPS = THREADS / 32;
    constexpr unsigned CAP = THREADS / 2;
    unsigned long long* cand = reinterpret_cast<unsigned long long*>(list);     // (key << 32 | ~index), distinct
    int* chosen = reinterpret_cast<int*>(hist);                                 // [CAP] index of a selected entry
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = p.k;
    unsigned w[NV], largest = 0u;
#pragma unroll
    for (int u = 0; u < NV; ++u) w[u] = tid + u * THREADS < p.d ? ws[tid + u * THREADS] : 0u;
#pragma unroll
    for (int u = 0; u < NV; ++u) largest = max(largest, w[u]);
    {
        const unsigned hi = __reduce_max_sync(0xffffffffu, largest), lo = __reduce_min_sync(0xffffffffu, largest);
        if (lane == 0) { wmax[warp] = hi; wmin[warp] = lo; }
    }
    __syncthreads();
    unsigned floor = __reduce_min_sync(0xffffffffu, wmin[lane < WARPS ? lane : 0]);
    unsigned top = __reduce_max_sync(0xffffffffu, wmax[lane < WARPS ? lane : 0]);            // largest: of floor k or more are at or above it, of top + 1 none
    floor = bisect_floor(floor, top, k, [&](unsigned key) { return __syncthreads_count(largest >= key); }) & ~1u;      // both signs of a magnitude
    unsigned n = 0u;
#pragma unroll
    for (int u = 0; u < NV; ++u) n += w[u] >= floor && tid + u * THREADS < p.d ? 1u : 0u;
    const unsigned upto = warp_incl_scan(n);
    unsigned at = lane == 31 && upto ? atomicAdd(&list_n, upto) : 0u;
    at = __shfl_sync(0xffffffffu, at, 31) + upto - n;
    if (n != 0u) {
#pragma unroll
        for (int u = 0; u < NV; ++u)
            if (w[u] >= floor && tid + u * THREADS < p.d) {
                if (at < CAP) cand[at] = ((unsigned long long)(w[u] >> 1) << 32) | (0xffffffffu - (unsigned)(tid + u * THREADS));
                ++at;
            }
    }
    __syncthreads();
    const unsigned c = list_n;
    if (c > CAP) return false;
    const unsigned log_lanes = c <= THREADS / 8 ? 3u : (c <= THREADS / 4 ? 2u : 1u), lanes = 1u << log_lanes, sub = (unsigned)tid & (lanes - 1u);
    const unsigned e = (unsigned)tid >> log_lanes;
    const bool have = e < c, first = have && sub == 0u;
    const unsigned long long mine = have ? cand[e] : 0ull;
    const int j = (int)(0xffffffffu - (unsigned)mine);
    float* app = p.apply ? p.apply + (i64)vec * p.pitch_apply : nullptr;
    const float old = MODE == TC_DIFF && first && app ? app[j] : 0.f;          // (arrives while the entries are ranked)
    unsigned above = 0u;
#pragma unroll 4
    for (unsigned o = sub; o < c; o += lanes) above += cand[o] > mine ? 1u : 0u;
    for (unsigned off = 1u; off < lanes; off <<= 1) above += __shfl_xor_sync(0xffffffffu, above, off);
    const bool sel = have && above < (unsigned)k;
    if (first) chosen[e] = sel ? j : 0x7fffffff;
    __syncthreads();
    unsigned pos = 0u;
#pragma unroll 4
    for (unsigned o = sub; o < c; o += lanes) pos += chosen[o] < j ? 1u : 0u;
    for (unsigned off = 1u; off < lanes; off <<= 1) pos += __shfl_xor_sync(0xffffffffu, pos, off);
    if (sel && first) {
        const unsigned wv = ws[j];
        const float v = __uint_as_float(__funnelshift_r(wv, wv, 1));
        p.idx_out[(i64)vec * k + pos] = j; p.val_out[(i64)vec * k + pos] = v;
        flag_nonfinite(p.status, v);
        if (above + 1u == (unsigned)k && p.cut_out) p.cut_out[vec] = mine;
        if (app) app[j] = MODE == TC_DIFF ? __fadd_rn(old, v) : (MODE == TC_PLAIN ? __fadd_rn(0.f, v) : __fsub_rn(v, v));
    }
    return true;
}

// The same for a cluster: every block finds a floor that at least k / C of its entries reach, the lowest of the C floors is the cluster's (k
// entries or more reach it), and the entries from there on are handed around.  Every block finds the k-th of them by a histogram of 2,047
// even steps between the floor and the maximum and by ranking the few in the deciding step, and places its own through a bitmap of its
// share.  Two cluster barriers as without, but no atomic per entry, no histogram over distributed shared memory, no sweep for the list and
// none for the compaction.  (Every own candidate ranked against all: a quarter of a million comparisons per block.)
// 20 x 70,001, Top-700: 14.0 -> 11.5 us; 1 x 81,822, Top-818: 16.2 -> 14.0 with the call.
// False (for the whole cluster): too many candidates, as where the large entries sit together in one block's share.
constexpr int TC_FEW_OWN = 1024, TC_FEW_ALL = 2048;

template <int MODE, int C, int THREADS>
__device__ __forceinline__ bool tc_few_cluster(const TcArgs& p, int vec, int rank, int j0, int len, const unsigned* ws, unsigned* hist, unsigned* list,
                                               unsigned long long* all, unsigned largest, unsigned* wmin, unsigned* wmax, unsigned* wsum, unsigned* found,
                                               unsigned& list_n) {
    namespace cg = cooperative_groups;
    constexpr int WARPS = THREADS / 32, BITMAP = TC_MAX_SLICE / 32, GROUPS = BITMAP / 4;
    static_assert(BITMAP + GROUPS <= TC_BINS, "bitmap and its prefix sums take the histogram's place");
    __shared__ unsigned floor_sh, top_sh, before_sh, step_n, scratch[33];
    __shared__ unsigned long long kth_sh, step_sh[TC_RANKED];
    cg::cluster_group cluster = cg::this_cluster();
    unsigned long long* cand = reinterpret_cast<unsigned long long*>(list);     // this block's (key << 32 | ~index), [TC_FEW_OWN]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = p.k, share = (k + C - 1) / C;
    {
        const unsigned hi = __reduce_max_sync(0xffffffffu, largest), lo = __reduce_min_sync(0xffffffffu, largest);
        if (lane == 0) { wmax[warp] = hi; wmin[warp] = lo; }
        if (tid == 0) { before_sh = 0u; step_n = 0u; }
        hist[tid] = 0u; hist[tid + THREADS] = 0u;
        static_assert(TC_BINS == 2 * THREADS, "two bins per thread");
    }
    __syncthreads();
    unsigned floor = __reduce_min_sync(0xffffffffu, wmin[lane]), top = __reduce_max_sync(0xffffffffu, wmax[lane]);
    static_assert(WARPS == 32, "a lane per warp");
    if (tid == 0) top_sh = top;
    floor = bisect_floor(floor, top, share, [&](unsigned key) { return __syncthreads_count(largest >= key); });
    if (tid == 0) floor_sh = floor & ~1u;                                       // both signs of a magnitude
    cluster.sync();
    floor = 0xffffffffu; top = 0u;
#pragma unroll
    for (int r = 0; r < C; ++r) { floor = min(floor, *cluster.map_shared_rank(&floor_sh, r)); top = max(top, *cluster.map_shared_rank(&top_sh, r)); }
    if (largest >= floor) {
#pragma unroll 4
        for (int j = tid; j < len; j += THREADS) {
            const unsigned w = ws[j];
            if (w >= floor) {
                const unsigned at = atomicAdd(&list_n, 1u);
                if (at < (unsigned)TC_FEW_OWN) cand[at] = ((unsigned long long)(w >> 1) << 32) | (0xffffffffu - (unsigned)(j0 + j));
            }
        }
    }
    cluster.sync();
    unsigned n_of[C], total = 0u, first = 0u;
    bool fits = true;
#pragma unroll
    for (int r = 0; r < C; ++r) {
        n_of[r] = *cluster.map_shared_rank(&list_n, r);
        fits = fits && n_of[r] <= (unsigned)TC_FEW_OWN;
        if (r < rank) first += n_of[r];
        total += n_of[r];
    }
    if (!fits || total > (unsigned)TC_FEW_ALL) return false;
    const unsigned c = list_n, low = floor >> 1;
    int shift = 0;
    while ((((top >> 1) - low) >> shift) >= (unsigned)TC_BINS - 1u) ++shift;
    auto step_of = [&](unsigned long long x) { return 1u + (((unsigned)(x >> 32) - low) >> shift); };
#pragma unroll 1
    for (unsigned e = tid; e < total; e += THREADS) {
        unsigned off = e; int from = 0;
#pragma unroll
        for (int r = 0; r < C - 1; ++r) if (from == r && off >= n_of[r]) { off -= n_of[r]; from = r + 1; }
        const unsigned long long x = cluster.map_shared_rank(cand, from)[off];
        all[e] = x;
        atomicAdd(&hist[step_of(x)], 1u);
    }
    // this block's own, one per thread
    const bool have = tid < (int)c;
    const unsigned long long mine = have ? cand[tid] : 0ull;
    const int j = (int)(0xffffffffu - (unsigned)mine);
    float* app = p.apply ? p.apply + (i64)vec * p.pitch_apply : nullptr;
    const float old = MODE == TC_DIFF && have && app ? app[j] : 0.f;
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");       // done with the other blocks' memory
    tc_find_bin(hist, (unsigned)k, total, wsum, found);
    const unsigned step = found[0], need = (unsigned)k - found[1], pop = found[2];
    if (pop > (unsigned)TC_RANKED) {                                            // (the same in all blocks)
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        return false;
    }
#pragma unroll 1
    for (unsigned e = tid; e < total; e += THREADS) {
        const unsigned long long x = all[e];
        if (step_of(x) == step) step_sh[atomicAdd(&step_n, 1u)] = x;
    }
    hist[tid] = 0u; hist[tid + THREADS] = 0u;                                   // from here on the bitmap
    __syncthreads();
    if (tid < (int)pop) {
        const unsigned long long x = step_sh[tid];
        unsigned above = 0u;
        for (unsigned o = 0; o < pop; ++o) above += step_sh[o] > x ? 1u : 0u;
        if (above + 1u == need) kth_sh = x;
    }
    __syncthreads();
    const unsigned long long kth = kth_sh;
    const bool sel = have && mine >= kth;
    if (sel) atomicOr(&hist[(j - j0) >> 5], 1u << ((j - j0) & 31));
    unsigned before = 0u;                                                       // selected entries of the blocks before this one
    for (unsigned o = tid; o < first; o += THREADS) before += all[o] >= kth ? 1u : 0u;
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 0 && before) atomicAdd(&before_sh, before);
    __syncthreads();
    {
        const uint4 w = tid < GROUPS ? reinterpret_cast<const uint4*>(hist)[tid] : make_uint4(0u, 0u, 0u, 0u);
        unsigned sum;
        const unsigned up = block_excl_scan((unsigned)(__popc(w.x) + __popc(w.y) + __popc(w.z) + __popc(w.w)), scratch, sum);
        if (tid < GROUPS) hist[BITMAP + tid] = up;
    }
    __syncthreads();
    if (sel) {
        const int word = (j - j0) >> 5;
        unsigned pos = before_sh + hist[BITMAP + (word >> 2)] + (unsigned)__popc(hist[word] & ((1u << ((j - j0) & 31)) - 1u));
        for (int q = word & ~3; q < word; ++q) pos += (unsigned)__popc(hist[q]);
        const unsigned wv = ws[j - j0];
        const float v = __uint_as_float(__funnelshift_r(wv, wv, 1));
        p.idx_out[(i64)vec * k + pos] = j; p.val_out[(i64)vec * k + pos] = v;
        flag_nonfinite(p.status, v);
        if (mine == kth && p.cut_out) p.cut_out[vec] = mine;
        if (app) app[j] = MODE == TC_DIFF ? __fadd_rn(old, v) : (MODE == TC_PLAIN ? __fadd_rn(0.f, v) : __fsub_rn(v, v));
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");         // nobody reads this block's list any more
    return true;
}

// STREAM: the vector is longer than the cluster's shared memory; it stays in global memory and every sweep reads it again.
// REDO: of vectors that are flagged, one after the other.
// GRAD > 0: the local gradients are formed from the tile partials on the way in (no kernel and no array for them), by a cluster of GRAD
// blocks that each take a share of the columns and leave v in the first one's shared memory; that one selects alone (C = 1).
template <int MODE, int C, int THREADS, bool STREAM, int GRAD, bool REDO = STREAM>
__device__ __forceinline__ void tc_vector(const TcArgs& p, int vec) {
    namespace cg = cooperative_groups;
    constexpr int WARPS = THREADS / 32;
    extern __shared__ __align__(16) unsigned char tc_smem[];
    unsigned* ws = reinterpret_cast<unsigned*>(tc_smem);            // [slice] bits of v rotated left by one
    unsigned* hist = ws + (STREAM ? 0 : p.slice);                   // [TC_BINS] this block's histogram
    unsigned* list = hist + TC_BINS;                                // [TC_LIST] this block's keys of the deciding bin
    unsigned* all = C > 1 ? list + TC_LIST : list;                  // [TC_LIST] the lists of all blocks
    unsigned* hsum = C > 1 ? all + TC_LIST : hist;                  // [TC_BINS] the cluster's histogram (own bins first, then all)
    unsigned char* lwarp = reinterpret_cast<unsigned char*>(C > 1 ? hsum + TC_BINS : all + TC_LIST);    // [TC_LIST] warp of a listed key
    __shared__ unsigned list_n, above_n;                            // this block: keys in its list, entries in higher bins
    __shared__ unsigned found[3], result[2], before_sh[2];
    __shared__ unsigned wsum[8], wgt[WARPS], weq[WARPS];

    __shared__ uint2 blk_counts;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = C > 1 ? (int)cluster.block_rank() : 0;
    auto sync_all = [&]() { if (C > 1) cluster.sync(); else __syncthreads(); };

    const int j0 = (int)min((i64)rank * p.slice, (i64)p.d), len = min(p.slice, p.d - j0);
    const bool few = C == 1 && !STREAM && p.d <= THREADS * tc_few_values(THREADS) &&
                     p.k <= few_limit(THREADS, p.d, gridDim.x <= 148u * (GRAD > 1 ? GRAD : 1), GRAD > 0);
    // (Many blocks with a few entries each: their floors are uneven, the bisection in their tails is long, and a share of some ten entries per
    // thread is counted quickly.  Rounds, us, with the histogram / this way: 4 x 452,034 Top-452 in sixteen blocks 29.2 / 30.0, 16 x 79,311
    // Top-79 in eight 29.3 / 31.5; 20 x 116,750 Top-116 in four 24.9 / 22.9, 1 x 81,822 Top-818 in eight 16.2 / 14.0.  Eight rounds: 37 x 60,000 in four
    // Top-10 210 / 226, Top-60 241 / 243, Top-200 323 / 300; 70 x 30,000 in two Top-8 150 / 158, Top-30 169 / 172, Top-100 301 / 294.)
    constexpr bool MAY_FEW = C > 1 && C <= 8 && !STREAM && !REDO;
    const bool few_cluster = MAY_FEW && p.k <= TC_FEW_OWN && (p.k + C - 1) / C <= THREADS / 5 && p.k >= (C <= 4 ? 20 : 64) * C;
    unsigned largest = 0u;
    auto clear = [&]() {
#pragma unroll 1
        for (int q = tid; q < TC_BINS; q += THREADS) { hist[q] = 0u; if (C > 1) hsum[q] = 0u; }
    };
    if (!few && !few_cluster) clear();
    for (int j = len + tid; !STREAM && j < p.slice && j < len + 128; j += THREADS) ws[j] = 0u;       // the tail of the last tile
    if (tid < WARPS) { wgt[tid] = 0u; weq[tid] = 0u; }
    if (tid == 0) { list_n = 0u; above_n = 0u; before_sh[0] = 0u; before_sh[1] = 0u; result[0] = 0xffffffffu; }
    __syncthreads();
    if (C > 1 || GRAD > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");       // hsum is empty; all blocks run
    constexpr bool LATE = GRAD > 0 && THREADS == 512;               // see where it is used
    int t0 = 0, t1 = 0;
    i64 m_all = 0;
    // the tile table is complete before the gradient kernel in front of a wide selection lets anything start (see grad_wide_kernel)
    auto tables = [&]() { t0 = p.tile_begin[vec]; t1 = p.tile_begin[vec + 1]; m_all = p.row_off[vec + 1] - p.row_off[vec]; };
    if (LATE) tables();
    if (!STREAM) { if (!LATE) pdl_trigger(); pdl_wait(); }
    if (GRAD > 0 && !LATE) tables();
    const float* __restrict__ av = GRAD ? nullptr : pdl_ptr(p.a + (i64)vec * p.pitch_a + j0);
    float* bv = MODE == TC_PLAIN ? nullptr : p.b + (i64)vec * p.pitch_b + j0;
    float* dense = MODE == TC_PLAIN && !STREAM && p.apply ? p.apply + (i64)vec * p.pitch_apply + j0 : nullptr;
    // entries of bin 0 (zeros and the smallest magnitudes) are not counted: what the other bins leave over is theirs
    auto count = [&](unsigned w) { if (w >> 21) atomicAdd(&hist[w >> 21], 1u); };
    auto take = [&](int j, float a, float b, auto use) {
        float v = a;
        if (MODE == TC_DIFF) v = __fsub_rn(a, b);
        if (MODE == TC_EF) { v = __fadd_rn(b, __fmul_rn(p.gamma, a)); bv[j] = v; }
        if (MODE == TC_SENT) v = b;
        const unsigned w = __funnelshift_l(__float_as_uint(v), __float_as_uint(v), 1);
        if (MODE == TC_PLAIN && dense) dense[j] = 0.f;
        if (GRAD > 1) { cluster.map_shared_rank(ws, 0)[j] = w; return; }
        if (!STREAM) ws[j] = w;
        if (decltype(use)::value == TC_LARGEST) largest = max(largest, w);
        if (decltype(use)::value == TC_COUNT) count(w);
    };
    if (GRAD > 0) {
        const i64 m = p.batch_rows > 0 ? (i64)p.batch_rows : m_all;
        const int share = GRAD > 1 ? (len + GRAD - 1) / GRAD : len;
        const int c0 = GRAD > 1 ? (int)cluster.block_rank() * share : 0, c1 = min(c0 + share, len);
        if (GRAD > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        const float* partial = pdl_ptr(p.partial);
        // two columns at a time, a round of eight tiles of both on its way while the one before is added up (a tile behind the last one
        // is read again and left out)
        constexpr int U = 2, Q = GRAD_FINISH_LANES;
#pragma unroll 1
        for (int jj = c0 + tid; jj < c1; jj += U * THREADS) {
            const int js[U] = {jj, min(jj + THREADS, c1 - 1)};
            float acc[U][Q], next[U][Q], b[U], xj[U];
            auto fetch = [&](int t) {
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const float* row = partial + (i64)min(t + q, t1 - 1) * p.ld;
#pragma unroll
                    for (int u = 0; u < U; ++u) next[u][q] = __ldcg(row + js[u]);
                }
            };
            if (t0 < t1) fetch(t0);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                b[u] = MODE == TC_PLAIN ? 0.f : bv[js[u]]; xj[u] = p.x[js[u]];
#pragma unroll
                for (int q = 0; q < Q; ++q) acc[u][q] = 0.f;
            }
#pragma unroll 1
            for (int t = t0; t < t1; t += Q) {
                float w[U][Q];
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int q = 0; q < Q; ++q) w[u][q] = next[u][q];
                if (t + Q < t1) fetch(t + Q);
#pragma unroll
                for (int q = 0; q < Q; ++q)
#pragma unroll
                    for (int u = 0; u < U; ++u) acc[u][q] = t + q < t1 ? __fadd_rn(acc[u][q], w[u][q]) : acc[u][q];
            }
            float g[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
#pragma unroll
                for (int q = 1; q < Q; ++q) acc[u][0] = __fadd_rn(acc[u][0], acc[u][q]);
                g[u] = __fadd_rn(m > 0 ? __fdiv_rn(acc[u][0], (float)m) : 0.f, regulariser_grad(p.lambda, xj[u]));
            }
            auto both = [&](auto use) { take(js[0], g[0], b[0], use); if (jj + THREADS < c1) take(js[1], g[1], b[1], use); };
            if (few) both(TcUse<TC_KEEP>()); else both(TcUse<TC_COUNT>());
        }
        // Behind the aggregation waits grad_wide_kernel, which fetches rows as soon as it is placed: not before this kernel's own
        // loads are through (20 x 5,001: 38.4 us an iteration instead of 39.4).
        if (LATE) { __syncthreads(); pdl_trigger(); }
        if (GRAD > 1) {
            cluster.sync();
            if (cluster.block_rank() != 0) return;
            if (!few) for (int j = tid; j < len; j += THREADS) count(ws[j]);
        }
    } else {
        constexpr int U = THREADS == 1024 ? 8 : 4;
        auto sweep = [&](auto use) {
            int j = tid;
#pragma unroll 1
            for (; j + (U - 1) * THREADS < len; j += U * THREADS) {
                float a[U], b[U];
#pragma unroll
                for (int u = 0; u < U; ++u) { a[u] = MODE == TC_SENT ? 0.f : av[j + u * THREADS]; b[u] = MODE == TC_PLAIN ? 0.f : bv[j + u * THREADS]; }
#pragma unroll
                for (int u = 0; u < U; ++u) take(j + u * THREADS, a[u], b[u], use);
            }
#pragma unroll 1
            for (; j < len; j += THREADS) take(j, MODE == TC_SENT ? 0.f : av[j], MODE == TC_PLAIN ? 0.f : bv[j], use);
        };
        if (MAY_FEW && few_cluster) sweep(TcUse<MAY_FEW ? TC_LARGEST : TC_COUNT>());
        else if (C == 1 && few) sweep(TcUse<C == 1 ? TC_KEEP : TC_COUNT>());
        else sweep(TcUse<TC_COUNT>());
    }
    constexpr int OWN = TC_BINS / C;                                // bins summed by one block
    auto sum_histograms = [&]() {                                   // hist of all blocks -> hsum
        __syncthreads();
        if (C > 1) {
            // hsum of every block is empty here
#pragma unroll 1
            for (int q = tid; q < TC_BINS; q += THREADS) {
                const unsigned c = hist[q];
                if (c) atomicAdd(cluster.map_shared_rank(hsum, q / OWN) + q, c);
            }
            cluster.sync();
#pragma unroll 1
            for (int q = tid; q < TC_BINS; q += THREADS)            // hist becomes the cluster's histogram
                hist[q] = cluster.map_shared_rank(hsum, q / OWN)[q];
            __syncthreads();
        }
    };
    if constexpr (C == 1 && !STREAM) if (few) {
        __syncthreads();
        if (tc_few<MODE, THREADS>(p, vec, ws, hist, list, wgt, weq, list_n)) return;
        __syncthreads();
        clear();
        if (tid == 0) list_n = 0u;
        if (tid < WARPS) { wgt[tid] = 0u; weq[tid] = 0u; }
        __syncthreads();
#pragma unroll 1
        for (int j = tid; j < len; j += THREADS) { const unsigned w = ws[j]; if (w >> 21) atomicAdd(&hist[w >> 21], 1u); }
    }
    if (C > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if constexpr (MAY_FEW) if (few_cluster) {
        if (tc_few_cluster<MODE, C, THREADS>(p, vec, rank, j0, len, ws, hist, list, reinterpret_cast<unsigned long long*>(all), largest, wgt, weq, wsum, found, list_n))
            return;
        cluster.sync();                                             // (nobody reads this block's words any more)
        clear();
        if (tid == 0) list_n = 0u;
        if (tid < WARPS) { wgt[tid] = 0u; weq[tid] = 0u; }
        cluster.sync();
#pragma unroll 1
        for (int j = tid; j < len; j += THREADS) { const unsigned w = ws[j]; if (w >> 21) atomicAdd(&hist[w >> 21], 1u); }
    }
    sum_histograms();
    tc_find_bin(hist, (unsigned)p.k, (unsigned)p.d, wsum, found);
    const unsigned bin0 = found[0], pop0 = found[2];
    unsigned need = (unsigned)p.k - found[1];
    const bool listed = pop0 <= (unsigned)TC_LIST;
    // the word(s) of an entry (of four consecutive ones) again, zero behind the end
    auto word = [&](int j) {
        if (!STREAM) return ws[j];
        if (j >= len) return 0u;
        const float v = MODE == TC_SENT ? bv[j] : (MODE == TC_DIFF ? __fsub_rn(av[j], bv[j]) : av[j]);
        return __funnelshift_l(__float_as_uint(v), __float_as_uint(v), 1);
    };
    auto word4 = [&](int j) {
        if (!STREAM) return reinterpret_cast<const uint4*>(ws)[j >> 2];
        return make_uint4(word(j), word(j + 1), word(j + 2), word(j + 3));
    };
    // warp w owns the entries [w * chunk, (w + 1) * chunk) of the slice, in tiles of 128, four consecutive ones per lane
    const int chunk = ((len + WARPS - 1) / WARPS + 127) & ~127;
    const int w0 = min(warp * chunk, len), w1 = min(w0 + chunk, len);
    auto valid4 = [&](int j) { return j + 3 < w1 ? 15u : (j < w1 ? (1u << (w1 - j)) - 1u : 0u); };
    unsigned T, need_ties;
    unsigned gt_before = 0u, eq_before = 0u;                        // in the blocks before this one
    if (listed) {
        unsigned above = 0u;
        const unsigned lo = bin0 << 21;
#pragma unroll 1
        for (int base = w0; base < w1; base += 128) {
            const int j = base + 4 * lane;
            const uint4 w = word4(j);
            unsigned hit = 0u;
            // (w - lo) < 2^21: in the bin; beyond that and not below lo: above it
            const unsigned o[4] = {w.x - lo, w.y - lo, w.z - lo, w.w - lo};
            hit = (o[0] < (1u << 21) ? 1u : 0u) | (o[1] < (1u << 21) ? 2u : 0u) | (o[2] < (1u << 21) ? 4u : 0u) | (o[3] < (1u << 21) ? 8u : 0u);
            above += (w.x >= lo ? 1u : 0u) + (w.y >= lo ? 1u : 0u) + (w.z >= lo ? 1u : 0u) + (w.w >= lo ? 1u : 0u);
            if (lo == 0u || hit) {
                const unsigned ok = valid4(j);                      // zeros behind the end belong to no bin
                if (lo == 0u) above -= 4u - (unsigned)__popc(ok);
                hit &= ok;
                above -= (unsigned)__popc(hit);
                while (hit != 0u) {
                    const int e = __ffs((int)hit) - 1;
                    hit &= hit - 1u;
                    const unsigned at = atomicAdd(&list_n, 1u);
                    list[at] = word(j + e) >> 1;
                    lwarp[at] = (unsigned char)warp;
                }
            }
        }
        above = __reduce_add_sync(0xffffffffu, above);
        if (lane == 0) {
            if (above) atomicAdd(&wgt[warp], above);
            if (C > 1 && above) atomicAdd(&above_n, above);
        }
        sync_all();
        unsigned first = 0u;                                        // where this block's keys start in `all`
        if (C > 1) {
            unsigned n_of[C], ab[C];
#pragma unroll
            for (int r = 0; r < C; ++r) { n_of[r] = *cluster.map_shared_rank(&list_n, r); ab[r] = *cluster.map_shared_rank(&above_n, r); }
#pragma unroll
            for (int r = 0; r < C; ++r) if (r < rank) { first += n_of[r]; gt_before += ab[r]; }
#pragma unroll 1
            for (unsigned e = tid; e < pop0; e += THREADS) {
                unsigned off = e; int from = 0;
#pragma unroll
                for (int r = 0; r < C - 1; ++r) if (from == r && off >= n_of[r]) { off -= n_of[r]; from = r + 1; }
                all[e] = cluster.map_shared_rank(list, from)[off];
            }
        }
        if (tid < 4 && pop0 + tid < (unsigned)TC_LIST) all[pop0 + tid] = 0u;        // read in groups of four below
        __syncthreads();
        if (pop0 <= (unsigned)TC_RANKED) {
            // one key per thread: T is the smallest key that fewer than `need` keys exceed
            const bool have = tid < (int)pop0;
            const unsigned mine = have ? all[tid] : 0u;
            unsigned gt = 0u;
            if (have) {
#pragma unroll 2
                for (unsigned o = 0; o < (pop0 + 3u) >> 2; ++o) {
                    const uint4 x = reinterpret_cast<const uint4*>(all)[o];
                    gt += x.x > mine ? 1u : 0u; gt += x.y > mine ? 1u : 0u; gt += x.z > mine ? 1u : 0u; gt += x.w > mine ? 1u : 0u;
                }
                if (gt < need) atomicMin(&result[0], mine);
            }
            __syncthreads();
            T = result[0];
            if (have && mine == T) result[1] = need - gt;
            __syncthreads();
            need_ties = result[1];
        } else {
            unsigned prefix = bin0, pop = pop0;
#pragma unroll 1
            for (int shift = 9; shift >= 0; shift -= 9) {           // bits 19..9, then 8..0
#pragma unroll 1
                for (int q = tid; q < TC_BINS; q += THREADS) hist[q] = 0u;
                __syncthreads();
                const int up = shift == 9 ? 20 : 9;
                const unsigned mask = shift == 9 ? 2047u : 511u;
#pragma unroll 1
                for (unsigned e = tid; e < pop0; e += THREADS) {
                    const unsigned key = all[e], bin = (key >> shift) & mask;
                    if ((key >> up) == prefix && bin) atomicAdd(&hist[bin], 1u);
                }
                __syncthreads();
                tc_find_bin(hist, need, pop, wsum, found);
                prefix = (prefix << (shift == 9 ? 11 : 9)) | found[0]; need -= found[1]; pop = found[2];
            }
            T = prefix; need_ties = need;
        }
        // listed keys above and at T: this block's by warp, those of the blocks before it in total
        const unsigned mine_n = C > 1 ? list_n : pop0;
#pragma unroll 1
        for (unsigned e = tid; e < mine_n; e += THREADS) {
            const unsigned key = list[e];
            if (key > T) atomicAdd(&wgt[lwarp[e]], 1u);
            else if (key == T) atomicAdd(&weq[lwarp[e]], 1u);
        }
        if (C > 1) {
#pragma unroll 1
            for (unsigned e = tid; e < first; e += THREADS) {
                const unsigned key = all[e];
                if (key >= T) atomicAdd(&before_sh[key == T ? 1 : 0], 1u);
            }
        }
        __syncthreads();
        if (C > 1) { gt_before += before_sh[0]; eq_before += before_sh[1]; }
    } else {
        unsigned prefix = bin0, pop = pop0;
#pragma unroll 1
        for (int shift = 9; shift >= 0; shift -= 9) {
            sync_all();                                             // everybody has read the histograms
#pragma unroll 1
            for (int q = tid; q < TC_BINS; q += THREADS) { hist[q] = 0u; if (C > 1) hsum[q] = 0u; }
            sync_all();
            const int up = shift == 9 ? 20 : 9;
            const unsigned mask = shift == 9 ? 2047u : 511u;
#pragma unroll 1
            for (int j = tid; j < len; j += THREADS) {
                const unsigned key = word(j) >> 1, bin = (key >> shift) & mask;
                if ((key >> up) == prefix && bin) atomicAdd(&hist[bin], 1u);
            }
            sum_histograms();
            tc_find_bin(hist, need, pop, wsum, found);
            prefix = (prefix << (shift == 9 ? 11 : 9)) | found[0]; need -= found[1]; pop = found[2];
        }
        T = prefix; need_ties = need;
        if (rank == 0 && tid == 0 && p.slow_count && pop > (unsigned)TC_LIST) atomicAdd(p.slow_count, 1u);
        unsigned gt = 0u, eq = 0u;
#pragma unroll 1
        for (int j = w0 + lane; j < w1; j += 32) { const unsigned key = word(j) >> 1; gt += key > T ? 1u : 0u; eq += key == T ? 1u : 0u; }
        gt = __reduce_add_sync(0xffffffffu, gt); eq = __reduce_add_sync(0xffffffffu, eq);
        if (lane == 0) { wgt[warp] = gt; weq[warp] = eq; }
        __syncthreads();
        // the counts of the blocks before this one have to be handed around
        if (C > 1) {
            const unsigned bg = __reduce_add_sync(0xffffffffu, lane < WARPS ? wgt[lane] : 0u);
            const unsigned be = __reduce_add_sync(0xffffffffu, lane < WARPS ? weq[lane] : 0u);
            if (tid == 0) blk_counts = make_uint2(bg, be);
            sync_all();
            for (int r = 0; r < rank; ++r) { const uint2 o = *cluster.map_shared_rank(&blk_counts, r); gt_before += o.x; eq_before += o.y; }
        }
    }
    if (C > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");     // done with the other blocks' memory

    // ordered compaction
    if (wgt[warp] + weq[warp] != 0u) {
        gt_before += __reduce_add_sync(0xffffffffu, lane < warp ? wgt[lane] : 0u);
        eq_before += __reduce_add_sync(0xffffffffu, lane < warp ? weq[lane] : 0u);
        int* __restrict__ io = p.idx_out + (i64)vec * p.k;
        float* __restrict__ vo = p.val_out + (i64)vec * p.k;
        float* app = p.apply ? p.apply + (i64)vec * p.pitch_apply + j0 : nullptr;
        const unsigned lo = T << 1;
#pragma unroll 1
        for (int base = w0; base < w1; base += 128) {
            const int j = base + 4 * lane;
            const uint4 w = word4(j);
            if (!__any_sync(0xffffffffu, max(max(w.x, w.y), max(w.z, w.w)) >= lo)) continue;
            unsigned m = (w.x >= lo ? 1u : 0u) | (w.y >= lo ? 2u : 0u) | (w.z >= lo ? 4u : 0u) | (w.w >= lo ? 8u : 0u);
            m &= valid4(j);
            unsigned ties = ((w.x >> 1) == T ? 1u : 0u) | ((w.y >> 1) == T ? 2u : 0u) | ((w.z >> 1) == T ? 4u : 0u) | ((w.w >> 1) == T ? 8u : 0u);
            ties &= m;
            // entries above T (low half) and at T (high half) in lower lanes
            const unsigned mine = (unsigned)__popc(m & ~ties) | ((unsigned)__popc(ties) << 16);
            const unsigned incl = warp_incl_scan(mine), excl = incl - mine;
            const unsigned tile = __shfl_sync(0xffffffffu, incl, 31);
            unsigned g0 = gt_before + (excl & 0xffffu), e0 = eq_before + (excl >> 16);
            while (m != 0u) {
                const int e = __ffs((int)m) - 1;
                m &= m - 1u;
                const bool tie = (ties >> e) & 1u;
                if (!tie || e0 < need_ties) {
                    const unsigned wv = word(j + e);
                    const float v = __uint_as_float(__funnelshift_r(wv, wv, 1));
                    const unsigned pos = g0 + min(e0, need_ties);
                    io[pos] = j0 + j + e; vo[pos] = v;
                    flag_nonfinite(p.status, v);
                    if (tie && e0 + 1u == need_ties && p.cut_out)
                        p.cut_out[vec] = ((unsigned long long)T << 32) | (0xffffffffu - (unsigned)(j0 + j + e));
                    if (app) app[j + e] = MODE == TC_DIFF ? __fadd_rn(app[j + e], v) : (MODE == TC_PLAIN ? __fadd_rn(0.f, v) : __fsub_rn(v, v));
                }
                g0 += tie ? 0u : 1u; e0 += tie ? 1u : 0u;
            }
            gt_before += tile & 0xffffu; eq_before += tile >> 16;
        }
    }
    if (C > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (REDO && p.tile_off) {
        cluster.sync();                                              // the message is complete and visible to the cluster
        int* off = p.tile_off + (i64)vec * (p.ntiles + 1);
        const int* io = pdl_ptr(p.idx_out + (i64)vec * p.k);
        for (int b = rank * THREADS + tid; b <= p.ntiles; b += C * THREADS) {
            const i64 bound = (i64)b * p.tile;
            int lo = 0, hi = p.k;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if ((i64)__ldcg(&io[mid]) < bound) lo = mid + 1; else hi = mid;
            }
            off[b] = lo;
        }
    }
}

// (512 threads: left alone the compiler takes 40 registers; ten rounds of 20 x 8,192 Top-128 158.7 us with these, 149.5 with 56.)
template <int MODE, int C, int THREADS, bool STREAM = false, int GRAD = 0, bool REDO = STREAM>
__global__ void __launch_bounds__(THREADS, THREADS == 512 && GRAD == 0 ? 2 : 0)
tc_topk_kernel(const __grid_constant__ TcArgs p) {
    if (REDO) {
        // a few clusters look through the flags: as a rule there is nothing to do
        pdl_trigger();
        pdl_wait();
        for (int vec = (int)(blockIdx.x / (unsigned)C); vec < p.batch; vec += (int)(gridDim.x / (unsigned)C))
            if (p.flag[(i64)vec * p.flag_pitch] != 0u) {
                tc_vector<MODE, C, THREADS, STREAM, GRAD, REDO>(p, vec);
                cooperative_groups::this_cluster().sync();
            }
    } else {
        tc_vector<MODE, C, THREADS, STREAM, GRAD>(p, (int)(blockIdx.x / (unsigned)(GRAD > 1 ? GRAD : C)));
    }
}

// The exact fallback of both selections of EF21+ in one launch: flags of the vectors a - b (pm), then of the vectors a (pb).
template <int C, int THREADS>
__global__ void __launch_bounds__(THREADS)
tc_pair_kernel(const __grid_constant__ TcArgs pm, const __grid_constant__ TcArgs pb) {
    pdl_trigger();
    pdl_wait();
    for (int v = (int)(blockIdx.x / (unsigned)C); v < 2 * pm.batch; v += (int)(gridDim.x / (unsigned)C)) {
        const bool plain = v >= pm.batch;
        const int vec = plain ? v - pm.batch : v;
        const TcArgs& p = plain ? pb : pm;
        if (p.flag[(i64)vec * p.flag_pitch] == 0u) continue;
        if (plain) tc_vector<TC_PLAIN, C, THREADS, true, 0>(pb, vec);
        else tc_vector<TC_DIFF, C, THREADS, true, 0>(pm, vec);
        cooperative_groups::this_cluster().sync();
    }
}

}  // namespace ef21
