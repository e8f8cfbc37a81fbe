// Floor under the largest keys by bisection: what the selections of few entries start from (topk_cluster.cuh), and how many are few.  Free of CUDA apart from the
// qualifier, so that a host compiler takes it too and the search can be run over any keys without a GPU.
#pragma once
#ifdef __CUDACC__
#define EF21_BISECT_FN __device__ __forceinline__
#else
#define EF21_BISECT_FN inline
#endif

namespace ef21 {

// Between two keys, the upper one of the two in the middle.  (Not floor + (top - floor + 1) / 2: for floor 0 and a key with all bits
// set, a NaN, the sum wraps to 0 and the search stands still.)
EF21_BISECT_FN unsigned bisect_middle(unsigned floor, unsigned top) { return top - (top - floor) / 2u; }

// A key that `need` to 5/4 need + 4 of the counted ones reach, or, where ties leave no such key, the greatest one that at least `need`
// of them reach.  At least `need` reach `floor` and none lies above `top`; count(key) tells how many reach a key.  A step leaves at most
// half of the distance, rounded down, so that 32 of them always do; the bound holds whatever count returns.
template <typename Count>
EF21_BISECT_FN unsigned bisect_floor(unsigned floor, unsigned top, int need, Count count) {
#pragma unroll 1
    for (int step = 0; step < 32 && floor < top; ++step) {
        const unsigned mid = bisect_middle(floor, top);
        const int n = count(mid);
        if (n >= need) { floor = mid; if (n <= need + need / 4 + 4) break; }
        else top = mid - 1u;
    }
    return floor;
}

// Largest message for which one block finds its entries that way: ranking them costs their number squared, counting them in a histogram
// mostly the sweep over all d.  alone: at most one block per SM, where the barriers of the histogram weigh more; grad: the block (or its cluster)
// forms the gradients, too.  us, histogram / this way -- many vectors: 592 x 16,384 Top-128 32.7 / 32.9, Top-192 34.6 / 48.9, 592 x 9,000 Top-64
// 24.6 / 23.1, Top-128 26.4 / 30.9; 888 x 8,192 Top-80 24.2 / 20.4, Top-112 25.1 / 28.7, 888 x 2,100 Top-32 14.1 / 14.1, Top-64 14.8 / 16.8;
// 3,000 x 2,048 Top-48 26.7 / 23.7, Top-64 27.3 / 29.3, 3,000 x 300 Top-32 18.0 / 18.2.  Ten rounds of 20 workers: 9,000 Top-128 140.8 / 137.7, Top-192
// 149 / 194; 8,192 Top-96 131.8 / 121.3, Top-128 146.8 / 153.2; 4,000 Top-64 104.6 / 98.9, Top-96 108.3 / 111.4; 2,048 Top-64 99.7 / 90.5; 300 Top-32
// 76.6 / 77.2.  20 iterations on 10 x 100 rows: 8,000 columns Top-128 464 / 418, 5,001 Top-128 399 / 378, 1,500 Top-64 258 / 254, Top-128 279 / 314,
// 600 Top-64 247 / 235, Top-128 251 / 282.
EF21_BISECT_FN int few_limit(int threads, int d, bool alone, bool grad) {
    const int line = threads == 256 ? d / 48 + 16 : (threads == 512 ? (grad ? d / 60 + 36 : d / 112 + 18) : d / 133 + 32);
    const int more = !alone ? 0 : (threads == 256 ? 10 : (threads == 512 ? 30 : 32));
    return line + more < threads / 4 ? line + more : threads / 4;
}

}  // namespace ef21
