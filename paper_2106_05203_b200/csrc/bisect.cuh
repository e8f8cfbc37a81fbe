// Floor under the largest keys by bisection: what the selections of few entries start from (topk_cluster.cuh).  Free of CUDA apart from the
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

}  // namespace ef21
