// Shape of the gradient kernel of rows of 513 to 8,192 columns (grad_wide_kernel in grad.cuh) and of its ring in shared memory, by the
// row's length.  Free of CUDA apart from the qualifier, so that a host compiler takes it too and every length can be looked at without
// a GPU.
#pragma once
#ifdef __CUDACC__
#define EF21_WIDE_FN __host__ __device__ constexpr
#else
#define EF21_WIDE_FN constexpr
#endif

namespace ef21 {

constexpr int GRAD_WIDE_SMEM = 192 * 1024, GRAD_WIDE_MAX_STAGES = 8;      // of the rings, at most
constexpr int GRAD_WIDE_SUMS = 8192;                                    // at most, of a second group

// Threads per group, float4 columns per thread, groups of threads per block, rows a group takes at a time.
struct WideShape { int threads, columns, groups, rows; };

// Rows of up to 2,048 columns: two groups of 256 threads that hold 1,024 columns a chunk; longer ones: 512 threads, 2,048 columns a chunk.
constexpr WideShape GRAD_WIDE_SHAPES[5] = {{256, 1, 2, 8}, {256, 2, 2, 4}, {512, 2, 1, 4}, {512, 3, 1, 4}, {512, 4, 1, 2}};
EF21_WIDE_FN int grad_wide_shape(int ld) { return ld <= 1024 ? 0 : (ld <= 2048 ? 1 : (ld + 2047) / 2048); }

// Stages of a group's ring.  160 KB for all rings, which leaves room beside the block for those of the kernels in between; 192 KB where four rows
// are more than half of that (5,121 to 6,144 columns): with one stage the next rows are asked for when the last ones have been taken, and
// every batch waits for HBM.  20 iterations on 20 x 200 rows, us with one stage, with two rows at a time (three stages) and with 192 KB: 5,124
// columns 522, 541, 469; 5,600 columns 555, 562, 495; 6,144 columns 634, 586, 540.
EF21_WIDE_FN int grad_wide_stages(int groups, int rows, int ld) {
    const int batch = groups * rows * ld * 4, usual = 160 * 1024, fit = (2 * batch > usual ? GRAD_WIDE_SMEM : usual) / batch;
    return fit < GRAD_WIDE_MAX_STAGES ? fit : GRAD_WIDE_MAX_STAGES;
}

// Dynamic shared memory of a block: the rings, and behind them the sums of the groups other than the first (no copy of rows lands there).
EF21_WIDE_FN int grad_wide_ring_bytes(const WideShape& s, int ld) { return s.groups * grad_wide_stages(s.groups, s.rows, ld) * s.rows * ld * 4; }
EF21_WIDE_FN int grad_wide_smem_bytes(const WideShape& s, int ld) { return grad_wide_ring_bytes(s, ld) + (s.groups - 1) * ld * 4; }

// A group that stops early must not leave copies on their way into shared memory that others get: wait(stage, parity) for the last batch of
// every stage, of `issued` batches that went to the stages in turn.  (A wait for one that has been taken returns at once.)
template <typename Wait>
EF21_WIDE_FN void grad_wide_settle(int issued, int stages, Wait wait) {
    for (int b = issued > stages ? issued - stages : 0; b < issued; ++b) wait(b % stages, (unsigned)(b / stages) & 1u);
}

}  // namespace ef21
