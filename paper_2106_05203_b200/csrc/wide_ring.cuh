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

}  // namespace ef21
