// Copies and clears of state, several arrays in one launch.  A memcpy or memset node costs 2-4 us between two kernels and cannot
// be a programmatic dependent; the pitched copy of a large g_i (64 rows of 16 MB) ran at half the HBM rate as well (640 us
// against 330 us, measured).
#pragma once
#include "common.cuh"

namespace ef21 {

// rows x width 32-bit words from src (nullptr: zeros) to dst.
struct CopySeg {
    unsigned* dst; const unsigned* src;
    i64 dpitch, spitch, width, rows;
    i64 units;                              // blocks of this segment: rows * ceil(width / COPY_UNIT)
};
constexpr int COPY_UNIT = 8192, COPY_THREADS = 256, COPY_SEGS = 5;
struct CopyArgs { CopySeg seg[COPY_SEGS]; int count; };

__global__ void __launch_bounds__(COPY_THREADS)
copy_segments_kernel(const __grid_constant__ CopyArgs p) {
    pdl_trigger();
    pdl_wait();
    i64 u = blockIdx.x;
    int s = 0;
    while (s + 1 < p.count && u >= p.seg[s].units) { u -= p.seg[s].units; ++s; }
    const CopySeg& c = p.seg[s];
    const i64 per_row = (c.width + COPY_UNIT - 1) / COPY_UNIT;
    const i64 row = u / per_row, w0 = (u - row * per_row) * COPY_UNIT;
    const int len = (int)min((i64)COPY_UNIT, c.width - w0);
    unsigned* dst = c.dst + row * c.dpitch + w0;
    const unsigned* src = pdl_ptr(c.src ? c.src + row * c.spitch + w0 : nullptr);
    int done = 0;
    if (((reinterpret_cast<size_t>(dst) | reinterpret_cast<size_t>(src)) & 15u) == 0u) {
        const int quads = len >> 2;
        constexpr int U = COPY_UNIT / 4 / COPY_THREADS;
        uint4 v[U];
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int e = threadIdx.x + q * COPY_THREADS;
            v[q] = src && e < quads ? __ldcs(reinterpret_cast<const uint4*>(src) + e) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int q = 0; q < U; ++q) {
            const int e = threadIdx.x + q * COPY_THREADS;
            if (e < quads) reinterpret_cast<uint4*>(dst)[e] = v[q];
        }
        done = quads * 4;
    }
    // rows of odd length: word by word, sixteen loads in flight
    for (int e0 = done + threadIdx.x; e0 < len; e0 += 16 * COPY_THREADS) {
        unsigned v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) { const int e = e0 + q * COPY_THREADS; v[q] = src && e < len ? __ldcs(src + e) : 0u; }
#pragma unroll
        for (int q = 0; q < 16; ++q) { const int e = e0 + q * COPY_THREADS; if (e < len) dst[e] = v[q]; }
    }
}

}  // namespace ef21
