// EF21+ (Algorithm 3): every worker keeps the better of the plain compressor b_i = C(grad_i) and the
// Markov compressor m_i = g_i + C(grad_i - g_i), judged by the distortions
//     B_i = ||b_i - grad_i||^2,   M_i = ||m_i - grad_i||^2      (fp64 sums of fp32 terms),
// g_i <- m_i if M_i <= B_i else b_i; the master recomputes g = (1/n) sum_i g_i.
//
// Both messages come from the Top-k kernels, which also leave the cut of each selection -- entry j is in the message if and only
// if (key << 32 | ~j) >= cut -- so that membership is one compare.  Then three kernels: the distortions, several blocks per
// worker; the choice and the sparse update of the Markov workers; the dense mean, which also rewrites the rows of workers that
// took the plain branch.  Bound by HBM / L2: g_i and grad_i are read once for the distortions, g_i once for the mean (one block per
// worker did all of it before: 1,170 us for 16 workers of 1,000,003 entries against about 35 us).
#pragma once
#include "common.cuh"
#include "topk_stream.cuh"

namespace ef21 {

constexpr int PLUS_BLOCK = 256;
constexpr int PLUS_MAX_PARTS = 64;          // blocks per worker in the distortion pass

// Deterministic block sum of doubles (fixed tree): result valid in thread 0.
__device__ __forceinline__ double block_sum_f64(double v, double* scratch /* [PLUS_BLOCK/32] */) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < PLUS_BLOCK / 32; ++w) s += scratch[w];
    __syncthreads();
    return s;
}

// 0: Markov, 1: plain, 2: to be decided by the ordered sums (the whole warp calls it).  The sums that the selecting kernels leave decide
// where they differ by more than one part in 10,000.  They are off by less than a tenth of that: a term is a rounded difference squared and
// added to at most 128 others per lane in 32 bits, each rounding 2^-24 of a sum of non-negative terms, 131 x 2^-24 = 8e-6 in all, the
// rest is 64 bits; squares below the normal range lose at most 2^-150 each, 1e-30 for every vector that fits the device; an
// overflow makes the sum infinite.  Closer distortions, and vectors that the exact fallback has selected from, go through the ordered 64-bit
// sums below, where M and B are bit-identical whenever the candidates coincide.  (g_i = 0, the state of the first round: they coincide
// term by term, and a tie goes to the Markov compressor.)
__device__ __forceinline__ int plus_decision(const PlusSums& s, int i, int n) {
    const int lane = threadIdx.x & 31;
    double M = 0.0, B = 0.0;
    bool nonzero = false;
    for (int q = lane; q < s.low_parts; q += 32) {
        const double2 w = s.low[(i64)i * s.low_pitch + q];
        M += w.x; B += w.y;
        nonzero |= s.nonzero[(i64)i * s.low_pitch + q] != 0;
    }
    for (int q = lane; q < s.groups; q += 32) { M += s.cand[(i64)i * s.groups + q]; B += s.cand[(i64)(n + i) * s.groups + q]; }
    M = warp_sum(M); B = warp_sum(B);
    if (s.ctl[i].slow || s.ctl[n + i].slow || !(M + B <= 1.7e308)) return 2;
    if (!__any_sync(0xffffffffu, nonzero)) return 0;
    if (!(fabs(M - B) > 1e-4 * (M + B) + 1e-30)) return 2;
    return M <= B ? 0 : 1;
}

// The ordered sums.  grid = (parts, n); part p of worker i covers the coordinates [p * len, (p + 1) * len).  part_out[i][p] = (M, B) of the part.  M and B
// are summed over the same coordinates in the same order, so that they are bit-identical whenever the two candidates coincide
// (e.g. g_i = 0).
// SUMS: the selecting kernels have left sums that decide as a rule.
template <bool SUMS>
__global__ void __launch_bounds__(PLUS_BLOCK)
plus_distortion_kernel(const float* __restrict__ a, i64 pitch_a, const float* __restrict__ gi, i64 ld, i64 d, i64 len,
                       const unsigned long long* __restrict__ cuts /* [2][n]: Markov, plain */, double2* __restrict__ part_out, const __grid_constant__ PlusSums sums) {
    pdl_trigger();
    pdl_wait(a, gi, cuts, part_out);
    __shared__ double scratch[PLUS_BLOCK / 32];
    const int i = blockIdx.y, n = gridDim.y;
    if (SUMS && plus_decision(sums, i, n) != 2) return;                      // as a rule
    const unsigned long long cut_m = cuts[i], cut_b = cuts[n + i];
    const unsigned km = (unsigned)(cut_m >> 32), jm = 0xffffffffu - (unsigned)cut_m, kb = (unsigned)(cut_b >> 32), jb = 0xffffffffu - (unsigned)cut_b;
    const float* __restrict__ grad = a + (i64)i * pitch_a;
    const float* __restrict__ g = gi + (i64)i * ld;
    const i64 j_end = min((i64)(blockIdx.x + 1) * len, d);
    double m_part = 0.0, b_part = 0.0;
    constexpr int U = 8;
    for (i64 j0 = (i64)blockIdx.x * len + threadIdx.x; j0 < j_end; j0 += U * PLUS_BLOCK) {
        float x[U], o[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const i64 j = j0 + u * PLUS_BLOCK;
            x[u] = j < j_end ? grad[j] : 0.f; o[u] = j < j_end ? g[j] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned j = (unsigned)(j0 + u * PLUS_BLOCK);
            const float v = __fsub_rn(x[u], o[u]);
            const unsigned kv = mag_key(v), kx = mag_key(x[u]);
            const bool in_m = kv > km || (kv == km && j <= jm), in_b = kx > kb || (kx == kb && j <= jb);
            const double e = (double)(in_m ? __fadd_rn(o[u], v) : o[u]) - (double)x[u];       // entries behind the end are 0 - 0
            m_part += e * e;
            b_part += in_b ? 0.0 : (double)x[u] * (double)x[u];
        }
    }
    const double M = block_sum_f64(m_part, scratch), B = block_sum_f64(b_part, scratch);
    if (threadIdx.x == 0) part_out[(i64)i * PLUS_MAX_PARTS + blockIdx.x] = make_double2(M, B);
}

// grid = (ceil(k / 256), n).  Every block adds up the parts of its worker in the same fixed order; a Markov worker's entries are
// added to g_i, a plain worker's message takes the place of the Markov one (the rows are rewritten by plus_mean_kernel).
template <bool SUMS>
__global__ void __launch_bounds__(PLUS_BLOCK)
plus_choose_kernel(const double2* __restrict__ parts_in, int parts, float* __restrict__ gi, i64 ld, int k,
                   int* __restrict__ idx_m, float* __restrict__ val_m, const int* __restrict__ idx_b, const float* __restrict__ val_b,
                   int* __restrict__ choice, const __grid_constant__ PlusSums sums) {
    pdl_trigger();
    pdl_wait(parts_in, gi, idx_m, val_m, idx_b, val_b, choice);
    const int i = blockIdx.y, lane = threadIdx.x & 31;
    int plain = SUMS ? plus_decision(sums, i, gridDim.y) : 2;
    if (plain == 2) {
        double M = 0.0, B = 0.0;
        for (int q = lane; q < parts; q += 32) { const double2 s = parts_in[(i64)i * PLUS_MAX_PARTS + q]; M += s.x; B += s.y; }
        M = warp_sum(M); B = warp_sum(B);
        plain = M <= B ? 0 : 1;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) choice[i] = plain;
    const int t = blockIdx.x * PLUS_BLOCK + threadIdx.x;
    if (t >= k) return;
    const i64 e = (i64)i * k + t;
    if (plain) {
        idx_m[e] = idx_b[e]; val_m[e] = val_b[e];
    } else {
        float* p = gi + (i64)i * ld + idx_m[e];
        *p = __fadd_rn(*p, val_m[e]);
    }
}

// g_j = (sum over workers, ascending, of g_ij) * (1/n), four coordinates per thread (ld is a multiple of four); g_ij of a worker that took
// the plain branch becomes C(grad_i)_j first.  XMODE as in the aggregation kernels.  Four blocks per SM (107 registers and two blocks:
// 16.9 us for 16 x 1,000,003, now 14.2).
template <int XMODE>
__global__ void __launch_bounds__(256, 4)
plus_mean_kernel(const float* __restrict__ a, i64 pitch_a, const unsigned long long* __restrict__ cut_b, const int* __restrict__ choice,
                 float* __restrict__ gi, i64 ld, int n, i64 d, float inv_n, float gamma, float* __restrict__ g, float* __restrict__ x) {
    pdl_trigger();
    pdl_wait(a, cut_b, choice, gi, g, x);
    for (i64 j = 4 * (blockIdx.x * (i64)blockDim.x + threadIdx.x); j < d; j += 4 * (i64)gridDim.x * blockDim.x) {
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        // eight rows on their way at a time (a load behind the branch of every row: 100 workers, d = 356, 49 us a round)
        for (int i0 = 0; i0 < n; i0 += 8) {
            float4 w[8];
            bool plain[8], any = false;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                plain[q] = i0 + q < n && choice[i0 + q] != 0;
                w[q] = i0 + q < n ? *reinterpret_cast<const float4*>(gi + (i64)(i0 + q) * ld + j) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) any = any || plain[q];
            if (any) {
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    if (!plain[q]) continue;
                    const int i = i0 + q;
                    const unsigned long long cut = cut_b[i];
                    float b[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float v = j + e < d ? a[(i64)i * pitch_a + j + e] : 0.f;
                        const unsigned long long c = ((unsigned long long)mag_key(v) << 32) | (0xffffffffu - (unsigned)(j + e));
                        b[e] = j + e < d && c >= cut ? v : 0.f;
                    }
                    w[q] = make_float4(b[0], b[1], b[2], b[3]);
                    *reinterpret_cast<float4*>(gi + (i64)i * ld + j) = w[q];
                }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (i0 + q < n) {
                    s[0] = __fadd_rn(s[0], w[q].x); s[1] = __fadd_rn(s[1], w[q].y); s[2] = __fadd_rn(s[2], w[q].z); s[3] = __fadd_rn(s[3], w[q].w);
                }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (j + e >= d) break;
            const float now = __fmul_rn(s[e], inv_n);
            if (XMODE != 0) x[j + e] = fmaf(-gamma, XMODE == 1 ? g[j + e] : now, x[j + e]);
            g[j + e] = now;
        }
    }
}

}  // namespace ef21
