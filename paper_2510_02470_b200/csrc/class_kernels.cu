// Class-balanced variant (Algorithm 1, the class-balanced branch; section on agreement scoring and selection):
// per-class unit centroids u_c of the stored normalised projections, scores <zhat_i, u_c(i)>, and the top-k_c
// examples of every class. All reductions run in a fixed order (ascending example index), so results are
// reproducible bit for bit.
#include "sage_internal.h"

namespace sage {
namespace {

// The rows of a class are a run of `order` (rows grouped by class, ascending index). Block (s, c) sums the s-th of gridDim.x equal
// parts of class c in fp64: thread j of group g owns component j and takes rows g, g + G, ... (G = 256 / jw groups), the
// groups' sums are added in ascending order. parts: that sum (C x gridDim.x x ell), or, with one part per class, the result.
__global__ void __launch_bounds__(256) k_class_sums(const float* __restrict__ zhat, const unsigned* __restrict__ order,
                                                    const unsigned* __restrict__ starts, int ell, int jw, double* __restrict__ parts,
                                                    float* __restrict__ U, int* __restrict__ counts) {
    __shared__ double sh[256];
    __shared__ double red[8];
    const int c = blockIdx.y, j = threadIdx.x % jw, g = threadIdx.x / jw, G = 256 / jw;
    chain_wait();
    chain_release();
    const unsigned first = starts[c], n = starts[c + 1] - first;
    const unsigned len = (n + gridDim.x - 1) / gridDim.x;
    const unsigned r0 = blockIdx.x * len, r1 = min(n, r0 + len);
    double acc = 0.0;
    if (j < ell) {
        unsigned r = r0 + g;
        for (; r + 3 * G < r1; r += 4 * G) {                 // four rows' loads in flight, added in order
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = zhat[(int64_t)order[first + r + u * G] * ell + j];
#pragma unroll
            for (int u = 0; u < 4; ++u) acc += (double)v[u];
        }
        for (; r < r1; r += G) acc += (double)zhat[(int64_t)order[first + r] * ell + j];
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    double t = 0.0;
    if (g == 0)
        for (int q = 0; q < G; ++q) t += sh[q * jw + j];
    if (gridDim.x > 1) {
        if (g == 0 && j < ell) parts[((int64_t)c * gridDim.x + blockIdx.x) * ell + j] = t;
        return;
    }
    double sq = (g == 0 && j < ell) ? t * t : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sq;
    __syncthreads();
    double tot = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) tot += red[w];
    if (g == 0 && j < ell) U[(int64_t)c * ell + j] = tot > 0.0 ? (float)(t / sqrt(tot)) : 0.f;
    if (threadIdx.x == 0) counts[c] = (int)n;
}

// Block c: the parts of class c in ascending order, the unit vector (the mean's 1/|I_c| cancels), the class size.
__global__ void __launch_bounds__(256) k_class_units(const double* __restrict__ parts, int nparts, const unsigned* __restrict__ starts, int ell,
                                                     float* __restrict__ U, int* __restrict__ counts) {
    __shared__ double red[8];
    const int c = blockIdx.x, j = threadIdx.x;
    double t = 0.0;
    chain_wait();
    chain_release();
    if (j < ell) {
        int s = 0;
        for (; s + 8 <= nparts; s += 8) {                    // eight loads in flight, added in order
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = parts[((int64_t)c * nparts + s + u) * ell + j];
#pragma unroll
            for (int u = 0; u < 8; ++u) t += v[u];
        }
        for (; s < nparts; ++s) t += parts[((int64_t)c * nparts + s) * ell + j];
    }
    double sq = t * t;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if ((j & 31) == 0) red[j >> 5] = sq;
    __syncthreads();
    double tot = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) tot += red[w];
    if (j < ell) U[(int64_t)c * ell + j] = tot > 0.0 ? (float)(t / sqrt(tot)) : 0.f;
    if (j == 0) counts[c] = (int)(starts[c + 1] - starts[c]);
}

// One warp per example, four of a warp's in flight: score = <zhat_i, u_label(i)>; examples without a class in [0, C) score 0.
template <int T>
__global__ void __launch_bounds__(256) k_class_scores(const float* __restrict__ zhat, const int* __restrict__ labels, int64_t N,
                                                      int ell, int C, const float* __restrict__ U, float* __restrict__ scores) {
    constexpr int RB = T > 4 ? 2 : 4;
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * 8;
    chain_wait();
    chain_release();
    for (int64_t r0 = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); r0 < N; r0 += RB * stride) {
        float acc[RB];
        int lab[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            lab[r] = r0 + r * stride < N ? labels[r0 + r * stride] : -1;
            if (lab[r] >= C) lab[r] = -1;
        }
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            acc[r] = 0.f;
#pragma unroll
            for (int t = 0; t < T; ++t)
                if (lab[r] >= 0 && lane + 32 * t < ell)
                    acc[r] = fmaf(zhat[(r0 + r * stride) * ell + lane + 32 * t], U[(int64_t)lab[r] * ell + lane + 32 * t], acc[r]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int r = 0; r < RB; ++r) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
#pragma unroll
        for (int r = 0; r < RB; ++r)
            if (lane == 0 && r0 + r * stride < N) scores[r0 + r * stride] = fminf(1.f, fmaxf(-1.f, acc[r]));
    }
}

// Parts per class: enough blocks to fill the device when there are few classes, one when there are many.
int class_parts(int C) {
    const int p = 16384 / C;
    return p > 64 ? 64 : p < 1 ? 1 : p;
}
size_t up256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

size_t class_scratch_bytes(int64_t N, int ell, int C) {
    size_t sel = 0;
    select_scratch_bytes(N > 0 ? N : 1, &sel);
    return up256(sel) + up256((size_t)N * 4) + up256((size_t)(C + 1) * 4) + (size_t)C * class_parts(C) * ell * sizeof(double);
}

// Launches: the rows grouped by class, the sums of their projections, the scores. What it replaced walked all rows once per
// class in a block of its own, as did the picks from the sorted scores: scores, class scores and picks of 50,000 rows (10 classes,
// ell = 64, D = 5,130) 2.86 -> 0.58 ms.
cudaError_t launch_class_scores(const float* zhat, const int* labels, int64_t N, int ell, int C, float* U, int* counts, float* scores,
                                void* scratch, cudaStream_t st) {
    if (C <= 0) return cudaSuccess;
    size_t sel = 0;
    select_scratch_bytes(N > 0 ? N : 1, &sel);
    char* p = static_cast<char*>(scratch);
    unsigned* order = reinterpret_cast<unsigned*>(p + up256(sel));
    unsigned* starts = reinterpret_cast<unsigned*>(p + up256(sel) + up256((size_t)N * 4));
    double* parts = reinterpret_cast<double*>(p + up256(sel) + up256((size_t)N * 4) + up256((size_t)(C + 1) * 4));
    cudaError_t e = launch_class_order(labels, N, C, scratch, order, starts, st);
    if (e != cudaSuccess) return e;
    int jw = 32;
    while (jw < ell) jw <<= 1;
    const int np = class_parts(C);
    e = launch_chained(k_class_sums, dim3(np, C), dim3(256), 0, st, zhat, order, starts, ell, jw, parts, U, counts);
    if (e == cudaSuccess && np > 1) e = launch_chained(k_class_units, dim3(C), dim3(256), 0, st, parts, np, starts, ell, U, counts);
    if (e != cudaSuccess || N <= 0) return e;
    int64_t blocks = (N + 7) / 8;
    if (blocks > 148 * 8) blocks = 148 * 8;
    auto run = [&](auto kernel) { return launch_chained(kernel, dim3((unsigned)blocks), dim3(256), 0, st, zhat, labels, N, ell, C, U, scores); };
    return ell <= 32 ? run(k_class_scores<1>) : ell <= 64 ? run(k_class_scores<2>) : ell <= 128 ? run(k_class_scores<4>) : run(k_class_scores<8>);
}

}  // namespace sage
