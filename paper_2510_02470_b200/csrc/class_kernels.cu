// Class-balanced variant (Algorithm 1, the class-balanced branch; section on agreement scoring and selection):
// per-class unit centroids u_c of the stored normalised projections, scores <zhat_i, u_c(i)>, and the top-k_c
// examples of every class. All reductions run in a fixed order (ascending example index), so results are
// reproducible bit for bit.
#include "sage_internal.h"

namespace sage {
namespace {

// Sum in fp64 of the rows order[r0 .. r1): thread j of group g owns component j and takes rows g, g + G, ... (G = 256 / jw groups of a
// block), the groups' sums are added in ascending order. In the threads of group 0.
__device__ __forceinline__ double sum_rows(const float* __restrict__ zhat, const unsigned* order, unsigned r0, unsigned r1, int ell, int jw, double* sh) {
    const int j = threadIdx.x % jw, g = threadIdx.x / jw, G = 256 / jw;
    double acc = 0.0;
    if (j < ell) {
        unsigned r = r0 + g;
        for (; r + 3 * G < r1; r += 4 * G) {                 // four rows' loads in flight, added in order
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = zhat[(int64_t)order[r + u * G] * ell + j];
#pragma unroll
            for (int u = 0; u < 4; ++u) acc += (double)v[u];
        }
        for (; r < r1; r += G) acc += (double)zhat[(int64_t)order[r] * ell + j];
    }
    sh[threadIdx.x] = acc;
    __syncthreads();
    double t = 0.0;
    if (g == 0)
        for (int q = 0; q < G; ++q) t += sh[q * jw + j];
    return t;
}
// The unit vector of a class from its sum (components in the first jw threads; the mean's 1/|I_c| cancels), and the class size.
__device__ __forceinline__ void store_unit(double t, unsigned n, int c, int ell, int jw, float* __restrict__ U, int* __restrict__ counts, double* red) {
    const int j = threadIdx.x;
    double sq = j < jw && j < ell ? t * t : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if ((j & 31) == 0) red[j >> 5] = sq;
    __syncthreads();
    double tot = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) tot += red[w];
    if (j < jw && j < ell) U[(int64_t)c * ell + j] = tot > 0.0 ? (float)(t / sqrt(tot)) : 0.f;
    if (j == 0) counts[c] = (int)n;
}

// Few rows: block c finds the rows of its class by itself, in ascending order, and forms the centroid; no grouping, no parts. A block
// reads the rows of its class 4 x 256 / jw at a time, and every block looks at all labels: long rows in one or two classes, and very many
// classes, are grouped already when there are fewer rows (few_rows). 100 to 2,048 rows of 64 values in 10, 100, 1,000 classes: 9 to
// 12 us by this and the scores, 15, 21, 44 us by grouping; 512 rows of 256 values in one class 35 against 16, 2,048 rows in 20,000
// classes 100 against 75 us.
constexpr int kFewRows = 2048;
__global__ void __launch_bounds__(256) k_class_few(const float* __restrict__ zhat, const int* __restrict__ labels, int N, int ell, int jw,
                                                   float* __restrict__ U, int* __restrict__ counts) {
    __shared__ double sh[256];
    __shared__ double red[8];
    __shared__ unsigned order[kFewRows], found[8];
    const int c = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    chain_wait();
    chain_release();
    unsigned n = 0;
    for (int b0 = 0; b0 < N; b0 += 256) {
        const int i = b0 + threadIdx.x;
        const unsigned mine = __ballot_sync(0xffffffffu, i < N && labels[i] == c);
        if (lane == 0) found[warp] = (unsigned)__popc(mine);
        __syncthreads();
        unsigned at = n;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            if (w < warp) at += found[w];
            n += found[w];
        }
        if (mine >> lane & 1u) order[at + __popc(mine & ((1u << lane) - 1u))] = (unsigned)i;
        __syncthreads();
    }
    store_unit(sum_rows(zhat, order, 0, n, ell, jw, sh), n, c, ell, jw, U, counts, red);
}

// The rows of a class are a run of `order` (rows grouped by class, ascending index). Block (s, c) sums the s-th of gridDim.x equal
// parts of class c. parts: that sum (C x gridDim.x x ell), or, with one part per class, the result.
__global__ void __launch_bounds__(256) k_class_sums(const float* __restrict__ zhat, const unsigned* __restrict__ order,
                                                    const unsigned* __restrict__ starts, int ell, int jw, double* __restrict__ parts,
                                                    float* __restrict__ U, int* __restrict__ counts) {
    __shared__ double sh[256];
    __shared__ double red[8];
    const int c = blockIdx.y;
    chain_wait();
    chain_release();
    const unsigned first = starts[c], n = starts[c + 1] - first;
    const unsigned len = (n + gridDim.x - 1) / gridDim.x;
    const unsigned r0 = min(n, blockIdx.x * len), r1 = min(n, r0 + len);
    const double t = sum_rows(zhat, order, first + r0, first + r1, ell, jw, sh);
    if (gridDim.x > 1) {
        if (threadIdx.x < jw && threadIdx.x < ell) parts[((int64_t)c * gridDim.x + blockIdx.x) * ell + threadIdx.x] = t;
        return;
    }
    store_unit(t, n, c, ell, jw, U, counts, red);
}

// Block c: the parts of class c in ascending order, the unit vector, the class size.
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
    store_unit(t, starts[c + 1] - starts[c], c, ell, 256, U, counts, red);
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
int width_of(int ell) {                                  // ell rounded up to a power of two, at least 32
    int jw = 32;
    while (jw < ell) jw <<= 1;
    return jw;
}
bool few_rows(int64_t N, int ell, int C) { return N <= kFewRows && N * width_of(ell) <= (int64_t)32768 * C && N * C <= 20000000; }
size_t up256(size_t x) { return (x + 255) & ~size_t(255); }

cudaError_t scores_of(const float* zhat, const int* labels, int64_t N, int ell, int C, const float* U, float* scores, cudaStream_t st) {
    int64_t blocks = (N + 7) / 8;
    if (blocks > 148 * 8) blocks = 148 * 8;
    auto run = [&](auto kernel) { return launch_chained(kernel, dim3((unsigned)blocks), dim3(256), 0, st, zhat, labels, N, ell, C, U, scores); };
    return ell <= 32 ? run(k_class_scores<1>) : ell <= 64 ? run(k_class_scores<2>) : ell <= 128 ? run(k_class_scores<4>) : run(k_class_scores<8>);
}

}  // namespace

size_t class_scratch_bytes(int64_t N, int ell, int C) {
    if (few_rows(N, ell, C)) return 0;
    size_t sel = 0;
    select_scratch_bytes(N, &sel);
    return up256(sel) + up256((size_t)N * 4) + up256((size_t)(C + 1) * 4) + (size_t)C * class_parts(C) * ell * sizeof(double);
}

int class_score_launches(int64_t N, int ell, int C) {
    return few_rows(N, ell, C) ? (N > 0 ? 2 : 1) : class_order_launches(N, C) + (class_parts(C) > 1 ? 3 : 2);
}

// Launches of more than a few rows: the rows grouped by class, the sums of their projections, the scores. What it replaced walked all rows once per
// class in a block of its own, as did the picks from the sorted scores: scores, class scores and picks of 50,000 rows (10 classes,
// ell = 64, D = 5,130) 2.86 -> 0.58 ms.
cudaError_t launch_class_scores(const float* zhat, const int* labels, int64_t N, int ell, int C, float* U, int* counts, float* scores,
                                void* scratch, cudaStream_t st) {
    if (C <= 0) return cudaSuccess;
    const int jw = width_of(ell);
    cudaError_t e = cudaSuccess;
    if (few_rows(N, ell, C)) {
        e = launch_chained(k_class_few, dim3(C), dim3(256), 0, st, zhat, labels, (int)N, ell, jw, U, counts);
        return e != cudaSuccess || N <= 0 ? e : scores_of(zhat, labels, N, ell, C, U, scores, st);
    }
    size_t sel = 0;
    select_scratch_bytes(N, &sel);
    char* p = static_cast<char*>(scratch);
    unsigned* order = reinterpret_cast<unsigned*>(p + up256(sel));
    unsigned* starts = reinterpret_cast<unsigned*>(p + up256(sel) + up256((size_t)N * 4));
    double* parts = reinterpret_cast<double*>(p + up256(sel) + up256((size_t)N * 4) + up256((size_t)(C + 1) * 4));
    e = launch_class_order(labels, N, C, scratch, order, starts, st);
    if (e != cudaSuccess) return e;
    const int np = class_parts(C);
    e = launch_chained(k_class_sums, dim3(np, C), dim3(256), 0, st, zhat, order, starts, ell, jw, parts, U, counts);
    if (e == cudaSuccess && np > 1) e = launch_chained(k_class_units, dim3(C), dim3(256), 0, st, parts, np, starts, ell, U, counts);
    return e != cudaSuccess ? e : scores_of(zhat, labels, N, ell, C, U, scores, st);
}

}  // namespace sage
