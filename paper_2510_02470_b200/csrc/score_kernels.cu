// Phase II after the projection (Method, paragraph on two-pass scoring; Algorithm 1, Phase II):
// row normalisation zhat_i = z_i/||z_i|| (0 when z_i = 0), the consensus sum over all rows, the unit
// consensus u and the agreement scores alpha_i = <zhat_i, u>. All reductions run in a fixed order, so
// a given sequence of calls gives bit-identical results every time.
#include "sage_internal.h"

namespace sage {
namespace {

constexpr int kRowsPerBlock = 64;   // rows whose zhat are summed into one partial

// One warp per row, 8 warps per block, each warp walks rows w, w+8, ... of the block's 64 rows, 8 / T of them at a time (T: 32-wide
// pieces of a row): the kernel is bound by the latency of its loads and reductions, so several rows' are in flight (50,000 rows
// of 64 values in two planes, 38 MB: 52 us with one row at a time).
// planes > 1: the projections arrive as that many partial planes (K slices of the projection, `plane_stride` floats apart),
// which are summed here in ascending plane order with fp64 accumulation before the row is normalised.
template <int T>
__global__ void __launch_bounds__(256) k_normalise(const float* __restrict__ Z, int planes, int64_t plane_stride, int64_t ldz, int64_t n,
                                                   int ell, float* __restrict__ zhat, float* __restrict__ znorm,
                                                   float* __restrict__ partials, unsigned* __restrict__ flags) {
    constexpr int RB = 8 / T;
    __shared__ float part[8][32 * T];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t row0 = (int64_t)blockIdx.x * kRowsPerBlock + warp;
    float sum[T];
#pragma unroll
    for (int t = 0; t < T; ++t) sum[t] = 0.f;
    bool bad = false;
    chain_wait();
    chain_release();
#pragma unroll 1
    for (int q0 = 0; q0 < kRowsPerBlock / 8; q0 += RB) {
        float z[RB][T];
        if (planes == 1) {
#pragma unroll
            for (int r = 0; r < RB; ++r)
#pragma unroll
                for (int t = 0; t < T; ++t) {
                    const int64_t row = row0 + 8 * (q0 + r);
                    z[r][t] = row < n && lane + 32 * t < ell ? Z[row * ldz + lane + 32 * t] : 0.f;
                }
        } else {
            double acc[RB][T];
#pragma unroll
            for (int r = 0; r < RB; ++r)
#pragma unroll
                for (int t = 0; t < T; ++t) acc[r][t] = 0.0;
#pragma unroll 2
            for (int pz = 0; pz < planes; ++pz)
#pragma unroll
                for (int r = 0; r < RB; ++r)
#pragma unroll
                    for (int t = 0; t < T; ++t) {
                        const int64_t row = row0 + 8 * (q0 + r);
                        if (row < n && lane + 32 * t < ell) acc[r][t] += (double)Z[pz * plane_stride + row * ldz + lane + 32 * t];
                    }
#pragma unroll
            for (int r = 0; r < RB; ++r)
#pragma unroll
                for (int t = 0; t < T; ++t) z[r][t] = (float)acc[r][t];
        }
        float amax[RB], s[RB];
        bool finite[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            amax[r] = 0.f;
            finite[r] = true;
#pragma unroll
            for (int t = 0; t < T; ++t) {
                finite[r] = finite[r] && (fabsf(z[r][t]) <= 3.0e38f);   // false for NaN and Inf
                amax[r] = fmaxf(amax[r], fabsf(z[r][t]));
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int r = 0; r < RB; ++r) amax[r] = fmaxf(amax[r], __shfl_xor_sync(0xffffffffu, amax[r], o));
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            finite[r] = __all_sync(0xffffffffu, finite[r]);
            const float inv = finite[r] && amax[r] > 0.f ? 1.f / amax[r] : 0.f;
            s[r] = 0.f;
#pragma unroll
            for (int t = 0; t < T; ++t) {
                z[r][t] = inv > 0.f ? z[r][t] * inv : 0.f;
                s[r] = fmaf(z[r][t], z[r][t], s[r]);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int r = 0; r < RB; ++r) s[r] += __shfl_xor_sync(0xffffffffu, s[r], o);
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            const int64_t row = row0 + 8 * (q0 + r);
            const float rs = sqrtf(s[r]), scale = s[r] > 0.f ? 1.f / rs : 0.f;       // 0 for zero and non-finite rows
            if (!finite[r] && row < n) bad = true;
#pragma unroll
            for (int t = 0; t < T; ++t) {
                const float v = scale > 0.f ? z[r][t] * scale : 0.f;
                if (row < n && lane + 32 * t < ell) zhat[row * ell + lane + 32 * t] = v;
                sum[t] += v;
            }
            if (row < n && lane == 0) znorm[row] = s[r] > 0.f ? amax[r] * rs : 0.f;
        }
    }
#pragma unroll
    for (int t = 0; t < T; ++t) part[warp][lane + 32 * t] = sum[t];
    __syncthreads();
    if (threadIdx.x < ell) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) s += part[w][threadIdx.x];
        partials[(int64_t)blockIdx.x * ell + threadIdx.x] = s;
    }
    if (bad && lane == 0) atomicOr(flags, kFlagNonFinite);
}

// zsum[j] += sum over blocks b of partials[b][j], in a fixed order: the 1024 threads form 1024 / jw groups (jw = ell rounded up to
// a power of two, at least 32); group g adds the partials of blocks g, g + G, g + 2G, ... in ascending order in fp64, and the
// groups' sums are then added in ascending g.
__global__ void __launch_bounds__(1024) k_accumulate(const float* __restrict__ partials, int nblocks, int ell, int jw,
                                                     double* __restrict__ zsum) {
    __shared__ double sh[1024];
    const int G = 1024 / jw;
    const int j = threadIdx.x % jw, g = threadIdx.x / jw;
    double s = 0.0;
    chain_wait();
    chain_release();
    if (j < ell) {
        int b = g;
        for (; b + 7 * G < nblocks; b += 8 * G) {           // eight loads in flight, added in order
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = partials[(int64_t)(b + u * G) * ell + j];
#pragma unroll
            for (int u = 0; u < 8; ++u) s += (double)v[u];
        }
        for (; b < nblocks; b += G) s += (double)partials[(int64_t)b * ell + j];
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    if (g == 0 && j < ell) {
        double t = zsum[j];
        for (int q = 0; q < G; ++q) t += sh[q * jw + j];
        zsum[j] = t;
    }
}

// u = zsum/||zsum|| (the 1/N of the mean cancels); alpha_i = <zhat_i, u>. One warp per row, four rows of a warp in flight; a warp
// takes more rows when there are many (every block forms u for itself).
template <int T>
__global__ void __launch_bounds__(256) k_consensus_score(const double* __restrict__ zsum, const float* __restrict__ zhat,
                                                         int64_t N, int ell, float* __restrict__ u_out,
                                                         float* __restrict__ scores) {
    __shared__ float u[256];
    __shared__ double red[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    chain_wait();
    chain_release();
    double v = (tid < ell) ? zsum[tid] : 0.0;
    double sq = v * v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (lane == 0) red[warp] = sq;
    __syncthreads();
    double tot = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) tot += red[w];
    const double nrm = sqrt(tot);
    u[tid] = (nrm > 0.0 && tid < ell) ? (float)(v / nrm) : 0.f;
    if (blockIdx.x == 0 && tid < ell) u_out[tid] = u[tid];
    __syncthreads();
    float uu[T];
#pragma unroll
    for (int t = 0; t < T; ++t) uu[t] = u[lane + 32 * t];
    constexpr int RB = T > 4 ? 2 : 4;
    const int64_t stride = (int64_t)gridDim.x * 8;
    for (int64_t r0 = (int64_t)blockIdx.x * 8 + warp; r0 < N; r0 += RB * stride) {
        float acc[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            const int64_t row = r0 + r * stride;
            acc[r] = 0.f;
#pragma unroll
            for (int t = 0; t < T; ++t)
                if (row < N && lane + 32 * t < ell) acc[r] = fmaf(zhat[row * ell + lane + 32 * t], uu[t], acc[r]);
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


// Structured rows: the projection z_i = sum_c q_ic (S_c h_i + b_c), b_c = column c of the bias block of the sketch, from the
// per-class planes T_c = H S_c^T. A thread owns four consecutive columns of one row of Z and walks the classes in ascending
// order (fp32), four classes' loads in flight at a time. biasT is the bias block transposed (C x ell, by k_bias_transpose), so
// that its reads are contiguous and shared by all rows. Needs ell a multiple of 4 and 16-byte aligned planes.
template <typename T>
__global__ void __launch_bounds__(256) k_outer_combine(const T* __restrict__ q, int64_t ldq, int C, const float* __restrict__ planes, int pp,
                                                       int64_t plane_stride, const float* __restrict__ biasT, int64_t total4, int ell,
                                                       float* __restrict__ Z) {
    const int64_t e4 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e4 >= total4) return;
    const int ell4 = ell >> 2;
    const int64_t i = e4 / ell4;
    const int j = (int)(e4 - i * ell4) * 4;
    const T* qr = q + i * ldq;
    const float* t = planes + i * ell + j;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int cb = 0; cb < C; cb += 4) {
        float4 v[4];
        float qc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = cb + u;
            qc[u] = c < C ? (float)qr[c] : 0.f;
            v[u] = c < C ? __ldg(reinterpret_cast<const float4*>(biasT + (int64_t)c * ell + j)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int p = 0; p < pp; ++p) {
            float4 w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                w[u] = cb + u < C ? __ldcs(reinterpret_cast<const float4*>(t + ((int64_t)(cb + u) * pp + p) * plane_stride))
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 4; ++u) { v[u].x += w[u].x; v[u].y += w[u].y; v[u].z += w[u].z; v[u].w += w[u].w; }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            acc.x = fmaf(qc[u], v[u].x, acc.x);
            acc.y = fmaf(qc[u], v[u].y, acc.y);
            acc.z = fmaf(qc[u], v[u].z, acc.z);
            acc.w = fmaf(qc[u], v[u].w, acc.w);
        }
    }
    *reinterpret_cast<float4*>(Z + i * ell + j) = acc;
}

// biasT[c][j] = Sb[j][c] (Sb: ell rows of pitch lds)
__global__ void __launch_bounds__(256) k_bias_transpose(const float* __restrict__ Sb, int64_t lds, int C, int ell, float* __restrict__ biasT) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= C * ell) return;
    const int j = x / C, c = x - j * C;
    biasT[(int64_t)c * ell + j] = Sb[(int64_t)j * lds + c];
}

// any ell: one thread per element
template <typename T>
__global__ void __launch_bounds__(256) k_outer_combine_scalar(const T* __restrict__ q, int64_t ldq, int C, const float* __restrict__ planes,
                                                              int pp, int64_t plane_stride, const float* __restrict__ biasT,
                                                              int64_t total, int ell, float* __restrict__ Z) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= total) return;
    const int64_t i = e / ell;
    const int j = (int)(e - i * ell);
    const T* qr = q + i * ldq;
    const float* t = planes + e;
    float acc = 0.f;
    for (int c = 0; c < C; ++c) {
        float v = __ldg(biasT + (int64_t)c * ell + j);
        for (int p = 0; p < pp; ++p) v += t[((int64_t)c * pp + p) * plane_stride];
        acc = fmaf((float)qr[c], v, acc);
    }
    Z[e] = acc;
}

}  // namespace

cudaError_t launch_normalise(const float* Z, int planes, int64_t plane_stride, int64_t ldz, int64_t n, int ell, float* zhat,
                             float* znorm, float* partials, double* zsum, unsigned* flags, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const int nblocks = (int)((n + kRowsPerBlock - 1) / kRowsPerBlock);
    auto run = [&](auto kernel) { return launch_chained(kernel, dim3(nblocks), dim3(256), 0, st, Z, planes, plane_stride, ldz, n, ell, zhat, znorm, partials, flags); };
    const cudaError_t e = ell <= 32 ? run(k_normalise<1>) : ell <= 64 ? run(k_normalise<2>) : ell <= 128 ? run(k_normalise<4>) : run(k_normalise<8>);
    if (e != cudaSuccess || !zsum) return e;
    int jw = 32;
    while (jw < ell) jw <<= 1;
    return launch_chained(k_accumulate, dim3(1), dim3(1024), 0, st, partials, nblocks, ell, jw, zsum);
}

cudaError_t launch_outer_combine(const void* q, int64_t ldq, sage_dtype_t dt, int C, const float* planes, int pp, int64_t plane_stride,
                                 const float* Sb, int64_t lds, float* biasT, int64_t n, int ell, float* Z, cudaStream_t st) {
    const int64_t total = n * ell;
    if (total <= 0 || C <= 0) return cudaSuccess;
    k_bias_transpose<<<(unsigned)(((int64_t)C * ell + 255) / 256), 256, 0, st>>>(Sb, lds, C, ell, biasT);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const bool vec = ell % 4 == 0 && plane_stride % 4 == 0 && (reinterpret_cast<uintptr_t>(planes) & 15u) == 0 &&
                     (reinterpret_cast<uintptr_t>(Z) & 15u) == 0 && (reinterpret_cast<uintptr_t>(biasT) & 15u) == 0;
    if (vec) {
        const int64_t total4 = total / 4;
        const unsigned blocks = (unsigned)((total4 + 255) / 256);
        if (dt == SAGE_F32)
            k_outer_combine<float><<<blocks, 256, 0, st>>>(static_cast<const float*>(q), ldq, C, planes, pp, plane_stride, biasT, total4, ell, Z);
        else
            k_outer_combine<__nv_bfloat16><<<blocks, 256, 0, st>>>(static_cast<const __nv_bfloat16*>(q), ldq, C, planes, pp, plane_stride,
                                                                   biasT, total4, ell, Z);
        return cudaGetLastError();
    }
    const unsigned blocks = (unsigned)((total + 255) / 256);
    if (dt == SAGE_F32)
        k_outer_combine_scalar<float><<<blocks, 256, 0, st>>>(static_cast<const float*>(q), ldq, C, planes, pp, plane_stride, biasT, total, ell, Z);
    else
        k_outer_combine_scalar<__nv_bfloat16><<<blocks, 256, 0, st>>>(static_cast<const __nv_bfloat16*>(q), ldq, C, planes, pp, plane_stride,
                                                                      biasT, total, ell, Z);
    return cudaGetLastError();
}

cudaError_t launch_consensus_score(const double* zsum, const float* zhat, int64_t N, int ell, float* u, float* scores,
                                   cudaStream_t st) {
    int64_t blocks = N > 0 ? (N + 7) / 8 : 1;
    if (blocks > 148 * 8) blocks = 148 * 8;                 // one wave: 8 blocks of 256 threads per SM
    auto run = [&](auto kernel) { return launch_chained(kernel, dim3((unsigned)blocks), dim3(256), 0, st, zsum, zhat, N, ell, u, scores); };
    return ell <= 32 ? run(k_consensus_score<1>) : ell <= 64 ? run(k_consensus_score<2>) : ell <= 128 ? run(k_consensus_score<4>) : run(k_consensus_score<8>);
}

}  // namespace sage
