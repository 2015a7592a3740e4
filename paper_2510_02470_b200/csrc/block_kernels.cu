// Shrink cycles in blocks. A shrink replaces the buffer B by W B, W = diag(sigma'/sigma) U^T from the eigen-problem of B B^T, and the
// next shrink needs the inner products of W B and the new rows: combinations, by the same W, of inner products that are known. So the
// rows of several cycles are read together: their inner products are formed once (tc_gram_block.cu), the chain of solves runs on those
// small matrices alone (k_block_step between two solves), and the kept rows are formed once at the end, by the product of the W
// (k_block_factors, tc_rebuild_block.cu). The same sketch as shrinking cycle by cycle, in another order of summation: per cycle the rows
// are not read, and the two kernels that did so, with their launches, leave the chain.
// W is applied as it was computed: also the products of the kept rows with each other are W K W^T, not the diagonal matrix that exact
// arithmetic would make of it, so that what rounding leaves of one large row in the others is seen, as it is in the rows themselves.
// Everything here gives the same bits however the rows of a block were spread over calls: a column's products are formed in the same
// order whether it is there from the block's beginning or catches up later.
#include "sage_internal.h"

namespace sage {
namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float finite_or_zero(float v) { return fabsf(v) <= 3.402823466e38f ? v : 0.f; }

// ---- rows into planes -----------------------------------------------------------------------------------------------
// x = hi + mid + lo by cutting 8 significant bits at a time (cut, not rounded: no plane of a finite value overflows); 8 values a thread.
__device__ __forceinline__ void store_planes(const float (&x)[8], __nv_bfloat16* dst, int64_t pitch, int np) {
    float r[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) r[i] = x[i];
    for (int p = 0; p < np; ++p, dst += pitch) {
        unsigned w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const unsigned a = __float_as_uint(r[2 * i]) & 0xffff0000u, b = __float_as_uint(r[2 * i + 1]) & 0xffff0000u;
            r[2 * i] -= __uint_as_float(a);
            r[2 * i + 1] -= __uint_as_float(b);
            w[i] = (a >> 16) | b;
        }
        *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

template <typename T>
__global__ void __launch_bounds__(kThreads) k_block_append(const T* __restrict__ rows, int64_t ld, int64_t D, __nv_bfloat16* __restrict__ R, int64_t pitch, int np,
                                                           int64_t row0, int vec) {
    chain_wait();
    chain_release();
    const T* src = rows + (int64_t)blockIdx.y * ld;
    __nv_bfloat16* dst = R + (row0 + blockIdx.y) * np * pitch;
    for (int64_t d = ((int64_t)blockIdx.x * kThreads + threadIdx.x) * 8; d < pitch; d += (int64_t)gridDim.x * kThreads * 8) {
        float x[8];
        if (vec && d + 8 <= D) {                   // rows that start on 16-byte boundaries
            if constexpr (sizeof(T) == 4) {
                const float4 a = *reinterpret_cast<const float4*>(src + d), b = *reinterpret_cast<const float4*>(src + d + 4);
                x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
                x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
            } else {
                const uint4 a = *reinterpret_cast<const uint4*>(src + d);
                const unsigned w[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    x[2 * i] = __uint_as_float(w[i] << 16);
                    x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = d + i < D ? to_f32(src[d + i]) : 0.f;
        }
        store_planes(x, dst + d, pitch, np);
    }
}

template <typename T>
__global__ void __launch_bounds__(kThreads) k_block_append_outer(const T* __restrict__ q, int64_t ldq, const T* __restrict__ feat, int64_t ldf, int C, int F,
                                                                 __nv_bfloat16* __restrict__ R, int64_t pitch, int np, int64_t row0) {
    chain_wait();
    chain_release();
    const T* qr = q + (int64_t)blockIdx.y * ldq;
    const T* hr = feat + (int64_t)blockIdx.y * ldf;
    __nv_bfloat16* dst = R + (row0 + blockIdx.y) * np * pitch;
    const int64_t CF = (int64_t)C * F, D = CF + C;
    for (int64_t d = ((int64_t)blockIdx.x * kThreads + threadIdx.x) * 8; d < pitch; d += (int64_t)gridDim.x * kThreads * 8) {
        float x[8];
        int c = (int)(d / F), f = (int)(d - (int64_t)c * F);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int64_t e = d + i;
            x[i] = e < CF ? to_f32(qr[c]) * to_f32(hr[f]) : e < D ? to_f32(qr[e - CF]) : 0.f;
            if (++f == F) { f = 0; ++c; }
        }
        store_planes(x, dst + d, pitch, np);
    }
}

__global__ void __launch_bounds__(kThreads) k_block_unpack(const __nv_bfloat16* __restrict__ R, int64_t pitch, int np, int64_t D, float* __restrict__ out, int64_t ldo) {
    chain_wait();
    const __nv_bfloat16* src = R + (int64_t)blockIdx.y * np * pitch;
    for (int64_t d = (int64_t)blockIdx.x * kThreads + threadIdx.x; d < ldo; d += (int64_t)gridDim.x * kThreads) {
        float x = 0.f;
        if (d < D)
            for (int p = np - 1; p >= 0; --p) x += __bfloat162float(src[p * pitch + d]);   // small ones first: exact at every step
        out[blockIdx.y * ldo + d] = x;
    }
}

// ---- inner products of rows from those of planes ---------------------------------------------------------------------
// 4 rows x 32 columns of P per block, and their mirror image; NJ: the most planes that a new row has. The K slices are dealt to the 8
// warps, whose sums are added in order. (One thread an element, slices in turn: 41 us for 3 planes a row and 7 slices, all latency.)
// Products of a row whose norm is not finite take no part in anything but its own diagonal element, which the solve looks at: they are
// zero here, as a coefficient of zero does not make them harmless.
template <int NJ>
__global__ void __launch_bounds__(256) k_block_gram_reduce(const float* __restrict__ parts, BlockMap map, int first_new, int slices, float* __restrict__ P, int ldP) {
    __shared__ double part[8][4][32];
    const int nl = block_rows(map), i0 = blockIdx.x * 4, j0 = first_new + blockIdx.y * 32;
    if (i0 > j0 + 31) return;
    const int first = block_phys(map, first_new) >> 8, nb = (map.P + 255) >> 8;
    const int base = first * (first + 1) / 2;
    const int64_t stride = (int64_t)(nb * (nb + 1) / 2 - base) * 65536;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, j = j0 + lane;
    chain_wait();
    chain_release();
    double sum[4] = {0.0, 0.0, 0.0, 0.0};
    if (j < nl) {
        const int pj = block_phys(map, j), nj = block_planes(map, j);
        for (int z = w; z < slices; z += 8) {
            const float* slice = parts + z * stride;
#pragma unroll
            for (int a0 = 0; a0 < 3; ++a0) {
                float v[4][NJ];
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    const int i = min(i0 + s, j), a = block_phys(map, i) + a0;
                    const bool on = a0 < block_planes(map, i);
#pragma unroll
                    for (int t = 0; t < NJ; ++t) {
                        const int b = pj + t, r = min(a, b), c = max(a, b), cb = c >> 8;                       // (a > b only among the planes of one row)
                        v[s][t] = on && t < nj ? __ldcg(slice + (int64_t)(cb * (cb + 1) / 2 - base + (r >> 8)) * 65536 + (r & 255) * 256 + (c & 255)) : 0.f;
                    }
                }
#pragma unroll
                for (int s = 0; s < 4; ++s)
#pragma unroll
                    for (int t = 0; t < NJ; ++t) sum[s] += (double)v[s][t];
                if (a0 == 0 && map.np == 1 && i0 >= map.s_rows) break;                                          // one plane each
            }
        }
    }
#pragma unroll
    for (int s = 0; s < 4; ++s) part[w][s][lane] = sum[s];
    __syncthreads();
    if (w < 4 && j < nl && i0 + w <= j) {
        const int i = i0 + w;
        double t = part[0][w][lane];
#pragma unroll
        for (int u = 1; u < 8; ++u) t += part[u][w][lane];
        float v = (float)t;
        if (i != j) v = finite_or_zero(v);
        P[(int64_t)i * ldP + j] = v;
        P[(int64_t)j * ldP + i] = v;
    }
}

// ---- products with W ---------------------------------------------------------------------------------------------------
// out[r][c] = sum_{i < n} A[i][r] x[i][c] for r < rows, c < COLS, in fp32. A thread has 4 values of r and a quarter of the columns of one of KS
// parts of the sum over i, which are added in order: A's elements come out of L2 (or shared memory) as they are needed, AHEAD loads in
// flight a thread, x out of shared memory. A's rows hold at least rows rounded up to 4 values. clean: sums that are not finite count as
// zero. Ends with a barrier behind the last read of x and the last write of out. (16 columns, half the reads of A in all: steps of windows of
// 256 and 512 rows 30 and 25 % longer, as what each block reads is what it waits for.)
template <int JG>                            // groups of 4 r
struct Apply {
    static constexpr int NT = JG == 16 ? 512 : 1024, KS = NT / (4 * JG), AHEAD = JG == 16 ? 16 : 8, COLS = 8, OWN = COLS / 4;
    typedef float Row[COLS];
    float red[KS][COLS][4 * JG];

    __device__ __forceinline__ void run(const float* A, int64_t lda, int n, int rows, const Row* x, Row* out, bool clean) {
        const int jg = threadIdx.x % JG, cp = threadIdx.x / JG % 4, ks = threadIdx.x / (4 * JG);
        for (int r0 = 0; r0 < rows; r0 += 4 * JG) {
            const int r = r0 + 4 * jg;
            float4 acc[OWN];
#pragma unroll
            for (int u = 0; u < OWN; ++u) acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r < rows) {
                const int i0 = n * ks / KS, i1 = n * (ks + 1) / KS;
                const float* a = A + (int64_t)i0 * lda + r;
                int i = i0;
                for (; i + AHEAD <= i1; i += AHEAD, a += AHEAD * lda) {
                    float4 v[AHEAD];
#pragma unroll
                    for (int u = 0; u < AHEAD; ++u) v[u] = *reinterpret_cast<const float4*>(a + u * lda);
#pragma unroll
                    for (int u = 0; u < AHEAD; ++u) add(acc, v[u], x[i + u] + OWN * cp);
                }
#pragma unroll 4
                for (; i < i1; ++i, a += lda) add(acc, *reinterpret_cast<const float4*>(a), x[i] + OWN * cp);
            }
#pragma unroll
            for (int u = 0; u < OWN; ++u) *reinterpret_cast<float4*>(&red[ks][OWN * cp + u][4 * jg]) = acc[u];
            __syncthreads();
            for (int t = threadIdx.x; t < 4 * JG * COLS; t += NT) {
                const int c = t / (4 * JG), rr = t % (4 * JG);
                float s = red[0][c][rr];
#pragma unroll
                for (int z = 1; z < KS; ++z) s += red[z][c][rr];
                if (r0 + rr < rows) out[r0 + rr][c] = clean ? finite_or_zero(s) : s;
            }
            __syncthreads();
        }
    }
    static __device__ __forceinline__ void add(float4 (&acc)[OWN], float4 v, const float* row) {
        const float2 x = *reinterpret_cast<const float2*>(row);
        acc[0] = make_float4(fmaf(v.x, x.x, acc[0].x), fmaf(v.y, x.x, acc[0].y), fmaf(v.z, x.x, acc[0].z), fmaf(v.w, x.x, acc[0].w));
        acc[1] = make_float4(fmaf(v.x, x.y, acc[1].x), fmaf(v.y, x.y, acc[1].y), fmaf(v.z, x.y, acc[1].z), fmaf(v.w, x.y, acc[1].w));
    }
};

// K W^T for windows of more than 128 rows: Y (m x keep, pitch ldu), 4 JG rows and 8 columns a block. In k_block_step a block would read all
// of K by itself.
template <int JG>
__global__ void __launch_bounds__(Apply<JG>::NT, 1) k_block_inner(BlockSmall b, int c1) {
    constexpr int NT = Apply<JG>::NT, cols = Apply<JG>::COLS;
    extern __shared__ __align__(16) float smem[];
    auto x = reinterpret_cast<typename Apply<JG>::Row*>(smem), y = x + b.m;
    Apply<JG>& apply = *reinterpret_cast<Apply<JG>*>(y + 4 * JG);
    const float* U = b.U + (int64_t)(c1 - 1) * b.U_stride;
    const float* K = c1 == 1 ? b.P : b.K + ((c1 - 1) & 1) * b.K_stride;
    const int j0 = blockIdx.x * cols, r0 = blockIdx.y * 4 * JG, rows = min(4 * JG, b.m - r0);
    chain_wait();
    chain_release();
    for (int t = threadIdx.x; t < b.m * cols; t += NT) x[t / cols][t % cols] = j0 + t % cols < b.keep ? __ldcg(U + (int64_t)(t / cols) * b.ldu + j0 + t % cols) : 0.f;
    __syncthreads();
    apply.run(K + r0, c1 == 1 ? b.ldP : b.ldk, b.m, rows, x, y, true);       // (a row whose norm is not finite: its coefficients are zero)
    for (int t = threadIdx.x; t < rows * cols; t += NT)
        if (j0 + t % cols < b.keep) b.Y[(int64_t)(r0 + t / cols) * b.ldu + j0 + t % cols] = y[t / cols][t % cols];
}

// Between two solves: see launch_block_step. Blocks 0 .. n_inner - 1 take 8 columns of W K W^T each (K W^T first, see also k_block_inner), the others 8 of
// the products with rows still to come. Bound by latency: every round trip to L2 counts. ahead: the launch follows a solve, so that
// everything but W was there before that solve began; it is fetched before the wait for it (K into shared memory where it fits).
template <int JG>
__global__ void __launch_bounds__(Apply<JG>::NT, 1) k_block_step(BlockSmall b, int c0, int c1, int col0, int col1, int n_inner, int n_cols, int late1, int ahead) {
    constexpr int NT = Apply<JG>::NT, cols = Apply<JG>::COLS;
    extern __shared__ __align__(16) float smem[];
    auto x = reinterpret_cast<typename Apply<JG>::Row*>(smem), y = x + b.m;  // [m] each
    Apply<JG>& apply = *reinterpret_cast<Apply<JG>*>(y + b.m);
    const int m = b.m, keep = b.keep, step = b.step, tid = threadIdx.x;
    if (!ahead) chain_wait();
    float* Kn = b.K + (c1 & 1) * b.K_stride;
    if ((int)blockIdx.x < n_inner) {
        const int j0 = blockIdx.x * cols;
        const float* U = b.U + (int64_t)(c1 - 1) * b.U_stride;
        if constexpr (JG == 16) {
            const float* K = c1 == 1 ? b.P : b.K + ((c1 - 1) & 1) * b.K_stride;
            const int64_t ldk = c1 == 1 ? b.ldP : b.ldk;
            float* Ks = reinterpret_cast<float*>(&apply + 1);
            const int m4 = (m + 3) & ~3;
            for (int t = tid; t < m * (m4 / 4); t += NT) {
                const int i = t / (m4 / 4), c = 4 * (t % (m4 / 4));
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(Ks + i * m4 + c)), "l"(K + i * ldk + c) : "memory");
            }
            if (ahead) chain_wait();
            chain_release();
            for (int t = tid; t < m * cols; t += NT) {
                const int i = t / cols, c = t % cols;
                x[i][c] = j0 + c < keep ? __ldcg(U + (int64_t)i * b.ldu + j0 + c) : 0.f;
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();
            apply.run(Ks, m4, m, m, x, y, true);                             // (a row whose norm is not finite: its coefficients are zero)
        } else {
            if (ahead) chain_wait();
            chain_release();
            for (int t = tid; t < m * cols; t += NT) y[t / cols][t % cols] = j0 + t % cols < keep ? __ldcg(b.Y + (int64_t)(t / cols) * b.ldu + j0 + t % cols) : 0.f;
            __syncthreads();
        }
        apply.run(U, b.ldu, m, keep, y, x, false);
        for (int t = tid; t < keep * cols; t += NT) {                       // one triangle, and its mirror image
            const int i = t / cols, j = j0 + t % cols;
            if (j < keep && i <= j) {
                const float v = x[i][t % cols];
                Kn[(int64_t)i * b.ldk + j] = v;
                Kn[(int64_t)j * b.ldk + i] = v;
            }
        }
        return;
    }
    int g0 = col0 + ((int)blockIdx.x - n_inner) * cols;
    if ((int)blockIdx.x >= n_inner + n_cols) {                               // columns that come late, from cycle 0 on
        g0 = col1 + ((int)blockIdx.x - n_inner - n_cols) * cols;
        c0 = 0;
        col1 = late1;
    }
    const float* top = c0 == 0 ? b.P : b.C;
    const int e0 = keep + c0 * step, w0 = keep + c1 * step;                  // the first rows behind the kept ones of windows c0 and c1
    for (int t = tid; t < keep * cols; t += NT) {
        const int i = t / cols, g = g0 + t % cols;
        float v = 0.f;
        if (g < e0 && c0 == 0) v = g == i ? 1.f : 0.f;                       // coefficients: rows of window c0 enter as themselves
        else if (g < col1 && (g < e0 || g >= e0 + step || c1 > c0 + 1)) v = __ldcg(top + (int64_t)i * b.ldP + g);
        x[i][t % cols] = v;
    }
    if (g0 + cols > w0 && g0 < w0 + step)                                   // products of the window's rows with each other, as far as they are there
        for (int t = tid; t < step * cols; t += NT) {
            const int i = t / cols, g = g0 + t % cols;
            if (g < w0 || g >= col1 || g >= w0 + step || w0 + i >= col1) continue;
            const float v = __ldcg(b.P + (int64_t)(w0 + i) * b.ldP + g);
            Kn[(int64_t)(keep + i) * b.ldk + keep + g - w0] = v;
            Kn[(int64_t)(keep + g - w0) * b.ldk + keep + i] = v;
        }
    for (int c = c0; c < c1; ++c) {
        const int e = keep + c * step;
        for (int t = tid; t < step * cols; t += NT) {
            const int i = t / cols, g = g0 + t % cols;
            float v = 0.f;
            if (g >= e + step) v = g < col1 ? __ldcg(b.P + (int64_t)(e + i) * b.ldP + g) : 0.f;
            else if (g >= e) v = g - e == i ? 1.f : 0.f;
            x[keep + i][t % cols] = v;
        }
        if (ahead) chain_wait();                                             // (one cycle then)
        __syncthreads();
        apply.run(b.U + (int64_t)c * b.U_stride, b.ldu, m, keep, x, y, false);
        for (int t = tid; t < keep * cols; t += NT) x[t / cols][t % cols] = y[t / cols][t % cols];
    }
    chain_release();
    __syncthreads();
    for (int t = tid; t < keep * cols; t += NT) {
        const int i = t / cols, g = g0 + t % cols;
        if (g >= col1) continue;
        const float v = x[i][t % cols];
        b.C[(int64_t)i * b.ldP + g] = v;
        if (g >= w0 && g < w0 + step) {
            Kn[(int64_t)i * b.ldk + keep + g - w0] = v;
            Kn[(int64_t)(keep + g - w0) * b.ldk + i] = v;
        }
    }
}

// The product of the W of a block's cycles, a few logical rows (columns of the product) to a thread block: a row enters with its cycle's W and is
// multiplied by the later ones. c_from: the cycles before it have been multiplied by k_block_step already (C). The last block fills the
// surplus planes of the three places with zeros.
template <int JG>
__global__ void __launch_bounds__(Apply<JG>::NT, 1) k_block_factors(BlockSmall b, BlockMap map, int c_from, int ncyc, int r_last, int keep_last, unsigned short* __restrict__ T, int j_pad,
                                                            int64_t ldT) {
    constexpr int NT = Apply<JG>::NT, cols = Apply<JG>::COLS;
    extern __shared__ __align__(16) float smem[];
    auto x = reinterpret_cast<typename Apply<JG>::Row*>(smem), y = x + b.m;
    Apply<JG>& apply = *reinterpret_cast<Apply<JG>*>(y + b.m);
    const int tid = threadIdx.x, keep = b.keep;
    chain_wait();
    chain_release();
    if (blockIdx.x == gridDim.x - 1) {
        const int from[3] = {3 * map.s_rows, map.oR + map.np * map.n_store, map.oI + map.n_in};
        const int to[3] = {map.oR, map.oI, (map.P + 63) / 64 * 64};
        for (int s = 0; s < 3; ++s)
            for (int t = tid; t < (to[s] - from[s]) * 3 * j_pad; t += NT) T[(int64_t)(t / (to[s] - from[s])) * ldT + from[s] + t % (to[s] - from[s])] = 0;
        return;
    }
    const int nl = block_rows(map), g0 = blockIdx.x * cols;
    auto enters = [&](int g) { return g < b.m ? 0 : (g - b.m) / b.step + 1; };
    for (int t = tid; t < b.m * cols; t += NT) {
        const int i = t / cols, g = g0 + t % cols;
        x[i][t % cols] = i < keep && g < nl && enters(g) < c_from ? __ldcg(b.C + (int64_t)i * b.ldP + g) : 0.f;
    }
    __syncthreads();
    for (int c = max(enters(g0), c_from); c < ncyc; ++c) {
        const bool last = c == ncyc - 1;
        const float* U = b.U + (int64_t)c * b.U_stride;
        const int wide = last ? keep_last : keep;
        apply.run(U, b.ldu, last ? min(keep, r_last) : keep, wide, x, y, false);
        for (int t = tid; t < wide * cols; t += NT) {
            const int j = t / cols, g = g0 + t % cols;
            float v = y[j][t % cols];
            if (g < nl && enters(g) == c) v = U[(int64_t)(g - c * b.step) * b.ldu + j];      // its place in window c
            x[j][t % cols] = v;
        }
        __syncthreads();
    }
    for (int t = tid; t < j_pad * cols; t += NT) {
        const int j = t / cols, g = g0 + t % cols;
        if (g >= nl) continue;
        float v = j < keep_last ? x[j][t % cols] : 0.f;
        const int p0 = block_phys(map, g), np = block_planes(map, g);
        for (int s = 0; s < 3; ++s) {
            const unsigned hi = __float_as_uint(v) & 0xffff0000u;
            v -= __uint_as_float(hi);
            for (int p = p0; p < p0 + np; ++p) T[(int64_t)(s * j_pad + j) * ldT + p] = (unsigned short)(hi >> 16);
        }
    }
}

template <int JG>
size_t small_smem(int m) { return (size_t)2 * m * sizeof(typename Apply<JG>::Row) + sizeof(Apply<JG>); }
constexpr int kSmallSmem = 160 * 1024;
// Windows of up to this many rows: the product of the W is carried along from step to step, beside the inner products (columns before
// the window of C). Larger ones have more columns than there are SMs as it is, and form it at the end of the block.
constexpr int kCarryRows = 128;

dim3 row_grid(int64_t cols, int per_thread, int64_t n) {
    const int64_t bx = std::min<int64_t>((cols + kThreads * per_thread - 1) / (kThreads * per_thread), 1184);
    return dim3((unsigned)bx, (unsigned)n);
}

}  // namespace

void allow_work_beside_capture(bool on) {
    static thread_local cudaStreamCaptureMode before = cudaStreamCaptureModeGlobal;
    cudaStreamCaptureMode mode = on ? cudaStreamCaptureModeRelaxed : before;
    if (cudaThreadExchangeStreamCaptureMode(&mode) == cudaSuccess && on) before = mode;
}

cudaError_t launch_block_append(const void* rows, sage_dtype_t dt, int64_t n, int64_t ld, int64_t D, __nv_bfloat16* R, int64_t pitch, int np,
                                int64_t row0, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const dim3 grid = row_grid(pitch, 8, n);
    const int es = dt == SAGE_F32 ? 4 : 2, vec = (reinterpret_cast<uintptr_t>(rows) & 15u) == 0 && (ld * es) % 16 == 0;
    if (dt == SAGE_F32) return launch_chained(k_block_append<float>, grid, dim3(kThreads), 0, st, static_cast<const float*>(rows), ld, D, R, pitch, np, row0, vec);
    return launch_chained(k_block_append<__nv_bfloat16>, grid, dim3(kThreads), 0, st, static_cast<const __nv_bfloat16*>(rows), ld, D, R, pitch, np, row0, vec);
}

cudaError_t launch_block_append_outer(const void* q, int64_t ldq, const void* feat, int64_t ldf, sage_dtype_t dt, int64_t n, int C, int F,
                                      __nv_bfloat16* R, int64_t pitch, int np, int64_t row0, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const dim3 grid = row_grid(pitch, 8, n);
    if (dt == SAGE_F32)
        return launch_chained(k_block_append_outer<float>, grid, dim3(kThreads), 0, st, static_cast<const float*>(q), ldq, static_cast<const float*>(feat), ldf, C, F, R,
                              pitch, np, row0);
    using bf = __nv_bfloat16;
    return launch_chained(k_block_append_outer<bf>, grid, dim3(kThreads), 0, st, static_cast<const bf*>(q), ldq, static_cast<const bf*>(feat), ldf, C, F, R, pitch, np,
                          row0);
}

cudaError_t launch_block_unpack(const __nv_bfloat16* R, int64_t pitch, int np, int n, int64_t D, float* out, int64_t ldo, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    return launch_chained(k_block_unpack, row_grid(ldo, 1, n), dim3(kThreads), 0, st, R, pitch, np, D, out, ldo);
}

cudaError_t launch_block_gram_reduce(const float* parts, const BlockMap& map, int first_new, int slices, float* P, int ldP, cudaStream_t st) {
    const int nl = block_rows(map);
    if (first_new >= nl) return cudaSuccess;
    auto kernel = map.np == 1 && first_new >= map.s_rows ? k_block_gram_reduce<1> : k_block_gram_reduce<3>;
    return launch_chained(kernel, dim3((nl + 3) / 4, (nl - first_new + 31) / 32), dim3(256), 0, st, parts, map, first_new, slices, P, ldP);
}

cudaError_t launch_block_step(const BlockSmall& b, int c0, int c1, int col0, int col1, int late1, bool inner, cudaStream_t st) {
    if (inner && b.m <= kCarryRows) col0 = 0;
    constexpr int cols = Apply<16>::COLS;
    const int n_inner = inner ? (b.keep + cols - 1) / cols : 0, n_cols = col1 > col0 ? (col1 - col0 + cols - 1) / cols : 0;
    const int n_late = late1 > col1 ? (late1 - col1 + cols - 1) / cols : 0;
    if (n_inner + n_cols + n_late == 0) return cudaSuccess;
    auto go = [&](auto kernel, int threads, size_t smem) -> cudaError_t {
        const cudaError_t e = allow_smem((const void*)kernel, kSmallSmem);
        if (e != cudaSuccess) return e;
        return launch_chained(kernel, dim3(n_inner + n_cols + n_late), dim3(threads), smem, st, b, c0, c1, col0, col1, n_inner, n_cols, late1, inner && n_late == 0 ? 1 : 0);
    };
    if (inner && b.m > 128) {
        auto first = [&](auto kernel, int threads, int rows, size_t apply) -> cudaError_t {
            const cudaError_t e = allow_smem((const void*)kernel, kSmallSmem);
            if (e != cudaSuccess) return e;
            return launch_chained(kernel, dim3(n_inner, (b.m + rows - 1) / rows), dim3(threads), (size_t)(b.m + rows) * cols * sizeof(float) + apply, st, b, c1);
        };
        const cudaError_t e = b.m <= 256 ? first(k_block_inner<16>, Apply<16>::NT, 64, sizeof(Apply<16>)) : first(k_block_inner<32>, Apply<32>::NT, 128, sizeof(Apply<32>));
        if (e != cudaSuccess) return e;
    }
    if (b.m <= 128) return go(k_block_step<16>, Apply<16>::NT, small_smem<16>(b.m) + (inner ? (size_t)b.m * ((b.m + 3) & ~3) * sizeof(float) : 0));
    if (b.m <= 256) return go(k_block_step<32>, Apply<32>::NT, small_smem<32>(b.m));
    return go(k_block_step<64>, Apply<64>::NT, small_smem<64>(b.m));
}

cudaError_t launch_block_factors(const BlockSmall& b, const BlockMap& map, int carried, int ncyc, int r_last, int keep_last, __nv_bfloat16* T, int j_pad, int64_t ldT,
                                 cudaStream_t st) {
    auto go = [&](auto kernel, int threads, size_t smem) -> cudaError_t {
        const cudaError_t e = allow_smem((const void*)kernel, kSmallSmem);
        if (e != cudaSuccess) return e;
        return launch_chained(kernel, dim3((block_rows(map) + Apply<16>::COLS - 1) / Apply<16>::COLS + 1), dim3(threads), smem, st, b, map, b.m <= kCarryRows ? carried : 0, ncyc, r_last, keep_last,
                              reinterpret_cast<unsigned short*>(T), j_pad, ldT);
    };
    if (b.m <= 128) return go(k_block_factors<16>, Apply<16>::NT, small_smem<16>(b.m));
    if (b.m <= 256) return go(k_block_factors<32>, Apply<32>::NT, small_smem<32>(b.m));
    return go(k_block_factors<64>, Apply<64>::NT, small_smem<64>(b.m));
}

}  // namespace sage
