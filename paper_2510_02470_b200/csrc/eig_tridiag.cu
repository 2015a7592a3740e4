// Eigen-decomposition of the buffer's Gram matrix and the Frequent-Directions shrink factors (Method, first
// paragraph: the buffer's thin SVD is taken, delta is the squared ell-th singular value, and every squared singular
// value is reduced by delta and clamped at zero). With K = B B^T = U Sigma^2 U^T the left factor U and sigma^2 come
// from the symmetric eigen-problem of K, and Sigma' V^T = diag(sigma'/sigma) U^T B.
//
// Method (direct; only the number of passes in step 2 depends on the data):
//   1. K is scaled by 1 / max diagonal, ordered by falling diagonal and reduced to a tridiagonal T = Q^T K Q by Householder
//      reflections, fp32, the matrix in registers (k_tridiag). n <= 128: one thread block of 4 warps; larger: a cluster of 8
//      blocks works until 128 rows are left, the one-block kernel does the rest.
//   2. Every wanted eigenvalue of T (the kept ones and delta) is found by multisection on the sign changes of the
//      leading principal minors, in fp64, one warp per eigenvalue, 32 places per pass over T, with secants at the end: four
//      passes where eigenvalues are apart, up to twenty in a cluster.
//   3. Its eigenvector is read off the forward and the backward three-term recurrence, joined where their product (the
//      diagonal of the resolvent) is largest, in fp64.
//   4. The reflections are applied to it in reverse (fp32, groups of four), it is scaled and written.
//   2-4 are one kernel (k_tridiag_vectors), three vectors per thread block, no communication between blocks.
// T is perturbed by less than half an ulp of fp32 (T's own rounding is larger) so that repeated eigenvalues of K come
// apart and vectors can be computed independently of each other. Gaps may be as small as 1e-11 of the largest eigenvalue, but the
// vectors across such a gap live at different places of T: rows of sketches were orthogonal to 1e-7 to 7e-7 of the largest squared
// row norm, 32 to 512 rows, over clusters of two, three and five values, eightfold eigenvalues, glued Wilkinson matrices and
// repeated Laplacians (the iterative solve: 7e-7 to 5e-4 on the same).
//
// Why: the solve is a chain of dependent steps, and this one is shorter than the iterative solve's (sweeps x (n - 1) rounds):
// n - 2 steps of about 1,050 cycles for the reduction, then 30 to 75 thousand cycles, all eigenvectors side by side. Measured, one
// solve in a row of solves, iterative -> direct: 64 rows 156 -> 46 us, 128 rows 377 -> 92 us, 256 rows 1,378 -> 214 us, 512 rows
// 6,479 -> 692 us (random matrices). Rows of low rank are the other way round: the iterative solve stops at the rank (rank 8 of 64,
// 128, 256, 512 rows: 25, 32, 55, 134 us) and this one does not: looking for the end of the rank cost its loop over the columns 3 to
// 12 % wherever it was put. Error of the shrunk sketch, relative to the
// largest eigenvalue: 3 to 5e-7 at every size (iterative: 1e-6 at 64 rows to 6e-6 at 512).
#include "sage_internal.h"

namespace sage {
namespace {

using u64 = unsigned long long;

// ---- pairs of fp32 values in one 64-bit register: one instruction for two multiply-adds --------------------
__device__ __forceinline__ u64 pk(float a, float b) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk(u64 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// ---- cluster exchange: asynchronous stores that count their bytes on a barrier of the receiving block -----------
__device__ __forceinline__ uint32_t s_addr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ uint32_t map_to_cta(uint32_t local, uint32_t cta) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(cta));
    return r;
}
__device__ __forceinline__ void send_pair(uint32_t addr, float x, float y, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(addr), "f"(x), "f"(y), "r"(bar)
                 : "memory");
}
constexpr long long kWaitCycles = 400000000ll;   // about 0.2 s
// A warp waits for a phase of a barrier of its block; gives up after kWaitCycles, or as soon as another block has (*abort).
// The same answer in every lane.
__device__ __forceinline__ bool wait_bytes(uint32_t bar, uint32_t parity, const int* abort) {
    long long t0 = 0;
    bool fine = true;
    for (int it = 0;; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n"
            ".reg .pred p;\n"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n"
            "}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) break;
        if ((it & 63) == 63) {
            if (t0 == 0) t0 = clock64();
            if (clock64() - t0 > kWaitCycles || __ldcg(abort) != 0) {
                fine = false;
                break;
            }
        }
    }
    return __all_sync(0xffffffffu, fine);
}

// ---- scratch of one solve (floats): reflectors, tridiagonal, what the cluster leaves, a header ---------------------
// G: 128, 256 or 512, the padded size. A matrix of n rows occupies positions o .. o + n - 1 of the G, o = (G - n) & ~3: the
// reduction ends at position G - 1 whatever n is, and rows stay 16-byte aligned.
struct TriWork {
    float* V;        // G x G: row k holds reflector k (positions > k; the quads that end before those are not written)
    float* tau;      // G
    float* d;        // G
    float* e;        // G: e[k] couples positions k and k + 1
    float* trail;    // 128 x 128
    float* dmax;     // the scale K was divided by
    int* abort;      // raised by a block that gave up a wait
    int* perm;       // G: row of K at each place of its order by falling diagonal
};
__host__ __device__ inline TriWork tri_work(float* w, int G) {
    TriWork t;
    t.V = w;
    t.tau = w + (size_t)G * G;
    t.d = t.tau + G;
    t.e = t.d + G;
    t.trail = t.e + G;
    t.dmax = t.trail + 128 * 128;
    t.abort = reinterpret_cast<int*>(t.dmax + 1);
    t.perm = t.abort + 3;
    return t;
}

// ---- Householder tridiagonalisation ---------------------------------------------------------------------------------
// Thread tile: RI rows x 16 columns in registers (column pairs packed). Lane (lr, lc) of warp w of block cta holds rows
// i RB + (cta W + w) LR + lr and columns q CB + 4 lc + s (q, s = 0 .. 3): as the reduction proceeds whole slots i and q
// die and the code for phase Q0 leaves them out.
template <int LC_, int W_, int RI_, int CL_>
struct TriShape {
    static constexpr int LC = LC_, W = W_, RI = RI_, CL = CL_;
    static constexpr int LR = 32 / LC, NT = 32 * W, G = 16 * LC, RB = CL * W * LR, CB = 4 * LC;
    static constexpr int LAST = CL == 1 ? G - 2 : G - 128;      // last column this kernel looks at
    static_assert(RI * RB == G, "");
};
using Tri128 = TriShape<8, 4, 8, 1>;      // 8 warps of half the rows each: 107 us instead of 90 for a solve of 128 rows
using Tri256 = TriShape<16, 4, 4, 8>;
using Tri512 = TriShape<32, 8, 8, 8>;

__host__ __device__ constexpr int pow2_at_least(int v) { return v <= 1 ? 1 : v <= 2 ? 2 : v <= 4 ? 4 : 8; }
__host__ __device__ constexpr int log2_of(int v) { return v <= 1 ? 0 : 1 + log2_of(v / 2); }

// Sums R values over the lanes that differ in the bits below 2 X: halves the values and the lanes at each level while there
// are values to halve, so that lane group lc ends up with value lc >> (log2(LC) - log2(R)).
template <int R, int X>
__device__ __forceinline__ float lane_sums(float (&y)[R], int lc) {
    if constexpr (X == 0) {
        return y[0];
    } else if constexpr (R > 1) {
        const bool up = (lc & X) != 0;
        float z[R / 2];
#pragma unroll
        for (int j = 0; j < R / 2; ++j) {
            const float keep = up ? y[j + R / 2] : y[j], give = up ? y[j] : y[j + R / 2];
            z[j] = keep + __shfl_xor_sync(0xffffffffu, give, X);
        }
        return lane_sums<R / 2, X / 2>(z, lc);
    } else {
        float z[1] = {y[0] + __shfl_xor_sync(0xffffffffu, y[0], X)};
        return lane_sums<1, X / 2>(z, lc);
    }
}

template <typename S>
struct TriShared {
    float2 x[2][S::G];                       // (A v, column kk of A) by row, alternate steps (one block: two arrays, y then column)
    float rows[2][S::W][S::LR][2][S::RI];    // the same for a warp's own rows
    float g[2][S::W][S::LR];                 // a^T A a, one part per warp and lane row (one-block form)
    __align__(16) unsigned key[S::G];        // the diagonal's leading bits, and the row in the others: larger key, earlier place
    __align__(16) unsigned short col[S::G];  // row of K at each place, or the zero column of the staged rows
    float red[S::W];
    u64 bar[2];
};
template <typename S>
constexpr int kOwnRows = S::G / S::CL;       // rows of the tile of a block

template <typename S>
struct TriState {
    u64 A[S::RI][8];
    u64 vc[8];           // a at this thread's columns, packed pairs; zero where position < kk
    float vr[S::RI];     // a at this thread's rows
    float y[S::RI];      // A a: this thread's part (its columns) of its rows
    float ak, b, tau;    // a at position kk; the reflector is v = a + b e_kk, H = I - tau v v^T
};

__device__ __forceinline__ float rsqrt_fast(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_fast(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float pick(const float (&t)[4], int s) { return (s & 2) ? ((s & 1) ? t[3] : t[2]) : ((s & 1) ? t[1] : t[0]); }

// Columns kk of phase Q0 (positions Q0 CB .. Q0 CB + CB - 1). Entering, the column before kk (below its diagonal) is a, its
// reflector v = a + b e_kk, not yet applied, and A a is known: with y = A v = A a + b A e_kk and
// w = tau y - (tau^2 v^T y / 2) v the update is A -= v w^T + w v^T, and column kk after it follows from the same vectors.
// One exchange of (y, A e_kk) between warps (blocks) per column; everything else is computed by every thread for its own rows and
// columns. The norm of the new column, its square root and the reciprocal only enter through b and tau: they overlap with the update
// of the tile and the product with the new column. Positions that are done keep being transformed like the others (their part
// of A is not used again, and a is zero there); only a is masked. What bounds it: n - 2 dependent steps, each the exchange, a few dozen
// dependent operations, 3 multiply-adds per element of the tile and log2(LC) shuffles.
template <typename S, int Q0>
__device__ __forceinline__ bool tri_phase(TriState<S>& T, TriShared<S>& sh, int o, const TriWork& wk, int base, int pitch, int cta, int w, int lr, int lc) {
    constexpr int LC = S::LC, RI = S::RI, RB = S::RB, CB = S::CB, CL = S::CL;
    constexpr int P0 = 2 * Q0;                              // first live column pair
    constexpr int NB = CB / RB, I0 = Q0 * NB;               // first live row slot; slots I0 .. I0 + NB - 1 hold kk's block
    constexpr int NR = RI - I0, R = pow2_at_least(NR);      // live row slots, rounded up for the lane sums
    constexpr int REP = LC / R;                             // lanes that end up with the same row
    const int rowbase = (cta * S::W + w) * S::LR + lr;
    const int irow = RI - R + (lc >> (log2_of(LC) - log2_of(R)));
    const int rglob = irow * RB + rowbase;
    const int kbeg = o > Q0 * CB ? o : Q0 * CB;
    const int kend = S::LAST < Q0 * CB + CB - 1 ? S::LAST : Q0 * CB + CB - 1;
    auto step = [&](int kk, int sk) -> bool {               // sk = kk % 4: element of position kk in its lane's four columns
        const int b = sk & 1;
        const int lk = (kk >> 2) & (LC - 1);                // lane column of position kk
        const int d0 = kk - (CB * Q0 + 4 * lc);             // position kk is this thread's element d0 of slot Q0
        float2* xb = sh.x[b];
        float* yb = reinterpret_cast<float*>(xb);           // one block: y, then column kk
        float* cb = yb + S::G;
        if constexpr (CL > 1) {
            if (threadIdx.x == 0)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s_addr(&sh.bar[b])), "r"(NR * RB * 8) : "memory");
        }
        // column kk of the warp's rows, from the lanes that hold it to the lanes that send it
        float* rows_y = sh.rows[b][w][lr][0];
        float* rows_c = sh.rows[b][w][lr][1];
        {
            float t[RI];
            t[I0 & ~1] = 0.f;
#pragma unroll
            for (int i = I0; i < RI; ++i) {
                float a0, a1;
                upk((sk & 2) ? T.A[i][P0 + 1] : T.A[i][P0], a0, a1);
                t[i] = (sk & 1) ? a1 : a0;
            }
            if (lc == lk) {
#pragma unroll
                for (int i = I0 & ~1; i < RI; i += 2) *reinterpret_cast<float2*>(rows_c + i) = make_float2(t[i], t[i + 1]);
            }
        }
        float gp = 0.f, y[R];
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int i = RI - R + j;
            y[j] = i >= I0 ? T.y[i] : 0.f;
            if (i >= I0) gp = fmaf(T.vr[i], T.y[i], gp);
        }
        float ysum = lane_sums<R, LC / 2>(y, lc);
        if constexpr (CL == 1) {
#pragma unroll
            for (int x = LC / 2; x > 0; x >>= 1) gp += __shfl_xor_sync(0xffffffffu, gp, x);
        }
        __syncwarp();
        const float cval = rows_c[irow];
        ysum = fmaf(T.b, cval, ysum);
        rows_y[irow] = ysum;
        if constexpr (CL == 1) {
            if (irow >= I0) {
                yb[rglob] = ysum;
                cb[rglob] = cval;
            }
            if (lc == 0) sh.g[b][w][lr] = gp;
            __syncthreads();
        } else {
            if (irow >= I0) {
                const uint32_t la = s_addr(&xb[rglob]), lb = s_addr(&sh.bar[b]);
                for (int t = lc & (REP - 1); t < CL; t += REP) send_pair(map_to_cta(la, t), ysum, cval, map_to_cta(lb, t));
            }
            if (!wait_bytes(s_addr(&sh.bar[b]), (sk >> 1) & 1, wk.abort)) return false;
            __syncwarp();                                   // rows_y and rows_c, written by other lanes
        }
        // both vectors at this thread's columns (pairs) and rows
        const float2 xk = CL == 1 ? make_float2(yb[kk], cb[kk]) : xb[kk];
        u64 yc[8], a2[8], nw[8];
#pragma unroll
        for (int q = Q0; q < 4; ++q) {
            if constexpr (CL == 1) {
                const float4 t0 = *reinterpret_cast<const float4*>(yb + CB * q + 4 * lc);
                const float4 t1 = *reinterpret_cast<const float4*>(cb + CB * q + 4 * lc);
                yc[2 * q] = pk(t0.x, t0.y);
                yc[2 * q + 1] = pk(t0.z, t0.w);
                a2[2 * q] = pk(t1.x, t1.y);
                a2[2 * q + 1] = pk(t1.z, t1.w);
            } else {
                const float4 t0 = *reinterpret_cast<const float4*>(&xb[CB * q + 4 * lc]);
                const float4 t1 = *reinterpret_cast<const float4*>(&xb[CB * q + 4 * lc + 2]);
                yc[2 * q] = pk(t0.x, t0.z);
                yc[2 * q + 1] = pk(t1.x, t1.z);
                a2[2 * q] = pk(t0.y, t0.w);
                a2[2 * q + 1] = pk(t1.y, t1.w);
            }
        }
        float g;                                            // v^T A v
        if constexpr (CL == 1) {
            float t[S::W];
#pragma unroll
            for (int j = 0; j < S::W; ++j) {
                const float4 u = *reinterpret_cast<const float4*>(&sh.g[b][j][0]);
                t[j] = (u.x + u.y) + (u.z + u.w);
            }
#pragma unroll
            for (int x = S::W / 2; x > 0; x >>= 1)
#pragma unroll
                for (int j = 0; j < x; ++j) t[j] += t[j + x];
            g = fmaf(T.b, fmaf(-T.b, xk.y, 2.f * xk.x), t[0]);
        } else {
            u64 acc = mul2(yc[P0], T.vc[P0]), acc1 = mul2(yc[P0 + 1], T.vc[P0 + 1]);
#pragma unroll
            for (int p = P0 + 2; p < 8; p += 2) {
                acc = fma2(yc[p], T.vc[p], acc);
                acc1 = fma2(yc[p + 1], T.vc[p + 1], acc1);
            }
            float a0, a1, a3, a4;
            upk(acc, a0, a1);
            upk(acc1, a3, a4);
            g = (a0 + a1) + (a3 + a4);
#pragma unroll
            for (int x = LC / 2; x > 0; x >>= 1) g += __shfl_xor_sync(0xffffffffu, g, x);
            g = fmaf(T.b, xk.x, g);
        }
        const float c = (0.5f * T.tau) * (T.tau * g);       // in this order: tau alone may be 1e30
        const float v1 = T.ak + T.b;
        const float nw1 = fmaf(v1, c, __fmul_rn(xk.x, -T.tau));   // -w at position kk
        {                                                   // from a to v
            float t[4];
            upk(T.vc[P0], t[0], t[1]);
            upk(T.vc[P0 + 1], t[2], t[3]);
#pragma unroll
            for (int s = 0; s < 4; ++s)
                if (d0 == s) t[s] = v1;
            T.vc[P0] = pk(t[0], t[1]);
            T.vc[P0 + 1] = pk(t[2], t[3]);
#pragma unroll
            for (int i = I0; i < I0 + NB; ++i)
                if (i * RB + rowbase == kk) T.vr[i] = v1;
        }
        const u64 nt2 = pk(-T.tau, -T.tau), c2 = pk(c, c), v12 = pk(v1, v1), nw12 = pk(nw1, nw1);
#pragma unroll
        for (int p = P0; p < 8; ++p) {
            nw[p] = fma2(T.vc[p], c2, mul2(yc[p], nt2));    // -w
            a2[p] = fma2(T.vc[p], nw12, fma2(nw[p], v12, a2[p]));
        }
        float ak[4];                                        // column kk (after the update) at slot Q0, then masked
        upk(a2[P0], ak[0], ak[1]);
        upk(a2[P0 + 1], ak[2], ak[3]);
        const float dk = pick(ak, sk);
#pragma unroll
        for (int s = 0; s < 4; ++s)
            if (d0 >= s) ak[s] = 0.f;
        a2[P0] = pk(ak[0], ak[1]);
        a2[P0 + 1] = pk(ak[2], ak[3]);
        u64 sq0 = mul2(a2[P0], a2[P0]), sq1 = mul2(a2[P0 + 1], a2[P0 + 1]);
#pragma unroll
        for (int p = P0 + 2; p < 8; p += 2) {
            sq0 = fma2(a2[p], a2[p], sq0);
            sq1 = fma2(a2[p + 1], a2[p + 1], sq1);
        }
        float s0, s1, s2, s3;
        upk(sq0, s0, s1);
        upk(sq1, s2, s3);
        s0 = (s0 + s1) + (s2 + s3);
        // position kk + 1: the next element, the next lane's first, or the first of slot Q0 + 1
        float an = pick(ak, (kk + 1) & 3);
        if (Q0 < 3) {
            float t0, t1;
            upk(a2[P0 + 2 < 8 ? P0 + 2 : 7], t0, t1);
            if (kk == Q0 * CB + CB - 1) an = t0;
        }
        an = __shfl_sync(0xffffffffu, an, ((kk + 1) >> 2) & (LC - 1), LC);
#pragma unroll
        for (int x = LC / 2; x > 0; x >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, x);
        // The same two vectors at this thread's rows, with the same operations in the same order as for the columns (a lives in
        // both forms from step to step, and a rounding difference between the two would be multiplied at every step); the update
        // of the tile and its product with the new column.
        float vsel[4];                                      // the reflector at the slot this warp writes
        upk(T.vc[P0], vsel[0], vsel[1]);
        upk(T.vc[P0 + 1], vsel[2], vsel[3]);
#pragma unroll
        for (int q = Q0 + 1; q < 4; ++q) {
            float t[4];
            upk(T.vc[2 * q], t[0], t[1]);
            upk(T.vc[2 * q + 1], t[2], t[3]);
#pragma unroll
            for (int s = 0; s < 4; ++s) vsel[s] = w == q ? t[s] : vsel[s];
        }
        float xy[RI], xc[RI];
#pragma unroll
        for (int i = I0 & ~1; i < RI; i += 2) {
            const float2 t0 = *reinterpret_cast<const float2*>(rows_y + i), t1 = *reinterpret_cast<const float2*>(rows_c + i);
            xy[i] = t0.x;
            xy[i + 1] = t0.y;
            xc[i] = t1.x;
            xc[i + 1] = t1.y;
        }
#pragma unroll
        for (int i = I0; i < RI; ++i) {
            const float nwr = fmaf(T.vr[i], c, __fmul_rn(xy[i], -T.tau));
            const int r = i * RB + rowbase;
            float ar = fmaf(T.vr[i], nw1, fmaf(nwr, v1, xc[i]));
            if (i < I0 + NB && r <= kk) ar = 0.f;
            const u64 v2 = pk(T.vr[i], T.vr[i]), n2 = pk(nwr, nwr);
            T.vr[i] = ar;
            u64 acc = 0ull;
#pragma unroll
            for (int p = P0; p < 8; ++p) {
                T.A[i][p] = fma2(n2, T.vc[p], fma2(v2, nw[p], T.A[i][p]));
                acc = fma2(T.A[i][p], a2[p], acc);
            }
            float a0, a1;
            upk(acc, a0, a1);
            T.y[i] = a0 + a1;
        }
        // results: the reflector of the column before (each warp a slot), its scalars, this column's diagonal
        if (cta == 0 && lr == 0 && w >= Q0 && w < 4 && kk > o)
            *reinterpret_cast<float4*>(wk.V + (size_t)(base + kk - 1) * pitch + base + CB * w + 4 * lc) = make_float4(vsel[0], vsel[1], vsel[2], vsel[3]);
        if (cta == 0 && w == 0 && lr == 0 && lc == lk) {
            wk.d[base + kk] = dk;
            if (kk > o) {
                wk.e[base + kk - 1] = -T.b;
                wk.tau[base + kk - 1] = T.tau;
            }
            if (CL == 1 && kk == S::LAST) wk.e[base + kk] = an;
        }
#pragma unroll
        for (int p = P0; p < 8; ++p) T.vc[p] = a2[p];
        // The reflector of column kk: b = sign(a_1) ||a||, tau = 2 / v^T v from the norm of this very v (no cancellation), so that
        // I - tau v v^T is orthogonal to rounding whatever the error of the square root.
        const float beta = s0 * rsqrt_fast(s0);
        const float vv = fmaf(beta, fmaf(2.f, fabsf(an), beta), s0);
        float q = rcp_fast(vv);
        q = fmaf(q, fmaf(-vv, q, 1.f), q);
        const bool some = s0 > 1e-30f;
        T.ak = an;
        T.b = some ? copysignf(beta, an) : 0.f;
        T.tau = some ? 2.f * q : 0.f;
        return true;
    };
#pragma unroll 1
    for (int kk = kbeg; kk <= kend; kk += 2) {              // kbeg is a multiple of 4; two steps, by four the code outgrows the instruction cache
        if (!step(kk, kk & 2)) return false;
        if (kk == kend) break;
        if (!step(kk + 1, (kk & 2) | 1)) return false;
    }
    return true;
}

// The rows are taken in order of falling diagonal. Reflections that start with the large rows leave the small ones' relative accuracy
// alone; in any other order a small eigenvalue is as uncertain as 1e-7 of the largest one. Rows of a sketch are so spread by
// construction, and gradients with heavy-tailed norms are. 64 rows, norms spread over a factor of 1,000 in no order, frozen: cosines
// between rows of the sketch 5e-3 -> 2e-5, singular values off by 1e-2 -> 2e-7 of themselves (they are x^T K x at a freeze).
// The diagonal and the places come before the tile, which is gathered from rows staged in shared memory: 2 to 3 us of 45 to 92 for 64
// to 128 rows, nothing measurable of 215 and 690 us for 256 and 512.
template <typename S>
__global__ void __launch_bounds__(S::NT, 1)
k_tridiag(const float* __restrict__ K, int ldk, int n, int scaled, TriWork wk, int base, int pitch, EigInfo* __restrict__ info) {
    __shared__ __align__(16) TriShared<S> sh;
    extern __shared__ __align__(16) float staged[];         // rows of K and a zero column (not for a matrix that comes scaled)
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, lr = lane / S::LC, lc = lane % S::LC;
    const int cta = S::CL == 1 ? 0 : (int)blockIdx.x;
    const int o = (S::G - n) & ~3, n4 = (n + 3) & ~3;
    chain_wait();
    TriState<S> T;
    if (S::CL == 1 && scaled) {                             // what a cluster left: every position in use, the order is made
#pragma unroll
        for (int i = 0; i < S::RI; ++i) {
            const int r = i * S::RB + (cta * S::W + w) * S::LR + lr;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 x = *reinterpret_cast<const float4*>(K + (size_t)r * ldk + q * S::CB + 4 * lc);
                T.A[i][2 * q] = pk(x.x, x.y);
                T.A[i][2 * q + 1] = pk(x.z, x.w);
            }
        }
    } else {
        const int ps = n4 + 4;                              // pitch of a staged row; columns n4 .. n4 + 3 are zero
        auto stage = [&](int row, int place) {              // by a warp
            for (int c = 4 * lane; c < n4; c += 128)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s_addr(staged + (size_t)place * ps + c)), "l"(K + (size_t)row * ldk + c) : "memory");
            if (lane == 0) *reinterpret_cast<float4*>(staged + (size_t)place * ps + n4) = make_float4(0.f, 0.f, 0.f, 0.f);
        };
        if (S::CL == 1)                                     // one block stages all rows while it looks at the diagonal, a cluster's blocks their own
            for (int r = w; r < n; r += S::W) stage(r, r);
        // scale by the largest finite diagonal; rows whose norm is not finite take no part
        constexpr int MINE = S::G / S::NT;                  // rows that a thread ranks
        float dm = 0.f;
        unsigned mine[MINE];
        bool fin[MINE];
#pragma unroll
        for (int u = 0; u < MINE; ++u) {
            const int i = tid + u * S::NT;
            const float v = i < n ? K[(size_t)i * ldk + i] : 0.f;
            fin[u] = fabsf(v) <= 3.0e38f;
            dm = fin[u] ? fmaxf(dm, v) : dm;
            mine[u] = i < n ? ((fin[u] ? __float_as_uint(fmaxf(v, 0.f)) : 0u) & ~511u) | (unsigned)(511 - i) : 0u;
            sh.key[i] = mine[u];
            if (!fin[u] && cta == 0) atomicOr(&info->flags, kFlagNonFinite);
        }
#pragma unroll
        for (int x = 16; x > 0; x >>= 1) dm = fmaxf(dm, __shfl_xor_sync(0xffffffffu, dm, x));
        if (lane == 0) sh.red[w] = dm;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < S::W; ++j) dm = fmaxf(dm, sh.red[j]);
        if (!(dm >= 1e-30f)) dm = 0.f;                      // nothing to factor
        const float kscale = dm > 0.f ? 1.f / dm : 0.f;
        if (cta == 0 && tid == 0) *wk.dmax = dm;
        int place[MINE];                                    // of a row: how many come before it
#pragma unroll
        for (int u = 0; u < MINE; ++u) place[u] = 0;
#pragma unroll 4
        for (int j = 0; j < n4; j += 4) {
            const uint4 k = *reinterpret_cast<const uint4*>(&sh.key[j]);
#pragma unroll
            for (int u = 0; u < MINE; ++u) place[u] += (k.x > mine[u]) + (k.y > mine[u]) + (k.z > mine[u]) + (k.w > mine[u]);
        }
#pragma unroll
        for (int u = 0; u < MINE; ++u) {
            const int i = tid + u * S::NT, p = i < n ? place[u] : i;
            sh.col[p] = (unsigned short)(i < n && fin[u] ? i : n4);
            if (cta == 0) wk.perm[p] = i;
        }
        __syncthreads();
        if (S::CL > 1) {
            for (int t = w; t < kOwnRows<S>; t += S::W) {   // place t: slot t / (W LR) of the block's rows
                const int p = (t / (S::W * S::LR)) * S::RB + cta * S::W * S::LR + t % (S::W * S::LR) - o;
                if (p >= 0 && p < n && sh.col[p] < n4) stage(sh.col[p], t);
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int c = q * S::CB + 4 * lc - o;
            const ushort4 pc = c >= 0 ? *reinterpret_cast<const ushort4*>(&sh.col[c]) : make_ushort4(n4, n4, n4, n4);
#pragma unroll
            for (int i = 0; i < S::RI; ++i) {
                const int p = i * S::RB + (cta * S::W + w) * S::LR + lr - o;
                const int row = p >= 0 ? sh.col[p] : n4;
                float t[4] = {0.f, 0.f, 0.f, 0.f};
                if (row < n4) {
                    const float* src = staged + (size_t)(S::CL == 1 ? row : i * S::W * S::LR + w * S::LR + lr) * ps;
                    t[0] = src[pc.x] * kscale;
                    t[1] = src[pc.y] * kscale;
                    t[2] = src[pc.z] * kscale;
                    t[3] = src[pc.w] * kscale;
                }
                T.A[i][2 * q] = pk(t[0], t[1]);
                T.A[i][2 * q + 1] = pk(t[2], t[3]);
            }
        }
    }
    if constexpr (S::CL > 1) {
        if (tid < 2) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(s_addr(&sh.bar[tid])) : "memory");
        if (tid == 0) {
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            if (cta == 0) *wk.abort = 0;
        }
    }
#pragma unroll
    for (int i = 0; i < S::RI; ++i) T.vr[i] = T.y[i] = 0.f;
#pragma unroll
    for (int p = 0; p < 8; ++p) T.vc[p] = 0ull;
    T.ak = T.b = T.tau = 0.f;
    if constexpr (S::CL > 1) {
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    bool ok = tri_phase<S, 0>(T, sh, o, wk, base, pitch, cta, w, lr, lc);
    ok = ok && tri_phase<S, 1>(T, sh, o, wk, base, pitch, cta, w, lr, lc);
    ok = ok && tri_phase<S, 2>(T, sh, o, wk, base, pitch, cta, w, lr, lc);
    chain_release();
    if constexpr (S::G != 256) ok = ok && tri_phase<S, 3>(T, sh, o, wk, base, pitch, cta, w, lr, lc);
    if constexpr (S::CL == 1) {
        if (tid == S::NT - 1) {                             // the last diagonal element; two positions have no reflector
            float a0, a1;
            upk(T.A[S::RI - 1][7], a0, a1);
            wk.d[base + S::G - 1] = a1;
            wk.e[base + S::G - 1] = 0.f;
            wk.tau[base + S::G - 1] = 0.f;
        }
    } else {
        if (!ok && lane == 0) {
            atomicOr(&info->flags, kFlagExchangeTimeout);
            atomicExch(wk.abort, 1);
        }
        constexpr int B0 = S::G - 128;                      // the 128 x 128 block that is left
#pragma unroll
        for (int i = 0; i < S::RI; ++i) {
            const int r = i * S::RB + (cta * S::W + w) * S::LR + lr - B0;
            if (r < 0) continue;
#pragma unroll
            for (int q = B0 / S::CB; q < 4; ++q) {
                float t0, t1, t2, t3;
                upk(T.A[i][2 * q], t0, t1);
                upk(T.A[i][2 * q + 1], t2, t3);
                *reinterpret_cast<float4*>(wk.trail + (size_t)r * 128 + (q * S::CB + 4 * lc - B0)) = make_float4(t0, t1, t2, t3);
            }
        }
        // no block leaves while another may still store into its shared memory
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// ---- eigenvalues, eigenvectors, factors -----------------------------------------------------------------------------
constexpr int kVecWarps = 3;                       // eigenvectors per block, a warp each
constexpr int kEvWarps = kVecWarps + 1;            // one more finds delta: one of these warps per scheduler
constexpr int kHelpWarps = 4;                      // inner products of reflectors, meanwhile
constexpr int kVecThreads = 32 * (kEvWarps + kHelpWarps);
constexpr int kChunk = 16;                         // reflectors per chunk in shared memory
constexpr int kPoints = 32 * kEvWarps;             // places of the first cut, shared by the block's eigenvalues
constexpr double kRankCut = 1e-7;                  // eigenvalues below this fraction of the largest diagonal count as zero (rounding of K and T)
template <int NQ>
constexpr int kRing = NQ == 4 ? 4 : 8;             // chunks in flight (all of them when n <= 128)

__device__ __forceinline__ double pow2(int ex) {   // 2^ex, 0 below the normal range
    return ex < -1022 ? 0.0 : __hiloint2double((1023 + (ex > 1023 ? 1023 : ex)) << 20, 0);
}
__device__ __forceinline__ int exponent_of(double a, double b) {   // of the larger magnitude, biased
    return max(__double2hiint(a) & 0x7ff00000, __double2hiint(b) & 0x7ff00000) >> 20;
}

// Number of eigenvalues of the N x N tridiagonal below x (|x| <= 1/2): sign changes of its leading principal minors,
// p_{i+1} = (d_i - x) p_i - e_{i-1}^2 p_{i-1}. Run from both ends to the middle row (two dependent chains of half the length),
// where the sign of the remaining pivot follows from the determinant. up[s] = (d_i, -e_{i-1}^2) and down[s] = (d_i, -e_i^2) in the
// order they are taken, M of each, a multiple of 16, filled up in front with (1, 0), which changes no sign; mid = (d_h, -e_{h-1}^2,
// -e_h^2). Rescaled by powers of two every 8 rows; the sign bits are shifted into a word, changes counted 8 at a time.
// det 2^ex receives the determinant of T - x.
__device__ __forceinline__ int count_below(const double2* up, const double2* down, const double (&mid)[3], int M, double x, double& det, int& ex) {
    double p = 1.0, pm = 0.0, q = 1.0, qm = 0.0;
    unsigned sp = 0u, sq = 0u;
    int cnt = 0;
    ex = 0;
    auto load = [&](int i, double2 (&t)[8], double2 (&u)[8]) {
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            t[s] = up[i + s];
            u[s] = down[i + s];
        }
    };
    auto rows = [&](const double2 (&t)[8], const double2 (&u)[8]) {
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            const double pn = fma(t[s].x - x, p, t[s].y * pm), qn = fma(u[s].x - x, q, u[s].y * qm);
            sp = __funnelshift_l((unsigned)__double2hiint(pn), sp, 1);
            sq = __funnelshift_l((unsigned)__double2hiint(qn), sq, 1);
            pm = p;
            p = pn;
            qm = q;
            q = qn;
        }
        cnt += __popc((sp ^ (sp >> 1)) & 0xffu) + __popc((sq ^ (sq >> 1)) & 0xffu);
        const int ep = min(exponent_of(p, pm), 2045), eq = min(exponent_of(q, qm), 2045);
        const double fp = __hiloint2double((2046 - ep) << 20, 0), fq = __hiloint2double((2046 - eq) << 20, 0);
        ex += ep + eq - 2046;
        p *= fp;
        pm *= fp;
        q *= fq;
        qm *= fq;
    };
    double2 t0[8], u0[8], t1[8], u1[8];
    load(0, t0, u0);
#pragma unroll 1
    for (int i = 0; i < M; i += 16) {
        load(i + 8, t1, u1);
        rows(t0, u0);
        load(i + 16 < M ? i + 16 : 0, t0, u0);
        rows(t1, u1);
    }
    det = fma(fma(mid[0] - x, p, mid[1] * pm), q, mid[2] * p * qm);
    return cnt + (int)(((unsigned)(__double2hiint(det) ^ __double2hiint(p) ^ __double2hiint(q))) >> 31);
}

// The eigenvalue with `below` smaller ones, by one warp: each pass over T cuts the interval at 32 places. first: counts at the
// kPoints places that cut (-1/2, 1/2) evenly.
__device__ __forceinline__ double eigenvalue(const double2* up, const double2* down, const double (&mid)[3], int M, int below, const int* first,
                                             int lane) {
    double lo = -0.5, hi = 0.5;
    int k = 0;
#pragma unroll
    for (int j = 0; j < kPoints / 32; ++j) k += __popc(__ballot_sync(0xffffffffu, first[32 * j + lane] <= below));
    double h = 1.0 / (kPoints + 1);
    if (k < kPoints) hi = fma(h, (double)(k + 1), lo);
    if (k > 0) lo = fma(h, (double)k, lo);
    // The secant through the determinants at the two places around an eigenvalue is off by no more than their distance squared over
    // four times the distance to the next eigenvalue, and that is at least the distance to the ends of an interval in which the
    // eigenvalue is known to be alone. Even cuts until the places are near by that measure, then cuts whose places close in on the
    // secant from both sides, each four times nearer than the one before; the last secant is exact to rounding. Four cuts where
    // eigenvalues are apart (even cuts alone: seven). In a cluster even cuts go on for longer.
    double lam = 0.5 * (lo + hi), ilo = lo, ihi = hi;
    bool alone = false;
    bool isolated = (k < kPoints ? first[k] : below + 1) == below + 1 && (k > 0 ? first[k - 1] : below) == below;
    for (int pass = 0; pass < 20; ++pass) {
        const double wid = hi - lo;
        double x;
        if (alone && 8.0 * wid < fmin(lam - ilo, ihi - lam)) {   // lanes 0 .. 15: lam - wid 4^-lane, lanes 16 .. 31: lam + wid 4^(lane - 31)
            const int e = lane < 16 ? lane : 31 - lane;
            const double off = wid * __hiloint2double((1023 - 2 * e) << 20, 0);
            x = lane < 16 ? fmax(lam - off, lo) : fmin(lam + off, hi);
        } else {
            x = lane == 31 ? hi : fma(wid * (1.0 / 31.0), (double)lane, lo);
        }
        double det;
        int ex;
        const int c = count_below(up, down, mid, M, x, det, ex);
        k = __popc(__ballot_sync(0xffffffffu, c <= below));
        const int a = min(max(k - 1, 0), 30), b = a + 1;   // lanes 0 and 31 are at lo and hi
        lo = __shfl_sync(0xffffffffu, x, a);
        hi = __shfl_sync(0xffffffffu, x, b);
        const double da = __shfl_sync(0xffffffffu, det, a), db = __shfl_sync(0xffffffffu, det, b);
        const int ea = __shfl_sync(0xffffffffu, ex, a), eb = __shfl_sync(0xffffffffu, ex, b);
        const int ca = __shfl_sync(0xffffffffu, c, a), cb = __shfl_sync(0xffffffffu, c, b);
        const double r = db / da * pow2(min(eb - ea, 1000));               // f(hi) / f(lo), negative with one eigenvalue between
        alone = cb == ca + 1 && r <= 0.0;
        lam = alone ? fma(hi - lo, 1.0 / (1.0 - r), lo) : 0.5 * (lo + hi);
        if (alone && !isolated) {
            ilo = lo;
            ihi = hi;
            isolated = true;
        }
        const double d = hi - lo;
        if ((alone && (d <= 2e-13 || 0.25 * d * d <= 5e-17 * fmin(lam - ilo, ihi - lam))) || d <= 1e-16) break;
    }
    return lam;
}

template <int NQ>
struct VecShared {
    float ring[kRing<NQ>][kChunk][128 * NQ];       // reflectors on their way through
    double2 up[64 * NQ], down[64 * NQ];            // T as count_below takes it
    double d[128 * NQ];
    double2 fwd[128 * NQ], bwd[128 * NQ];          // (1 / e_k, -e_{k-1} / e_k) and (1 / e_{k-1}, -e_k / e_{k-1})
    double rec[kVecWarps][2][128 * NQ];            // the two recurrences of a warp's eigenvector
    int rex[kVecWarps][2][32 * NQ];                // their exponents
    float gram[32 * NQ][8];                        // inner products inside each group of four reflectors: 01 02 03 12 13 23
    float tau[128 * NQ];
    unsigned short perm[128 * NQ];
    int first[kPoints];
    double red[2][kEvWarps + kHelpWarps];
    double delta, mid[3];
};

// One warp per eigenvector, three per block, whatever n: no communication between blocks (each finds delta for itself). Bound by
// dependent latency: five or so passes of n / 2 fp64 steps over T, n steps of the recurrences, n / 4 groups of reflections.
template <int NQ>                                  // quads of positions per lane: N <= 128 NQ
__global__ void __launch_bounds__(kVecThreads, 1)
k_tridiag_vectors(const float* __restrict__ K, int ldk, TriWork wk, int G, int n, int do_shrink, int delta_rank, int keep, float* __restrict__ Ur, int ldu,
                  float* __restrict__ sigma_out, int n_sigma, EigInfo* __restrict__ info, float* __restrict__ Wsplit, int ldw, int j_pad) {
    constexpr int RING = kRing<NQ>;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int o = (G - n) & ~3, N = G - o, nch = (N + kChunk - 1) / kChunk;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    VecShared<NQ>& sh = *reinterpret_cast<VecShared<NQ>*>(smem_raw);

    // reflector k of this problem acts on positions > k; quads that end before those were never written
    auto live = [&](int k, int quad) { return k < N - 2 && 4 * quad < N && quad >= ((k + 1) >> 2); };
    auto fetch = [&](int ch) {                     // chunks count from the last reflectors
        if (ch < nch) {
            const int k0 = (nch - 1 - ch) * kChunk;
            float* dst = &sh.ring[ch % RING][0][0];
            for (int t = tid; t < kChunk * 32 * NQ; t += kVecThreads) {
                const int k = k0 + t / (32 * NQ), quad = t % (32 * NQ);
                const bool on = live(k, quad);
                const float* src = wk.V + (size_t)(o + (on ? k : 0)) * G + o + 4 * (on ? quad : 0);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s_addr(dst + 4 * (size_t)t)), "l"(src), "r"(on ? 16 : 0) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    chain_wait();
    for (int c = 0; c < RING; ++c) fetch(c);       // on their way while the eigenvalues are found

    const float dmax = *wk.dmax;
    // T is shifted and scaled so that every eigenvalue lies in (-1/2, 1/2): with eigenvalues that all agree in their leading
    // digits (orthonormal rows) the resolution is that of their differences. Positions past the n-th (zero, uncoupled) get a
    // diagonal below all others.
    const double big = 1e300;
    double gu = -big, gl = big;                    // where the eigenvalues are (Gershgorin)
    auto finite = [](float v) { return fabsf(v) <= 3.0e38f ? (double)v : 0.0; };
    for (int i = tid; i < n; i += kVecThreads) {
        const double el = i > 0 ? fabs(finite(wk.e[o + i - 1])) : 0.0, er = i < n - 1 ? fabs(finite(wk.e[o + i])) : 0.0, d = finite(wk.d[o + i]);
        gu = fmax(gu, d + (el + er));
        gl = fmin(gl, d - (el + er));
    }
    for (int i = tid; i < 128 * NQ; i += kVecThreads) {
        sh.tau[i] = i < N - 2 ? wk.tau[o + i] : 0.f;
        sh.perm[i] = (unsigned short)(i < n ? wk.perm[i] : i);
    }
#pragma unroll
    for (int x = 16; x > 0; x >>= 1) {
        gu = fmax(gu, __shfl_xor_sync(0xffffffffu, gu, x));
        gl = fmin(gl, __shfl_xor_sync(0xffffffffu, gl, x));
    }
    if (lane == 0) {
        sh.red[0][w] = gu;
        sh.red[1][w] = gl;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kEvWarps + kHelpWarps; ++j) {
        gu = fmax(gu, sh.red[0][j]);
        gl = fmin(gl, sh.red[1][j]);
    }
    const double gm = fmax(fabs(gu), fabs(gl));
    constexpr double kPert = 2.98e-8;              // below 2^-25, relative
    const double range = (gu - gl) + 4.0 * kPert * gm + 1e-30, low = gl - kPert * gm - range * (1.0 / 32.0);
    const double shift = (double)(float)(0.5 * (gu + low));
    const int gex = ((__double2hiint(range * 1.25 + fabs(gm) * 1e-7) >> 20) & 2047) - 1023 + 1;
    const double tsc = pow2(-gex), wid = pow2(gex);
    const int h = N >> 1, M = (h + 15) & ~15;      // rows 0 .. h - 1 from above, N - 1 .. h + 1 from below, h in the middle
    if (tid < M - h) sh.up[tid] = make_double2(1.0, 0.0);
    if (tid < M - h + 1) sh.down[tid] = make_double2(1.0, 0.0);
    for (int i = tid; i < N; i += kVecThreads) {
        // the perturbation of the diagonal, spread evenly by a multiplicative sequence
        const double psi = (double)(int)((unsigned)(i + 1) * 2654435769u) * (1.0 / 2147483648.0);
        const double di = i < n ? finite(wk.d[o + i]) : low;
        const double d = fma(i < n ? kPert * psi : 0.0, di, di - shift) * tsc;
        auto off = [&](int k) {                                            // couplings kept away from zero
            const double e = k < n - 1 ? finite(wk.e[o + k]) * tsc : 0.0;
            return fabs(e) < 1e-12 ? 1e-12 : e;
        };
        const double el = i > 0 ? off(i - 1) : 0.0, er = i < N - 1 ? off(i) : 0.0;
        const double il = i > 0 ? 1.0 / el : 0.0, ir = i < N - 1 ? 1.0 / er : 0.0;
        sh.d[i] = d;
        if (i < h) sh.up[M - h + i] = make_double2(d, -el * el);
        if (i > h) sh.down[M - 1 - (i - h - 1)] = make_double2(d, -er * er);
        if (i == h) {
            sh.mid[0] = d;
            sh.mid[1] = -el * el;
            sh.mid[2] = -er * er;
        }
        sh.fwd[i] = make_double2(ir, -el * ir);
        sh.bwd[i] = make_double2(il, -er * il);
    }
    __syncthreads();
    const bool empty = !(dmax > 0.f);
    const double cut = (kRankCut - shift) * tsc;
    const int j = blockIdx.x * kVecWarps + w;      // this warp's eigenvector (w == kVecWarps: delta)
    double det;
    int dex;
    if (w < kEvWarps)
        sh.first[tid] = count_below(sh.up, sh.down, sh.mid, M, fma((double)(tid + 1), 1.0 / (kPoints + 1), -0.5), det, dex);
    __syncthreads();

    const bool mine = w < kVecWarps && j < keep && j < n && !empty;
    double lam = 0.0;
    if (mine) lam = eigenvalue(sh.up, sh.down, sh.mid, M, N - 1 - j, sh.first, lane);
    if (w == kVecWarps) {
        double delta = 0.0;
        if (do_shrink && delta_rank - 1 < n && !empty) {
            delta = eigenvalue(sh.up, sh.down, sh.mid, M, N - delta_rank, sh.first, lane);
            delta = delta > cut ? fma(delta, wid, shift) : 0.0;
        }
        if (lane == 0) sh.delta = delta;
        if (blockIdx.x == 0) {
            const int rank = empty ? 0 : min(n, N - count_below(sh.up, sh.down, sh.mid, M, cut, det, dex));
            if (lane == 0) {
                const float df = (float)(delta * (double)dmax);
                info->delta = df;
                info->sweeps = 0;
                info->rank = rank;
                if (do_shrink) {
                    info->sum_delta += (double)df;
                    info->shrinks += 1;
                }
            }
            for (int t = keep + lane; t < n_sigma; t += 32) sigma_out[t] = 0.f;
        }
    }
    if (w >= kEvWarps) {                           // helpers: inner products inside each group of four reflectors
        for (int grp = w - kEvWarps; grp < nch * (kChunk / 4); grp += kHelpWarps) {
            float4 v[4][NQ];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const int k = 4 * grp + a, quad = lane + 32 * q;
                    v[a][q] = live(k, quad) ? *reinterpret_cast<const float4*>(wk.V + (size_t)(o + k) * G + o + 4 * quad) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            int t = 0;
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = a + 1; b < 4; ++b, ++t)
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        s[t] = fmaf(v[a][q].x, v[b][q].x, s[t]);
                        s[t] = fmaf(v[a][q].y, v[b][q].y, s[t]);
                        s[t] = fmaf(v[a][q].z, v[b][q].z, s[t]);
                        s[t] = fmaf(v[a][q].w, v[b][q].w, s[t]);
                    }
            const float r = lane_sums<8, 16>(s, lane);
            if ((lane & 3) == 0) sh.gram[grp][lane >> 2] = r;
        }
    }
    const bool alive = mine && lam > cut;
    float x[4 * NQ];
#pragma unroll
    for (int t = 0; t < 4 * NQ; ++t) x[t] = 0.f;
    if (alive) {
        // (T - lambda) v = 0 from both ends: lane 0 forwards, lane 1 backwards
        const double* F = sh.rec[w][0];
        const double* B = sh.rec[w][1];
        const int* FE = sh.rex[w][0];
        const int* BE = sh.rex[w][1];
        if (lane < 2) {
            const int dir = lane ? -1 : 1, k0 = lane ? N - 1 : 0;
            const double2* co = (lane ? sh.bwd : sh.fwd) + k0;
            const double* dd = sh.d + k0;
            double* out = sh.rec[w][lane] + k0;
            int* oex = sh.rex[w][lane] + (k0 >> 2);
            double f = 1.0, fm = 0.0;
            int ex = 0;
            double2 t[4];
            double a[4];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                t[s] = co[dir * s];
                a[s] = (lam - dd[dir * s]) * t[s].x;
            }
#pragma unroll 2
            for (int m = 0; m < N; m += 4) {
                double2 tn[4];
                double an[4];
                const int nx = m + 4 < N ? m + 4 : 0;                      // the next rows are on their way meanwhile
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    tn[s] = co[dir * (nx + s)];
                    an[s] = (lam - dd[dir * (nx + s)]) * tn[s].x;
                }
                if ((m & 4) == 0) {                                        // rescale at every second block of four positions
                    const int q = exponent_of(f, fm) - 1023;
                    const double sc = __hiloint2double((1023 - q) << 20, 0);
                    f *= sc;
                    fm *= sc;
                    ex += q;
                }
                oex[dir * (m >> 2)] = ex;
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    out[dir * (m + s)] = f;
                    const double fn = fma(a[s], f, t[s].y * fm);
                    fm = f;
                    f = fn;
                    t[s] = tn[s];
                    a[s] = an[s];
                }
            }
        }
        __syncwarp();
        // where the two meet: the largest product, compared through exponent and leading bits
        long long best = -(1ll << 62);
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int quad = lane + 32 * q;
            if (4 * quad < N) {
                const long long ee = ((long long)FE[quad] + BE[quad]) << 20;
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    const int k = 4 * quad + s;
                    const long long v = ee + (__double2hiint(F[k]) & 0x7fffffff) + (__double2hiint(B[k]) & 0x7fffffff);
                    const long long key = v * 512 + (511 - k);
                    if (key > best) best = key;
                }
            }
        }
#pragma unroll
        for (int y = 16; y > 0; y >>= 1) {
            const long long other = __shfl_xor_sync(0xffffffffu, best, y);
            if (other > best) best = other;
        }
        const int r = 511 - (int)(best & 511);
        const double invF = 1.0 / F[r], invB = 1.0 / B[r];
        const int exF = FE[r >> 2], exB = BE[r >> 2];
        double v[4 * NQ];
        double nrm = 0.0;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int quad = lane + 32 * q;
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const int k = 4 * quad + s;
                double t = 0.0;
                if (k < N) t = k <= r ? F[k] * invF * pow2(FE[quad] - exF) : B[k] * invB * pow2(BE[quad] - exB);
                v[4 * q + s] = t;
                nrm = fma(t, t, nrm);
            }
        }
#pragma unroll
        for (int y = 16; y > 0; y >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, y);
        const double inv = 1.0 / sqrt(nrm);
#pragma unroll
        for (int t = 0; t < 4 * NQ; ++t) x[t] = (float)(v[t] * inv);
    }

    chain_release();
    // ---- U = H_0 H_1 ... applied to the vectors, the last reflector first, four at a time: with c_i = v_i . x and the inner
    // products of the four among each other the four coefficients follow without another pass over x
    const bool resident = nch <= RING;
    if (resident) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
    }
    for (int ch = 0; ch < nch; ++ch) {
        if (!resident) {
            asm volatile("cp.async.wait_group %0;" ::"n"(RING - 1) : "memory");
            __syncthreads();                       // chunk ch has landed
        }
        if (alive) {
            const int k0 = (nch - 1 - ch) * kChunk;
#pragma unroll (NQ == 4 ? 1 : 4)
            for (int grp = kChunk / 4 - 1; grp >= 0; --grp) {
                const float* V = &sh.ring[ch % RING][4 * grp][0];
                float4 v[4][NQ];
                float c[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int q = 0; q < NQ; ++q) v[i][q] = *reinterpret_cast<const float4*>(V + i * 128 * NQ + 4 * (lane + 32 * q));
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    c[i] = 0.f;
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        c[i] = fmaf(v[i][q].x, x[4 * q], c[i]);
                        c[i] = fmaf(v[i][q].y, x[4 * q + 1], c[i]);
                        c[i] = fmaf(v[i][q].z, x[4 * q + 2], c[i]);
                        c[i] = fmaf(v[i][q].w, x[4 * q + 3], c[i]);
                    }
                }
#pragma unroll
                for (int y = 16; y > 0; y >>= 1) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) c[i] += __shfl_xor_sync(0xffffffffu, c[i], y);
                }
                const float4 g0 = *reinterpret_cast<const float4*>(&sh.gram[(k0 >> 2) + grp][0]);
                const float2 g1 = *reinterpret_cast<const float2*>(&sh.gram[(k0 >> 2) + grp][4]);
                const float4 tk = *reinterpret_cast<const float4*>(&sh.tau[k0 + 4 * grp]);
                const float a3 = tk.w * c[3];
                const float a2 = tk.z * fmaf(-g1.y, a3, c[2]);
                const float a1 = tk.y * fmaf(-g0.w, a2, fmaf(-g1.x, a3, c[1]));
                const float a0 = tk.x * fmaf(-g0.x, a1, fmaf(-g0.y, a2, fmaf(-g0.z, a3, c[0])));
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    x[4 * q] -= fmaf(a0, v[0][q].x, fmaf(a1, v[1][q].x, fmaf(a2, v[2][q].x, a3 * v[3][q].x)));
                    x[4 * q + 1] -= fmaf(a0, v[0][q].y, fmaf(a1, v[1][q].y, fmaf(a2, v[2][q].y, a3 * v[3][q].y)));
                    x[4 * q + 2] -= fmaf(a0, v[0][q].z, fmaf(a1, v[1][q].z, fmaf(a2, v[2][q].z, a3 * v[3][q].z)));
                    x[4 * q + 3] -= fmaf(a0, v[0][q].w, fmaf(a1, v[1][q].w, fmaf(a2, v[2][q].w, a3 * v[3][q].w)));
                }
            }
        }
        if (!resident) {
            __syncthreads();                       // chunk ch has been used
            fetch(ch + RING);
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");

    // ---- factors ----
    if (w < kVecWarps && j < (Wsplit && j_pad > keep ? j_pad : keep)) {
        float* px = reinterpret_cast<float*>(sh.rec[w][0]);                 // from the order of the reduction to that of K
#pragma unroll
        for (int q = 0; q < NQ; ++q)
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const int i = 4 * (lane + 32 * q) + s;
                px[sh.perm[i]] = i < n ? x[4 * q + s] : 0.f;
            }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const float4 t = *reinterpret_cast<const float4*>(px + 4 * (lane + 32 * q));
            x[4 * q] = t.x;
            x[4 * q + 1] = t.y;
            x[4 * q + 2] = t.z;
            x[4 * q + 3] = t.w;
        }
        float fac = 0.f, sp = 0.f;
        if (alive) {
            const double l = fma(lam, wid, shift), kept = l - sh.delta;
            if (kept > 0.0) {
                fac = (float)sqrt(kept / l);
                sp = (float)sqrt(kept * (double)dmax);
            }
            if (!do_shrink) {
                // a freeze that keeps the eigenvalues as they are: x^T K x in fp64, off by the square of the vector's error only
                double dot = 0.0, nn = 0.0;
#pragma unroll
                for (int t = 0; t < 4 * NQ; ++t) nn = fma((double)x[t], (double)x[t], nn);
#pragma unroll 4
                for (int i = 0; i < n; ++i) {
                    const float xi = px[i];
                    double y = 0.0;
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        const int c = 4 * (lane + 32 * q);
                        if (c >= n) continue;
                        const float4 k = *reinterpret_cast<const float4*>(K + (size_t)i * ldk + c);
                        // rows that take no part are zero in x and may be anything in K
                        y = fma(x[4 * q] != 0.f ? (double)k.x : 0.0, (double)x[4 * q], y);
                        y = fma(x[4 * q + 1] != 0.f ? (double)k.y : 0.0, (double)x[4 * q + 1], y);
                        y = fma(x[4 * q + 2] != 0.f ? (double)k.z : 0.0, (double)x[4 * q + 2], y);
                        y = fma(x[4 * q + 3] != 0.f ? (double)k.w : 0.0, (double)x[4 * q + 3], y);
                    }
                    if (xi != 0.f) dot = fma(y, (double)xi, dot);
                }
#pragma unroll
                for (int y = 16; y > 0; y >>= 1) {
                    dot += __shfl_xor_sync(0xffffffffu, dot, y);
                    nn += __shfl_xor_sync(0xffffffffu, nn, y);
                }
                if (dot > 0.0) sp = (float)sqrt(dot / nn);
            }
        }
        if (j < n_sigma && j < keep && lane == 0) sigma_out[j] = sp;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const int i = 4 * (lane + 32 * q) + s;
                if (j < keep && i < n) Ur[(size_t)i * ldu + j] = x[4 * q + s] * fac;
            }
        }
        if (Wsplit && j < j_pad) {                 // transposed and split for the tensor-core rebuild, zero padded
            float* hi_row = Wsplit + split_row(j, j_pad, false) * ldw;
            float* lo_row = Wsplit + split_row(j, j_pad, true) * ldw;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int i = 4 * (lane + 32 * q);
                if (i < ldw) {
                    float h4[4], l4[4];
#pragma unroll
                    for (int s = 0; s < 4; ++s) {
                        const float v = i + s < n ? x[4 * q + s] * fac : 0.f;
                        h4[s] = __uint_as_float((__float_as_uint(v) + 0x1000u) & 0xffffe000u);
                        l4[s] = v - h4[s];
                    }
                    *reinterpret_cast<float4*>(hi_row + i) = make_float4(h4[0], h4[1], h4[2], h4[3]);
                    *reinterpret_cast<float4*>(lo_row + i) = make_float4(l4[0], l4[1], l4[2], l4[3]);
                }
            }
            for (int i = 128 * NQ + lane; i < ldw; i += 32) hi_row[i] = lo_row[i] = 0.f;
        }
    }
}

// A matrix as it comes: one block, or a cluster where the shape says so.
template <typename S>
cudaError_t run_tridiag(const float* K, int ldk, int n, TriWork wk, EigInfo* info, cudaStream_t st) {
    const int n4 = (n + 3) & ~3;
    constexpr int most = (S::CL == 1 ? S::G : kOwnRows<S>) * (S::G + 4) * 4;
    const int smem = (S::CL == 1 ? n : kOwnRows<S>) * (n4 + 4) * 4;
    cudaError_t e = allow_smem((const void*)k_tridiag<S>, most);
    if (e != cudaSuccess) return e;
    return launch(k_tridiag<S>, LaunchShape{dim3(S::CL), dim3(S::NT), (size_t)smem, (unsigned)S::CL}, st, K, ldk, n, 0, wk, 0, (int)S::G, info);
}

template <int NQ>
cudaError_t run_vectors(const float* K, int ldk, TriWork wk, int G, int n, int do_shrink, int delta_rank, int keep, float* Ur, int ldu, float* sigma_out, int n_sigma,
                        EigInfo* info, float* Wsplit, int ldw, int j_pad, cudaStream_t st) {
    const int rows = Wsplit && j_pad > keep ? j_pad : keep;
    const int blocks = rows > 0 ? (rows + kVecWarps - 1) / kVecWarps : 1;
    cudaError_t e = allow_smem((const void*)k_tridiag_vectors<NQ>, (int)sizeof(VecShared<NQ>));
    if (e != cudaSuccess) return e;
    return launch_chained(k_tridiag_vectors<NQ>, dim3(blocks), dim3(kVecThreads), sizeof(VecShared<NQ>), st, K, ldk, wk, G, n, do_shrink, delta_rank, keep, Ur, ldu,
                          sigma_out, n_sigma, info, Wsplit, ldw, j_pad);
}

}  // namespace

size_t eig_work_floats(int n) {
    const size_t G = n <= 128 ? 128 : n <= 256 ? 256 : 512;
    const size_t direct = G * G + 4 * G + 128 * 128 + 16, iterative = (n > 256 ? (size_t)512 * 512 : (size_t)256 * 256) + 64;
    return direct > iterative ? direct : iterative;
}

int eig_launches(int n, int variant) { return variant != 0 ? 1 : n <= 128 ? 2 : 3; }

cudaError_t launch_eig_direct(const float* K, int ldk, int n, int do_shrink, int delta_rank, int keep, float* Ur, int ldu, float* sigma_out,
                              int n_sigma, float* work, EigInfo* info, float* Wsplit, int ldw, int j_pad, cudaStream_t st) {
    if (n <= 0 || n > 512 || (ldk & 3) != 0) return cudaErrorInvalidValue;
    const int G = n <= 128 ? 128 : n <= 256 ? 256 : 512;
    const TriWork wk = tri_work(work, G);
    cudaError_t e = cudaSuccess;
    if (G == 128) {
        e = run_tridiag<Tri128>(K, ldk, n, wk, info, st);
    } else {
        e = G == 256 ? run_tridiag<Tri256>(K, ldk, n, wk, info, st) : run_tridiag<Tri512>(K, ldk, n, wk, info, st);
        if (e != cudaSuccess) return e;
        e = launch_chained(k_tridiag<Tri128>, dim3(1), dim3(Tri128::NT), 0, st, wk.trail, 128, 128, 1, wk, G - 128, G, info);
    }
    if (e != cudaSuccess) return e;
    if (G == 128) return run_vectors<1>(K, ldk, wk, G, n, do_shrink, delta_rank, keep, Ur, ldu, sigma_out, n_sigma, info, Wsplit, ldw, j_pad, st);
    if (G == 256) return run_vectors<2>(K, ldk, wk, G, n, do_shrink, delta_rank, keep, Ur, ldu, sigma_out, n_sigma, info, Wsplit, ldw, j_pad, st);
    return run_vectors<4>(K, ldk, wk, G, n, do_shrink, delta_rank, keep, Ur, ldu, sigma_out, n_sigma, info, Wsplit, ldw, j_pad, st);
}

}  // namespace sage
