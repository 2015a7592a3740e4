// The iterative eigen-solve (option 5 = 1; the direct one in eig_tridiag.cu is the default): eigen-decomposition of the
// buffer's Gram matrix and the Frequent-Directions shrink factors (Method, first paragraph). With K = B B^T = U Sigma^2 U^T
// the left factor U and sigma^2 come from the symmetric eigen-problem of K, and Sigma' V^T = diag(sigma'/sigma) U^T B.
//
// Method: implicit (one-sided) cyclic Jacobi on a Cholesky factor. K is factored with diagonal pivoting,
// P^T K P = L L^T (stopping at the numerical rank), then plane rotations are applied to column pairs of L from the
// right until all columns are mutually orthogonal: L V = U Sigma. The columns of the result are sigma_j u_j, so U
// needs no separate accumulation. Two kernel families: one thread block with the factor in shared memory (buffers of up to
// 192 rows), a cluster of 8 thread blocks with the factor in L2. All loops and waits are bounded; hitting the sweep limit
// sets a flag instead of spinning.
#include <cooperative_groups.h>

#include "sage_internal.h"

namespace sage {
namespace {

namespace cg = cooperative_groups;

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;

struct ArgMax {
    float v;
    int i;
};

__device__ __forceinline__ ArgMax better(ArgMax a, ArgMax b) {
    // larger value wins; ties (and NaN on the right) keep the smaller index
    if (b.v > a.v || (b.v == a.v && b.i < a.i)) return b;
    return a;
}

// Round-robin pairing: n_even players, rounds 0..n_even-2, slots 0..n_even/2-1 give disjoint pairs.
__device__ __forceinline__ void rr_pair(int n_even, int round, int slot, int& p, int& q) {
    const int nm1 = n_even - 1;
    int a, b;
    if (slot == 0) {
        a = nm1;
        b = round % nm1;
    } else {
        a = (round + slot) % nm1;
        b = (round + nm1 - slot) % nm1;
    }
    p = min(a, b);
    q = max(a, b);
}

// Rotation that orthogonalises two columns with squared norms a, b and inner product g:
// tan 2theta = 2g / (b - a), cos 2theta = |b - a| / r, c = sqrt((1 + cos 2theta) / 2), s = sin 2theta / (2c), from two
// approximate reciprocal square roots, followed by one Newton step towards c^2 + s^2 = 1 taken from the residual
// itself: scaling by 1.5 - 0.5 (c^2 + s^2) would be lost to the coarser float grid above 1 whenever c^2 + s^2 < 1,
// a one-sided correction that shrinks every column a little at every rotation (measured 1e-5 relative on the
// singular values after a few thousand rotations; with the residual form they agree with fp64 to 1e-7).
__device__ __forceinline__ void jacobi_rotation(float a, float b, float g, float& c, float& s) {
    const float tau = b - a, gam = 2.f * g;
    const float inv_r = rsqrtf(fmaf(tau, tau, gam * gam));
    const float c2 = fmaf(0.5f * fabsf(tau), inv_r, 0.5f);
    const float invc = rsqrtf(c2);
    c = c2 * invc;
    s = copysignf(0.5f, tau) * gam * inv_r * invc;
    const float half_res = 0.5f * fmaf(-s, s, fmaf(-c, c, 1.f));
    c = fmaf(c, half_res, c);
    s = fmaf(s, half_res, s);
}

// ------------------------------------------------------------------------------------------------
// Shared-memory solver for n <= 192 (the common case: n = 2*ell <= 128, and partly filled buffers at
// the freeze). Same mathematics as k_eig_shrink below, restructured for instruction count and latency:
//   * K is scaled by 1/max(diag) on load, so every intermediate is O(1) and fast reciprocal / rsqrt
//     intrinsics are safe; eigenvalues are scaled back at the end;
//   * Cholesky with diagonal pivoting but WITHOUT data movement: the pivot column stays where it is and
//     a per-index pivot order replaces the row/column swaps; every warp keeps the running diagonal in
//     registers and finds the pivot redundantly with one warp-wide integer max, so a step costs one
//     block barrier;
//   * one-sided Jacobi with one pair per QUARTER-warp: 8 lanes hold both columns in registers (float4
//     accesses, conflict-free), reduce the three dot products with 3 shuffle steps and rotate; warps
//     without a pair only take part in the barrier;
//   * a sweep whose largest pre-rotation cosine is below 1e-3 ends the iteration (the next sweep
//     would find cosines near 1e-6, the rotation threshold).
// X is column-major with a row pitch of LD = 64*T floats; column c of the factor stays at the physical
// position of the c-th pivot, so the rows of U come out in the original buffer order.
// ------------------------------------------------------------------------------------------------
constexpr int kMaxFast = 192;      // largest n whose matrix fits in shared memory
constexpr int kMaxN = 256;         // largest n of this kernel (above kMaxFast the matrix stays in global memory, i.e. L2)

template <int T, int NT, bool G>
__global__ void __launch_bounds__(NT, 1)
k_eig_shrink_fast(const float* __restrict__ K, int ldk, int n, int do_shrink, int delta_rank, int keep, float* __restrict__ Ur,
                  int ldu, float* __restrict__ sigma_out, int n_sigma, int max_sweeps, EigInfo* __restrict__ info,
                  float* __restrict__ Wsplit, int ldw, int j_pad, float* __restrict__ gwork) {
    constexpr int LD = 64 * T;
    constexpr int NW = NT / 32;
    constexpr int R = 2 * T;            // rows per lane when 32 lanes span a column
    constexpr int Q = 2 * T;            // float4 per lane when 8 lanes span a column
    extern __shared__ __align__(16) float smem[];
    float* X = G ? gwork : smem;                        // LD x LD (global scratch when it does not fit on chip)
    float* lam = G ? smem : smem + LD * LD;             // kMaxN each from here on
    float* fac = lam + kMaxN;
    float* scl = fac + kMaxN;
    int* ord = reinterpret_cast<int*>(scl + kMaxN);     // physical index -> pivot step (-1: never pivoted)
    int* perm = ord + kMaxN;                            // pivot step -> physical index
    int* order = perm + kMaxN;                          // sorted position -> pivot step
    float* sh_f = reinterpret_cast<float*>(order + kMaxN);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // running diagonal and liveness of the rows this lane owns (rows lane + 32 t), one copy per warp
    float dg[R];
    bool alive[R];
    bool bad = false;
    float dmax = 0.f;
#pragma unroll
    for (int t = 0; t < R; ++t) {
        const int i = lane + 32 * t;
        dg[t] = (i < n) ? K[(size_t)i * ldk + i] : -1.f;
        alive[t] = i < n;
        if (alive[t] && !(fabsf(dg[t]) <= 3.0e38f)) { bad = true; alive[t] = false; }
        if (alive[t]) dmax = fmaxf(dmax, dg[t]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    if (warp == 0 && bad) atomicOr(&info->flags, kFlagNonFinite);
    const bool empty = !(dmax >= 1e-30f);              // nothing to factor: rank 0
    const float kscale = empty ? 0.f : 1.f / dmax;
    for (int e = tid; e < n * LD; e += NT) {
        const int c = e / LD, i = e - c * LD;
        X[e] = (i < n) ? K[(size_t)c * ldk + i] * kscale : 0.f;  // K is symmetric: row c serves as column c
    }
#pragma unroll
    for (int t = 0; t < R; ++t) dg[t] *= kscale;
    for (int i = tid; i < kMaxN; i += NT) ord[i] = -1;
    __syncthreads();

    // ---- pivoted Cholesky without swaps (scaled matrix: diagonal <= 1) ----
    constexpr int CW = (LD + NW - 1) / NW;                     // columns a warp owns: warp + NW u
    unsigned colmask = 0u;                                     // bit u: column warp + 32 u is still unpivoted
#pragma unroll
    for (int u = 0; u < CW; ++u)
        if (warp + NW * u < n) colmask |= 1u << u;
    const float tol = 1e-7f;
    int rank = empty ? 0 : n;
    for (int k = 0; k < rank; ++k) {
        unsigned key = 0u;
#pragma unroll
        for (int t = 0; t < R; ++t)
            if (alive[t]) key = max(key, (__float_as_uint(fmaxf(dg[t], 0.f)) & 0xffffff00u) | (unsigned)(255 - (lane + 32 * t)));
        key = __reduce_max_sync(0xffffffffu, key);                // largest diagonal (24 significant bits), smaller index on ties
        const int p = 255 - (int)(key & 255u);
        if (key == 0u || p >= n) { rank = k; break; }             // identical in every warp
        const float* Xp = X + p * LD;
        const float d = Xp[p];
        if (!(d > tol)) { rank = k; break; }
        const float inv = rsqrtf(d);
        if ((p & (NW - 1)) == warp) colmask &= ~(1u << (p / NW));
        float li[R];
#pragma unroll
        for (int t = 0; t < R; ++t) {
            const int i = lane + 32 * t;
            if (i == p) alive[t] = false;
            li[t] = alive[t] ? Xp[i] * inv : 0.f;
            dg[t] = fmaf(-li[t], li[t], dg[t]);
        }
#pragma unroll
        for (int u0 = 0; u0 < CW; u0 += 2) {                      // two columns at a time: loads first, then stores
            const bool on0 = (colmask >> u0) & 1u, on1 = (u0 + 1 < CW) && ((colmask >> (u0 + 1)) & 1u);
            if (!on0 && !on1) continue;
            float* c0 = X + (warp + NW * u0) * LD;
            float* c1 = X + (warp + NW * (u0 + 1)) * LD;
            const float l0 = on0 ? Xp[warp + NW * u0] * inv : 0.f;
            const float l1 = on1 ? Xp[warp + NW * (u0 + 1)] * inv : 0.f;
            float v0[R], v1[R];
#pragma unroll
            for (int t = 0; t < R; ++t) {
                v0[t] = on0 ? c0[lane + 32 * t] : 0.f;
                v1[t] = on1 ? c1[lane + 32 * t] : 0.f;
            }
#pragma unroll
            for (int t = 0; t < R; ++t) {
                if (on0) c0[lane + 32 * t] = fmaf(-li[t], l0, v0[t]);
                if (on1) c1[lane + 32 * t] = fmaf(-li[t], l1, v1[t]);
            }
        }
        if (tid == 0) { ord[p] = k; perm[k] = p; scl[k] = inv; }
        __syncthreads();
    }
    __syncthreads();
    // ---- scale the pivot columns into the factor L (zero above the pivot order, zero unpivoted columns) ----
    for (int e = tid; e < n * LD; e += NT) {
        const int c = e / LD, i = e - c * LD;
        const int kc = ord[c];
        float v = 0.f;
        if (kc >= 0 && i < n) {
            const int ki = ord[i];
            if (!(ki >= 0 && ki < kc)) v = X[e] * scl[kc];
        }
        X[e] = v;
    }
    __syncthreads();

    // ---- one-sided cyclic Jacobi on the rank pivot columns ----
    // Columns (in pivot order) form blocks of 4. A block round pairs the blocks round-robin, one block
    // pair per warp; the warp rotates the 16 cross pairs of its two blocks in 4 local rounds (one pair per
    // quarter-warp, synchronised inside the warp only), and in the first block round of a sweep also the
    // pairs inside each block. Only the warps that own a block pair take part, on a named barrier.
    const int l8 = tid & 7, qd = lane >> 3;
    int sweeps = 0;
    float worst2 = 0.f;                 // largest squared cosine met in the current sweep
    int* sh_flag = reinterpret_cast<int*>(sh_f + 2);
    if (tid < 2) sh_flag[tid] = 0;
    __syncthreads();
    if (rank >= 2) {
        const int nb = (rank + 3) >> 2, nbe = nb + (nb & 1), nbm1 = nbe - 1, nact = nbe >> 1;   // block pairs per round
        const int nwork = nact < NW ? nact : NW;                  // warps that take part; each owns slots w, w + nwork, ...
        if (warp < nwork) {
            const int nthreads = nwork * 32;
            auto pair_step = [&](int p, int q) {                  // p, q: pivot-order columns, q >= rank means no pair
                const bool valid = p < rank && q < rank;
                float4* xp = reinterpret_cast<float4*>(X + (valid ? perm[p] : 0) * LD) + l8;
                float4* xq = reinterpret_cast<float4*>(X + (valid ? perm[q] : 0) * LD) + l8;
                float4 x[Q], y[Q];
                float a0 = 0.f, a1 = 0.f, b0 = 0.f, b1 = 0.f, g0 = 0.f, g1 = 0.f;
#pragma unroll
                for (int t = 0; t < Q; ++t) {
                    x[t] = xp[8 * t];
                    y[t] = xq[8 * t];
                    a0 = fmaf(x[t].x, x[t].x, a0); a1 = fmaf(x[t].y, x[t].y, a1); a0 = fmaf(x[t].z, x[t].z, a0); a1 = fmaf(x[t].w, x[t].w, a1);
                    b0 = fmaf(y[t].x, y[t].x, b0); b1 = fmaf(y[t].y, y[t].y, b1); b0 = fmaf(y[t].z, y[t].z, b0); b1 = fmaf(y[t].w, y[t].w, b1);
                    g0 = fmaf(x[t].x, y[t].x, g0); g1 = fmaf(x[t].y, y[t].y, g1); g0 = fmaf(x[t].z, y[t].z, g0); g1 = fmaf(x[t].w, y[t].w, g1);
                }
                float a = a0 + a1, b = b0 + b1, g = g0 + g1;
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) {
                    a += __shfl_xor_sync(0xffffffffu, a, o);
                    b += __shfl_xor_sync(0xffffffffu, b, o);
                    g += __shfl_xor_sync(0xffffffffu, g, o);
                }
                const float ab = a * b, g2 = g * g;
                if (valid && ab > 0.f && g2 > 1e-12f * ab) {
                    worst2 = fmaxf(worst2, __fdividef(g2, ab));
                    float c, s;
                    jacobi_rotation(a, b, g, c, s);
#pragma unroll
                    for (int t = 0; t < Q; ++t) {
                        float4 nx, ny;
                        nx.x = fmaf(-s, y[t].x, c * x[t].x); ny.x = fmaf(s, x[t].x, c * y[t].x);
                        nx.y = fmaf(-s, y[t].y, c * x[t].y); ny.y = fmaf(s, x[t].y, c * y[t].y);
                        nx.z = fmaf(-s, y[t].z, c * x[t].z); ny.z = fmaf(s, x[t].z, c * y[t].z);
                        nx.w = fmaf(-s, y[t].w, c * x[t].w); ny.w = fmaf(s, x[t].w, c * y[t].w);
                        xp[8 * t] = nx;
                        xq[8 * t] = ny;
                    }
                }
                __syncwarp();
            };
            int more = 0;
            while (sweeps < max_sweeps) {
                worst2 = 0.f;
                for (int br = 0; br < nbm1; ++br) {
                  for (int slot = warp; slot < nact; slot += nwork) {
                    int ba, bb;                                   // the two blocks of this slot in this block round
                    if (slot == 0) { ba = nbm1; bb = br; }
                    else {
                        ba = br + slot; if (ba >= nbm1) ba -= nbm1;
                        bb = br + nbm1 - slot; if (bb >= nbm1) bb -= nbm1;
                    }
                    if (br == 0) {                                // pairs inside each block: quarters 0,1 -> ba, 2,3 -> bb
                        const int base = 4 * ((qd < 2) ? ba : bb), h = qd & 1;
                        pair_step(base + (h ? 2 : 0), base + (h ? 3 : 1));
                        pair_step(base + (h ? 1 : 0), base + (h ? 3 : 2));
                        pair_step(base + (h ? 1 : 0), base + (h ? 2 : 3));
                    }
                    const int lo = min(ba, bb), hi = max(ba, bb);
                    {   // the 16 cross pairs, columns held in registers: quarter qd keeps column qd of block lo and
                        // the columns of block hi travel from quarter to quarter by shuffles between the 4 rounds
                        const int pa = 4 * lo + qd, pb = 4 * hi + qd;
                        const bool va = pa < rank, vb0 = pb < rank;
                        float4* xa = reinterpret_cast<float4*>(X + (va ? perm[pa] : 0) * LD) + l8;
                        float4* xb = reinterpret_cast<float4*>(X + (vb0 ? perm[pb] : 0) * LD) + l8;
                        float4 x[Q], y[Q];
#pragma unroll
                        for (int t = 0; t < Q; ++t) {
                            x[t] = va ? xa[8 * t] : make_float4(0.f, 0.f, 0.f, 0.f);
                            y[t] = vb0 ? xb[8 * t] : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const bool valid = va && (4 * hi + ((qd + r) & 3) < rank);
                            float a0 = 0.f, a1 = 0.f, b0 = 0.f, b1 = 0.f, g0 = 0.f, g1 = 0.f;
#pragma unroll
                            for (int t = 0; t < Q; ++t) {
                                a0 = fmaf(x[t].x, x[t].x, a0); a1 = fmaf(x[t].y, x[t].y, a1); a0 = fmaf(x[t].z, x[t].z, a0); a1 = fmaf(x[t].w, x[t].w, a1);
                                b0 = fmaf(y[t].x, y[t].x, b0); b1 = fmaf(y[t].y, y[t].y, b1); b0 = fmaf(y[t].z, y[t].z, b0); b1 = fmaf(y[t].w, y[t].w, b1);
                                g0 = fmaf(x[t].x, y[t].x, g0); g1 = fmaf(x[t].y, y[t].y, g1); g0 = fmaf(x[t].z, y[t].z, g0); g1 = fmaf(x[t].w, y[t].w, g1);
                            }
                            float a = a0 + a1, b = b0 + b1, g = g0 + g1;
#pragma unroll
                            for (int o = 4; o > 0; o >>= 1) {
                                a += __shfl_xor_sync(0xffffffffu, a, o);
                                b += __shfl_xor_sync(0xffffffffu, b, o);
                                g += __shfl_xor_sync(0xffffffffu, g, o);
                            }
                            const float ab = a * b, g2 = g * g;
                            if (valid && ab > 0.f && g2 > 1e-12f * ab) {
                                worst2 = fmaxf(worst2, __fdividef(g2, ab));
                                float c, s;
                                jacobi_rotation(a, b, g, c, s);
#pragma unroll
                                for (int t = 0; t < Q; ++t) {
                                    float4 nx, ny;
                                    nx.x = fmaf(-s, y[t].x, c * x[t].x); ny.x = fmaf(s, x[t].x, c * y[t].x);
                                    nx.y = fmaf(-s, y[t].y, c * x[t].y); ny.y = fmaf(s, x[t].y, c * y[t].y);
                                    nx.z = fmaf(-s, y[t].z, c * x[t].z); ny.z = fmaf(s, x[t].z, c * y[t].z);
                                    nx.w = fmaf(-s, y[t].w, c * x[t].w); ny.w = fmaf(s, x[t].w, c * y[t].w);
                                    x[t] = nx;
                                    y[t] = ny;
                                }
                            }
                            if (r < 3) {                          // quarter qd takes over the column quarter qd + 1 holds
                                const int src = (lane + 8) & 31;
#pragma unroll
                                for (int t = 0; t < Q; ++t) {
                                    y[t].x = __shfl_sync(0xffffffffu, y[t].x, src);
                                    y[t].y = __shfl_sync(0xffffffffu, y[t].y, src);
                                    y[t].z = __shfl_sync(0xffffffffu, y[t].z, src);
                                    y[t].w = __shfl_sync(0xffffffffu, y[t].w, src);
                                }
                            }
                        }
                        const int pl = 4 * hi + ((qd + 3) & 3);   // the hi column this quarter ends up with
                        if (va) {
#pragma unroll
                            for (int t = 0; t < Q; ++t) xa[8 * t] = x[t];
                        }
                        if (pl < rank) {
                            float4* xl = reinterpret_cast<float4*>(X + perm[pl] * LD) + l8;
#pragma unroll
                            for (int t = 0; t < Q; ++t) xl[8 * t] = y[t];
                        }
                        __syncwarp();
                    }
                  }
                    asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
                }
                ++sweeps;
                const int par = sweeps & 1;
                if (__any_sync(0xffffffffu, worst2 > 1e-6f) && lane == 0) atomicOr(&sh_flag[par], 1);
                if (tid == 0) sh_flag[par ^ 1] = 0;
                asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
                more = sh_flag[par];
                if (!more) break;               // every cosine of this sweep was below 1e-3: converged after it
            }
            if (tid == 0) { sh_f[1] = (float)sweeps; sh_f[4] = more ? 1.f : 0.f; }
        }
    }
    __syncthreads();
    sweeps = rank >= 2 ? (int)sh_f[1] : 0;
    const int not_converged = rank >= 2 && sh_f[4] != 0.f;     // stopped at the sweep limit while still rotating visibly

    // ---- eigenvalues = squared column norms (pivot-step order), scaled back; sort descending, stable ----
    for (int k = warp; k < n; k += NW) {
        float a = 0.f;
        if (k < rank) {
            const float* x = X + perm[k] * LD;
#pragma unroll
            for (int t = 0; t < R; ++t) a = fmaf(x[lane + 32 * t], x[lane + 32 * t], a);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        }
        if (lane == 0) lam[k] = a * dmax;
    }
    __syncthreads();
    if (tid < n) {
        const float mine = lam[tid];
        int pos = 0;
        for (int i = 0; i < n; ++i) {
            const float o = lam[i];
            pos += (o > mine) || (o == mine && i < tid);
        }
        order[pos] = tid;
    }
    __syncthreads();
    if (tid == 0) {
        float delta = 0.f;
        if (do_shrink && delta_rank - 1 < n) delta = lam[order[delta_rank - 1]];
        sh_f[0] = delta;
        info->delta = delta;
        info->sweeps = sweeps;
        if (sweeps > info->max_sweeps) info->max_sweeps = sweeps;
        info->rank = rank;
        if (not_converged) info->flags |= kFlagNotConverged;
        if (do_shrink) {
            info->sum_delta += (double)delta;
            info->shrinks += 1;
        }
    }
    __syncthreads();
    const float delta = sh_f[0];
    const float back = sqrtf(dmax);     // columns of X are sigma_j u_j / sqrt(dmax)
    if (tid < n) {
        const float l = lam[order[tid]];
        float f = 0.f, sp = 0.f;
        if (l > 0.f && tid < keep) {
            const float kept = fmaxf(l - delta, 0.f);
            sp = sqrtf(kept);
            f = sqrtf(kept / l) * rsqrtf(l) * back;   // (sigma'/sigma) / sigma, for the unscaled column
        }
        fac[tid] = f;
        if (tid < n_sigma) sigma_out[tid] = sp;
    }
    for (int j = n + tid; j < n_sigma; j += NT) sigma_out[j] = 0.f;
    __syncthreads();
    for (int e = tid; e < n * keep; e += NT) {
        const int j = e / n, i = e - j * n;
        float v = 0.f;
        if (j < n) {
            const int k = order[j];
            if (k < rank) v = X[perm[k] * LD + i] * fac[j];
        }
        Ur[(size_t)i * ldu + j] = v;
    }
    if (Wsplit) {   // the same factors transposed and split for the tensor-core rebuild: [W_hi ; W_lo], zero padded
        for (int e = tid; e < j_pad * ldw; e += NT) {
            const int j = e / ldw, i = e - j * ldw;
            float v = 0.f;
            if (j < keep && j < n && i < n) {
                const int k = order[j];
                if (k < rank) v = X[perm[k] * LD + i] * fac[j];
            }
            const float hi = __uint_as_float((__float_as_uint(v) + 0x1000u) & 0xffffe000u);
            Wsplit[split_row(j, j_pad, false) * ldw + i] = hi;
            Wsplit[split_row(j, j_pad, true) * ldw + i] = v - hi;
        }
    }
}

// ------------------------------------------------------------------------------------------------
// Cluster solver for 192 < n <= 512: the same algorithm as k_eig_shrink_fast, run by a thread-block cluster
// (8 CTAs of 256 threads on 8 SMs) with the matrix in global memory (L2-resident) and a hardware cluster
// barrier where the one-CTA kernel has a block barrier. Every warp of the cluster owns Cholesky columns and one
// Jacobi block pair, so a block round costs one L2 round trip for its 8 columns, 4 register-resident local rounds
// and one cluster barrier, instead of several passes over 16 warps on one SM. Control flow is identical in
// every CTA (pivot search and convergence flag are computed from identical data), so every thread of the cluster
// reaches every barrier; the small tables (pivot order, eigenvalues, factors) are kept per CTA.
// ------------------------------------------------------------------------------------------------
template <int T>
__global__ void __launch_bounds__(256, 1)
k_eig_shrink_cluster(const float* __restrict__ K, int ldk, int n, int do_shrink, int delta_rank, int keep, float* __restrict__ Ur,
                  int ldu, float* __restrict__ sigma_out, int n_sigma, int max_sweeps, EigInfo* __restrict__ info,
                  float* __restrict__ Wsplit, int ldw, int j_pad, float* __restrict__ gwork) {
    constexpr int LD = 64 * T;
    constexpr int NT = 256;                              // threads per CTA
    constexpr int kMaxN = 512;                           // shadows the namespace constant: this kernel serves n <= 512
    cg::cluster_group cluster = cg::this_cluster();
    const int csize = (int)cluster.num_blocks(), crank = (int)cluster.block_rank();
    const int NW = 8 * csize;                            // warps of the whole cluster
    const int GT = NT * csize;                           // threads of the whole cluster
    constexpr int R = 2 * T;            // rows per lane when 32 lanes span a column
    constexpr int Q = 2 * T;            // float4 per lane when 8 lanes span a column
    extern __shared__ __align__(16) float smem[];
    float* X = gwork;                                   // LD x LD in global memory (L2), shared by the cluster
    int* gflag = reinterpret_cast<int*>(gwork + (size_t)LD * LD);   // two convergence words after the matrix
    float* lam = smem;                                  // kMaxN each from here on (one copy per CTA)
    float* fac = lam + kMaxN;
    float* scl = fac + kMaxN;
    int* ord = reinterpret_cast<int*>(scl + kMaxN);     // physical index -> pivot step (-1: never pivoted)
    int* perm = ord + kMaxN;                            // pivot step -> physical index
    int* order = perm + kMaxN;                          // sorted position -> pivot step
    float* sh_f = reinterpret_cast<float*>(order + kMaxN);

    const int tid = threadIdx.x, lane = tid & 31, lwarp = tid >> 5;
    const int warp = crank * 8 + lwarp;                  // warp index within the cluster
    const int gtid = crank * NT + tid;

    // running diagonal and liveness of the rows this lane owns (rows lane + 32 t), one copy per warp
    float dg[R];
    bool alive[R];
    bool bad = false;
    float dmax = 0.f;
#pragma unroll
    for (int t = 0; t < R; ++t) {
        const int i = lane + 32 * t;
        dg[t] = (i < n) ? K[(size_t)i * ldk + i] : -1.f;
        alive[t] = i < n;
        if (alive[t] && !(fabsf(dg[t]) <= 3.0e38f)) { bad = true; alive[t] = false; }
        if (alive[t]) dmax = fmaxf(dmax, dg[t]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    if (warp == 0 && bad) atomicOr(&info->flags, kFlagNonFinite);
    const bool empty = !(dmax >= 1e-30f);              // nothing to factor: rank 0
    const float kscale = empty ? 0.f : 1.f / dmax;
    for (int e = gtid; e < n * LD; e += GT) {
        const int c = e / LD, i = e - c * LD;
        X[e] = (i < n) ? K[(size_t)c * ldk + i] * kscale : 0.f;  // K is symmetric: row c serves as column c
    }
    if (gtid < 2) gflag[gtid] = 0;
#pragma unroll
    for (int t = 0; t < R; ++t) dg[t] *= kscale;
    for (int i = tid; i < kMaxN; i += NT) ord[i] = -1;
    cluster.sync();

    // ---- pivoted Cholesky without swaps (scaled matrix: diagonal <= 1) ----
    constexpr int CW = (LD + 63) / 64 * 2;                     // upper bound of columns a warp owns (warp + NW u) for NW >= 32
    unsigned colmask = 0u;                                     // bit u: column warp + 32 u is still unpivoted
#pragma unroll
    for (int u = 0; u < CW; ++u)
        if (warp + NW * u < n) colmask |= 1u << u;
    const float tol = 1e-7f;
    int rank = empty ? 0 : n;
    for (int k = 0; k < rank; ++k) {
        unsigned key = 0u;
#pragma unroll
        for (int t = 0; t < R; ++t)
            if (alive[t]) key = max(key, (__float_as_uint(fmaxf(dg[t], 0.f)) & 0xfffffe00u) | (unsigned)(511 - (lane + 32 * t)));
        key = __reduce_max_sync(0xffffffffu, key);                // largest diagonal (24 significant bits), smaller index on ties
        const int p = 511 - (int)(key & 511u);
        if (key == 0u || p >= n) { rank = k; break; }             // identical in every warp
        const float* Xp = X + p * LD;
        const float d = __ldcg(Xp + p);
        if (!(d > tol)) { rank = k; break; }
        const float inv = rsqrtf(d);
        if ((p % NW) == warp) colmask &= ~(1u << (p / NW));
        float li[R];
#pragma unroll
        for (int t = 0; t < R; ++t) {
            const int i = lane + 32 * t;
            if (i == p) alive[t] = false;
            li[t] = alive[t] ? __ldcg(Xp + i) * inv : 0.f;
            dg[t] = fmaf(-li[t], li[t], dg[t]);
        }
#pragma unroll
        for (int u0 = 0; u0 < CW; u0 += 2) {                      // two columns at a time: loads first, then stores
            const bool on0 = (colmask >> u0) & 1u, on1 = (u0 + 1 < CW) && ((colmask >> (u0 + 1)) & 1u);
            if (!on0 && !on1) continue;
            float* c0 = X + (warp + NW * u0) * LD;
            float* c1 = X + (warp + NW * (u0 + 1)) * LD;
            const float l0 = on0 ? __ldcg(Xp + warp + NW * u0) * inv : 0.f;
            const float l1 = on1 ? __ldcg(Xp + warp + NW * (u0 + 1)) * inv : 0.f;
            float v0[R], v1[R];
#pragma unroll
            for (int t = 0; t < R; ++t) {
                v0[t] = on0 ? __ldcg(c0 + lane + 32 * t) : 0.f;
                v1[t] = on1 ? __ldcg(c1 + lane + 32 * t) : 0.f;
            }
#pragma unroll
            for (int t = 0; t < R; ++t) {
                if (on0) c0[lane + 32 * t] = fmaf(-li[t], l0, v0[t]);
                if (on1) c1[lane + 32 * t] = fmaf(-li[t], l1, v1[t]);
            }
        }
        if (tid == 0) { ord[p] = k; perm[k] = p; scl[k] = inv; }   // every CTA keeps its own copy of the tables
        cluster.sync();
    }
    cluster.sync();
    // ---- scale the pivot columns into the factor L (zero above the pivot order, zero unpivoted columns) ----
    for (int e = gtid; e < n * LD; e += GT) {
        const int c = e / LD, i = e - c * LD;
        const int kc = ord[c];
        float v = 0.f;
        if (kc >= 0 && i < n) {
            const int ki = ord[i];
            if (!(ki >= 0 && ki < kc)) v = __ldcg(X + e) * scl[kc];
        }
        X[e] = v;
    }
    cluster.sync();

    // ---- one-sided cyclic Jacobi on the rank pivot columns ----
    // Columns (in pivot order) form blocks of 4. A block round pairs the blocks round-robin, one block
    // pair per warp; the warp rotates the 16 cross pairs of its two blocks in 4 local rounds (one pair per
    // quarter-warp, synchronised inside the warp only), and in the first block round of a sweep also the
    // pairs inside each block. Only the warps that own a block pair take part, on a named barrier.
    const int l8 = tid & 7, qd = lane >> 3;
    int sweeps = 0;
    float worst2 = 0.f;                 // largest squared cosine met in the current sweep
    if (rank >= 2) {
        const int nb = (rank + 3) >> 2, nbe = nb + (nb & 1), nbm1 = nbe - 1, nact = nbe >> 1;   // block pairs per round
        const int nwork = nact < NW ? nact : NW;                  // warps that take part; each owns slots w, w + nwork, ...
        {
            const bool active = warp < nwork;                     // the other warps only take part in the cluster barriers
            auto pair_step = [&](int p, int q) {                  // p, q: pivot-order columns, q >= rank means no pair
                const bool valid = p < rank && q < rank;
                float4* xp = reinterpret_cast<float4*>(X + (valid ? perm[p] : 0) * LD) + l8;
                float4* xq = reinterpret_cast<float4*>(X + (valid ? perm[q] : 0) * LD) + l8;
                float4 x[Q], y[Q];
                float a0 = 0.f, a1 = 0.f, b0 = 0.f, b1 = 0.f, g0 = 0.f, g1 = 0.f;
#pragma unroll
                for (int t = 0; t < Q; ++t) {
                    x[t] = __ldcg(xp + 8 * t);
                    y[t] = __ldcg(xq + 8 * t);
                    a0 = fmaf(x[t].x, x[t].x, a0); a1 = fmaf(x[t].y, x[t].y, a1); a0 = fmaf(x[t].z, x[t].z, a0); a1 = fmaf(x[t].w, x[t].w, a1);
                    b0 = fmaf(y[t].x, y[t].x, b0); b1 = fmaf(y[t].y, y[t].y, b1); b0 = fmaf(y[t].z, y[t].z, b0); b1 = fmaf(y[t].w, y[t].w, b1);
                    g0 = fmaf(x[t].x, y[t].x, g0); g1 = fmaf(x[t].y, y[t].y, g1); g0 = fmaf(x[t].z, y[t].z, g0); g1 = fmaf(x[t].w, y[t].w, g1);
                }
                float a = a0 + a1, b = b0 + b1, g = g0 + g1;
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) {
                    a += __shfl_xor_sync(0xffffffffu, a, o);
                    b += __shfl_xor_sync(0xffffffffu, b, o);
                    g += __shfl_xor_sync(0xffffffffu, g, o);
                }
                const float ab = a * b, g2 = g * g;
                if (valid && ab > 0.f && g2 > 1e-12f * ab) {
                    worst2 = fmaxf(worst2, __fdividef(g2, ab));
                    float c, s;
                    jacobi_rotation(a, b, g, c, s);
#pragma unroll
                    for (int t = 0; t < Q; ++t) {
                        float4 nx, ny;
                        nx.x = fmaf(-s, y[t].x, c * x[t].x); ny.x = fmaf(s, x[t].x, c * y[t].x);
                        nx.y = fmaf(-s, y[t].y, c * x[t].y); ny.y = fmaf(s, x[t].y, c * y[t].y);
                        nx.z = fmaf(-s, y[t].z, c * x[t].z); ny.z = fmaf(s, x[t].z, c * y[t].z);
                        nx.w = fmaf(-s, y[t].w, c * x[t].w); ny.w = fmaf(s, x[t].w, c * y[t].w);
                        xp[8 * t] = nx;
                        xq[8 * t] = ny;
                    }
                }
                __syncwarp();
            };
            int more = 0;
            while (sweeps < max_sweeps) {
                worst2 = 0.f;
                for (int br = 0; br < nbm1; ++br) {
                  for (int slot = active ? warp : nact; slot < nact; slot += nwork) {
                    int ba, bb;                                   // the two blocks of this slot in this block round
                    if (slot == 0) { ba = nbm1; bb = br; }
                    else {
                        ba = br + slot; if (ba >= nbm1) ba -= nbm1;
                        bb = br + nbm1 - slot; if (bb >= nbm1) bb -= nbm1;
                    }
                    if (br == 0) {                                // pairs inside each block: quarters 0,1 -> ba, 2,3 -> bb
                        const int base = 4 * ((qd < 2) ? ba : bb), h = qd & 1;
                        pair_step(base + (h ? 2 : 0), base + (h ? 3 : 1));
                        pair_step(base + (h ? 1 : 0), base + (h ? 3 : 2));
                        pair_step(base + (h ? 1 : 0), base + (h ? 2 : 3));
                    }
                    const int lo = min(ba, bb), hi = max(ba, bb);
                    {   // the 16 cross pairs, columns held in registers: quarter qd keeps column qd of block lo and
                        // the columns of block hi travel from quarter to quarter by shuffles between the 4 rounds
                        const int pa = 4 * lo + qd, pb = 4 * hi + qd;
                        const bool va = pa < rank, vb0 = pb < rank;
                        float4* xa = reinterpret_cast<float4*>(X + (va ? perm[pa] : 0) * LD) + l8;
                        float4* xb = reinterpret_cast<float4*>(X + (vb0 ? perm[pb] : 0) * LD) + l8;
                        float4 x[Q], y[Q];
#pragma unroll
                        for (int t = 0; t < Q; ++t) {
                            x[t] = va ? __ldcg(xa + 8 * t) : make_float4(0.f, 0.f, 0.f, 0.f);
                            y[t] = vb0 ? __ldcg(xb + 8 * t) : make_float4(0.f, 0.f, 0.f, 0.f);
                        }
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const bool valid = va && (4 * hi + ((qd + r) & 3) < rank);
                            float a0 = 0.f, a1 = 0.f, b0 = 0.f, b1 = 0.f, g0 = 0.f, g1 = 0.f;
#pragma unroll
                            for (int t = 0; t < Q; ++t) {
                                a0 = fmaf(x[t].x, x[t].x, a0); a1 = fmaf(x[t].y, x[t].y, a1); a0 = fmaf(x[t].z, x[t].z, a0); a1 = fmaf(x[t].w, x[t].w, a1);
                                b0 = fmaf(y[t].x, y[t].x, b0); b1 = fmaf(y[t].y, y[t].y, b1); b0 = fmaf(y[t].z, y[t].z, b0); b1 = fmaf(y[t].w, y[t].w, b1);
                                g0 = fmaf(x[t].x, y[t].x, g0); g1 = fmaf(x[t].y, y[t].y, g1); g0 = fmaf(x[t].z, y[t].z, g0); g1 = fmaf(x[t].w, y[t].w, g1);
                            }
                            float a = a0 + a1, b = b0 + b1, g = g0 + g1;
#pragma unroll
                            for (int o = 4; o > 0; o >>= 1) {
                                a += __shfl_xor_sync(0xffffffffu, a, o);
                                b += __shfl_xor_sync(0xffffffffu, b, o);
                                g += __shfl_xor_sync(0xffffffffu, g, o);
                            }
                            const float ab = a * b, g2 = g * g;
                            if (valid && ab > 0.f && g2 > 1e-12f * ab) {
                                worst2 = fmaxf(worst2, __fdividef(g2, ab));
                                float c, s;
                                jacobi_rotation(a, b, g, c, s);
#pragma unroll
                                for (int t = 0; t < Q; ++t) {
                                    float4 nx, ny;
                                    nx.x = fmaf(-s, y[t].x, c * x[t].x); ny.x = fmaf(s, x[t].x, c * y[t].x);
                                    nx.y = fmaf(-s, y[t].y, c * x[t].y); ny.y = fmaf(s, x[t].y, c * y[t].y);
                                    nx.z = fmaf(-s, y[t].z, c * x[t].z); ny.z = fmaf(s, x[t].z, c * y[t].z);
                                    nx.w = fmaf(-s, y[t].w, c * x[t].w); ny.w = fmaf(s, x[t].w, c * y[t].w);
                                    x[t] = nx;
                                    y[t] = ny;
                                }
                            }
                            if (r < 3) {                          // quarter qd takes over the column quarter qd + 1 holds
                                const int src = (lane + 8) & 31;
#pragma unroll
                                for (int t = 0; t < Q; ++t) {
                                    y[t].x = __shfl_sync(0xffffffffu, y[t].x, src);
                                    y[t].y = __shfl_sync(0xffffffffu, y[t].y, src);
                                    y[t].z = __shfl_sync(0xffffffffu, y[t].z, src);
                                    y[t].w = __shfl_sync(0xffffffffu, y[t].w, src);
                                }
                            }
                        }
                        const int pl = 4 * hi + ((qd + 3) & 3);   // the hi column this quarter ends up with
                        if (va) {
#pragma unroll
                            for (int t = 0; t < Q; ++t) xa[8 * t] = x[t];
                        }
                        if (pl < rank) {
                            float4* xl = reinterpret_cast<float4*>(X + perm[pl] * LD) + l8;
#pragma unroll
                            for (int t = 0; t < Q; ++t) xl[8 * t] = y[t];
                        }
                        __syncwarp();
                    }
                  }
                    cluster.sync();
                }
                ++sweeps;
                const int par = sweeps & 1;
                if (__any_sync(0xffffffffu, worst2 > 1e-6f) && lane == 0) atomicOr(&gflag[par], 1);
                if (gtid == 0) gflag[par ^ 1] = 0;
                cluster.sync();
                more = __ldcg(&gflag[par]);
                if (!more) break;               // every cosine of this sweep was below 1e-3: converged after it
            }
            if (tid == 0) { sh_f[1] = (float)sweeps; sh_f[4] = more ? 1.f : 0.f; }
        }
    }
    __syncthreads();
    sweeps = rank >= 2 ? (int)sh_f[1] : 0;
    const int not_converged = rank >= 2 && sh_f[4] != 0.f;     // stopped at the sweep limit while still rotating visibly

    // ---- eigenvalues = squared column norms (pivot-step order), scaled back; sort descending, stable ----
    for (int k = lwarp; k < n; k += 8) {                          // every CTA forms all eigenvalues for its own tables
        float a = 0.f;
        if (k < rank) {
            const float* x = X + perm[k] * LD;
#pragma unroll
            for (int t = 0; t < R; ++t) { const float xv = __ldcg(x + lane + 32 * t); a = fmaf(xv, xv, a); }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        }
        if (lane == 0) lam[k] = a * dmax;
    }
    __syncthreads();
    for (int t = tid; t < n; t += NT) {
        const float mine = lam[t];
        int pos = 0;
        for (int i = 0; i < n; ++i) {
            const float o = lam[i];
            pos += (o > mine) || (o == mine && i < t);
        }
        order[pos] = t;
    }
    __syncthreads();
    if (tid == 0) {
        float delta = 0.f;
        if (do_shrink && delta_rank - 1 < n) delta = lam[order[delta_rank - 1]];
        sh_f[0] = delta;
        if (crank == 0) {
            info->delta = delta;
            info->sweeps = sweeps;
            if (sweeps > info->max_sweeps) info->max_sweeps = sweeps;
            info->rank = rank;
            if (not_converged) info->flags |= kFlagNotConverged;
            if (do_shrink) {
                info->sum_delta += (double)delta;
                info->shrinks += 1;
            }
        }
    }
    __syncthreads();
    const float delta = sh_f[0];
    const float back = sqrtf(dmax);     // columns of X are sigma_j u_j / sqrt(dmax)
    for (int t = tid; t < n; t += NT) {
        const float l = lam[order[t]];
        float f = 0.f, sp = 0.f;
        if (l > 0.f && t < keep) {
            const float kept = fmaxf(l - delta, 0.f);
            sp = sqrtf(kept);
            f = sqrtf(kept / l) * rsqrtf(l) * back;   // (sigma'/sigma) / sigma, for the unscaled column
        }
        fac[t] = f;
        if (t < n_sigma && crank == 0) sigma_out[t] = sp;
    }
    if (crank == 0)
        for (int j = n + tid; j < n_sigma; j += NT) sigma_out[j] = 0.f;
    __syncthreads();
    for (int e = gtid; e < n * keep; e += GT) {
        const int j = e / n, i = e - j * n;
        float v = 0.f;
        if (j < n) {
            const int k = order[j];
            if (k < rank) v = __ldcg(X + perm[k] * LD + i) * fac[j];
        }
        Ur[(size_t)i * ldu + j] = v;
    }
    if (Wsplit) {   // the same factors transposed and split for the tensor-core rebuild: [W_hi ; W_lo], zero padded
        for (int e = gtid; e < j_pad * ldw; e += GT) {
            const int j = e / ldw, i = e - j * ldw;
            float v = 0.f;
            if (j < keep && j < n && i < n) {
                const int k = order[j];
                if (k < rank) v = __ldcg(X + perm[k] * LD + i) * fac[j];
            }
            const float hi = __uint_as_float((__float_as_uint(v) + 0x1000u) & 0xffffe000u);
            Wsplit[split_row(j, j_pad, false) * ldw + i] = hi;
            Wsplit[split_row(j, j_pad, true) * ldw + i] = v - hi;
        }
    }
}

__global__ void __launch_bounds__(kThreads, 1)
k_eig_shrink(const float* __restrict__ K, int ldk, int n, int do_shrink, int delta_rank, int keep, float* __restrict__ Ur,
             int ldu, float* __restrict__ sigma_out, int n_sigma, float* __restrict__ work, int use_smem, int max_sweeps,
             EigInfo* __restrict__ info, float* __restrict__ Wsplit, int ldw, int j_pad) {
    extern __shared__ __align__(16) float smem[];
    float* lam = smem;                 // n   eigenvalues (unsorted), later reused
    float* fac = lam + 512;            // n   per sorted position: r_j / sigma_j
    int* perm = reinterpret_cast<int*>(fac + 512);   // n   physical row -> original buffer row
    int* order = perm + 512;           // n   sorted position -> column
    float* red_v = reinterpret_cast<float*>(order + 512);   // kWarps
    int* red_i = reinterpret_cast<int*>(red_v + kWarps);    // kWarps
    int* sh_int = red_i + kWarps;      // [0] pivot index, [1] rank
    float* sh_f = reinterpret_cast<float*>(sh_int + 4);     // [0] pivot value, [1] delta
    float* X = use_smem ? (sh_f + 4) : work;
    const int ldx = n;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // ---- load K (full symmetric storage, column-major X[c*ldx + i] = K[i][c]) ----
    for (int e = tid; e < n * n; e += kThreads) {
        const int i = e / n, c = e % n;
        X[(size_t)c * ldx + i] = K[(size_t)i * ldk + c];
    }
    if (tid < n) perm[tid] = tid;
    if (tid == 0) sh_int[1] = n;
    __syncthreads();

    // ---- pivoted Cholesky, right-looking, in place ----
    float tol = 0.f;
    int rank = n;
    for (int k = 0; k < n; ++k) {
        ArgMax am{-1.f, 0x7fffffff};
        if (tid >= k && tid < n) {
            const float d = X[(size_t)tid * ldx + tid];
            if (fabsf(d) <= 3.0e38f) am = ArgMax{d, tid};
            else if (k == 0) atomicOr(&info->flags, kFlagNonFinite);    // NaN/Inf rows reached the buffer
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            ArgMax other{__shfl_xor_sync(0xffffffffu, am.v, o), __shfl_xor_sync(0xffffffffu, am.i, o)};
            am = better(am, other);
        }
        if (lane == 0) { red_v[warp] = am.v; red_i[warp] = am.i; }
        __syncthreads();
        if (warp == 0) {
            ArgMax a{red_v[lane], red_i[lane]};
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                ArgMax other{__shfl_xor_sync(0xffffffffu, a.v, o), __shfl_xor_sync(0xffffffffu, a.i, o)};
                a = better(a, other);
            }
            if (lane == 0) { sh_f[0] = a.v; sh_int[0] = a.i; }
        }
        __syncthreads();
        const float d = sh_f[0];
        const int p = sh_int[0];
        if (k == 0) tol = fmaxf(d * 1e-7f, 1e-37f);
        if (!(d > tol) || p >= n) { rank = k; break; }     // uniform across the block
        if (p != k) {
            // swap rows k and p in every column, then columns k and p for rows >= k
            for (int c = tid; c < n; c += kThreads) {
                const float a = X[(size_t)c * ldx + k], b = X[(size_t)c * ldx + p];
                X[(size_t)c * ldx + k] = b;
                X[(size_t)c * ldx + p] = a;
            }
            __syncthreads();
            for (int i = k + tid; i < n; i += kThreads) {
                const float a = X[(size_t)k * ldx + i], b = X[(size_t)p * ldx + i];
                X[(size_t)k * ldx + i] = b;
                X[(size_t)p * ldx + i] = a;
            }
            if (tid == 0) { const int t = perm[k]; perm[k] = perm[p]; perm[p] = t; }
            __syncthreads();
        }
        const float lkk = sqrtf(d), inv = 1.f / lkk;
        for (int i = tid; i < n; i += kThreads) {
            float v = X[(size_t)k * ldx + i];
            v = (i < k) ? 0.f : (i == k ? lkk : v * inv);
            X[(size_t)k * ldx + i] = v;
        }
        __syncthreads();
        {   // trailing update S[i][j] -= L[i][k] L[j][k], rows along lanes
            const float* Lk = X + (size_t)k * ldx;
            for (int j = k + 1 + warp; j < n; j += kWarps) {
                const float lj = Lk[j];
                float* col = X + (size_t)j * ldx;
                for (int i = k + 1 + lane; i < n; i += 32) col[i] = fmaf(-Lk[i], lj, col[i]);
            }
        }
        __syncthreads();
    }
    // columns >= rank do not take part; zero them so that later norms are exact zeros
    for (int e = tid; e < (n - rank) * n; e += kThreads) X[(size_t)rank * ldx + e] = 0.f;
    __syncthreads();

    // ---- one-sided cyclic Jacobi on columns 0..rank-1 ----
    const float jtol = 1e-6f;
    int sweeps = 0;
    float worst = 0.f;
    if (rank >= 2) {
        const int ne = rank + (rank & 1);
        for (; sweeps < max_sweeps; ++sweeps) {
            int rotated = 0;
            worst = 0.f;
            for (int round = 0; round < ne - 1; ++round) {
                for (int slot = warp; slot < ne / 2; slot += kWarps) {
                    int p, q;
                    rr_pair(ne, round, slot, p, q);
                    if (q >= rank) continue;
                    float* xp = X + (size_t)p * ldx;
                    float* xq = X + (size_t)q * ldx;
                    float a = 0.f, b = 0.f, g = 0.f;
                    for (int i = lane; i < n; i += 32) {
                        const float x = xp[i], y = xq[i];
                        a = fmaf(x, x, a);
                        b = fmaf(y, y, b);
                        g = fmaf(x, y, g);
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        a += __shfl_xor_sync(0xffffffffu, a, o);
                        b += __shfl_xor_sync(0xffffffffu, b, o);
                        g += __shfl_xor_sync(0xffffffffu, g, o);
                    }
                    const float lim = sqrtf(a) * sqrtf(b);
                    const float ag = fabsf(g);
                    if (!(lim > 0.f) || !(ag > jtol * lim)) continue;
                    worst = fmaxf(worst, ag / lim);
                    const float zeta = (b - a) / (2.f * g);
                    const float t = copysignf(1.f, zeta) / (fabsf(zeta) + sqrtf(fmaf(zeta, zeta, 1.f)));
                    const float c = rsqrtf(fmaf(t, t, 1.f));
                    const float s = c * t;
                    for (int i = lane; i < n; i += 32) {
                        const float x = xp[i], y = xq[i];
                        xp[i] = c * x - s * y;
                        xq[i] = fmaf(s, x, c * y);
                    }
                    rotated = 1;
                }
                __syncthreads();
            }
            if (!__syncthreads_or(rotated)) break;
        }
    }
    // a run that stopped at the sweep limit while still rotating by a visible amount did not converge
    const int not_converged = __syncthreads_or(sweeps >= max_sweeps && worst > 1e-4f);

    // ---- eigenvalues = squared column norms; sort descending (stable by column index) ----
    for (int c = warp; c < n; c += kWarps) {
        float a = 0.f;
        if (c < rank) {
            const float* x = X + (size_t)c * ldx;
            for (int i = lane; i < n; i += 32) a = fmaf(x[i], x[i], a);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        }
        if (lane == 0) lam[c] = a;
    }
    __syncthreads();
    if (tid < n) {
        const float mine = lam[tid];
        int pos = 0;
        for (int i = 0; i < n; ++i) {
            const float o = lam[i];
            pos += (o > mine) || (o == mine && i < tid);
        }
        order[pos] = tid;
    }
    __syncthreads();
    if (tid == 0) {
        float delta = 0.f;
        if (do_shrink && delta_rank - 1 < n) delta = lam[order[delta_rank - 1]];
        sh_f[1] = delta;
        info->delta = delta;
        info->sweeps = sweeps;
        if (sweeps > info->max_sweeps) info->max_sweeps = sweeps;
        info->rank = rank;
        if (not_converged) info->flags |= kFlagNotConverged;
        if (do_shrink) {
            info->sum_delta += (double)delta;
            info->shrinks += 1;
        }
    }
    __syncthreads();
    const float delta = sh_f[1];
    if (tid < n) {
        const float l = lam[order[tid]];
        float f = 0.f, sp = 0.f;
        if (l > 0.f && tid < keep) {
            const float kept = fmaxf(l - delta, 0.f);
            sp = sqrtf(kept);
            f = sqrtf(kept / l) * rsqrtf(l);       // (sigma'/sigma) / sigma : scales the column sigma_j u_j
        }
        fac[tid] = f;
        if (tid < n_sigma) sigma_out[tid] = sp;
    }
    for (int j = n + tid; j < n_sigma; j += kThreads) sigma_out[j] = 0.f;
    __syncthreads();

    // ---- Ur[orig_row][j] = u_j[orig_row] * sigma'_j / sigma_j ----
    for (int e = tid; e < n * keep; e += kThreads) {
        const int j = e / n, i = e % n;      // i fastest: conflict-free reads of X
        float v = 0.f;
        if (j < n) v = X[(size_t)order[j] * ldx + i] * fac[j];
        Ur[(size_t)perm[i] * ldu + j] = v;
    }
    if (Wsplit) {
        for (int e = tid; e < j_pad * ldw; e += kThreads) {
            const int j = e / ldw, c = e - j * ldw;
            Wsplit[split_row(j, j_pad, false) * ldw + c] = 0.f;
            Wsplit[split_row(j, j_pad, true) * ldw + c] = 0.f;
        }
        __syncthreads();
        for (int e = tid; e < n * keep; e += kThreads) {
            const int j = e / n, i = e % n;
            if (j >= n || j >= j_pad) continue;
            const float v = X[(size_t)order[j] * ldx + i] * fac[j];
            const float hi = __uint_as_float((__float_as_uint(v) + 0x1000u) & 0xffffe000u);
            Wsplit[split_row(j, j_pad, false) * ldw + perm[i]] = hi;
            Wsplit[split_row(j, j_pad, true) * ldw + perm[i]] = v - hi;
        }
    }
}

}  // namespace

cudaError_t launch_eig_shrink(const float* K, int ldk, int n, int do_shrink, int delta_rank, int keep, float* Ur, int ldu,
                              float* sigma_out, int n_sigma, float* work, int max_sweeps, EigInfo* info, float* Wsplit, int ldw,
                              int j_pad, int variant, cudaStream_t st) {
    if (n <= 0 || n > 512) return cudaErrorInvalidValue;
    if (variant == 0) {
        const cudaError_t e = launch_eig_direct(K, ldk, n, do_shrink, delta_rank, keep, Ur, ldu, sigma_out, n_sigma, work, info, Wsplit, ldw, j_pad, st);
        // where a cluster of eight blocks cannot be launched (its first launch), the kernels below serve every n <= 512
        if (n <= 128 || (e != cudaErrorInvalidClusterSize && e != cudaErrorLaunchOutOfResources)) return e;
        (void)cudaGetLastError();
    }
    if (n <= kMaxFast) {
        const int T = (n + 63) / 64;
        const size_t aux_bytes = 3 * kMaxN * sizeof(float) + 3 * kMaxN * sizeof(int) + 32;
        const size_t bytes = (size_t)(64 * T) * (64 * T) * sizeof(float) + aux_bytes;
        cudaError_t e;
#define SAGE_EIG_FAST(TT)                                                                                              \
    e = cudaFuncSetAttribute(k_eig_shrink_fast<TT, 1024, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes); \
    if (e != cudaSuccess) return e;                                                                                    \
    return launch(k_eig_shrink_fast<TT, 1024, false>, LaunchShape{dim3(1), dim3(1024), bytes, 1, false}, st, K, ldk, n, do_shrink, delta_rank, keep, \
                  Ur, ldu, sigma_out, n_sigma, max_sweeps, info, Wsplit, ldw, j_pad, work);
        if (T == 1) { SAGE_EIG_FAST(1) } else if (T == 2) { SAGE_EIG_FAST(2) } else { SAGE_EIG_FAST(3) }
#undef SAGE_EIG_FAST
    }
    {   // thread-block cluster, matrix in `work` (>= 512*512 + 64 floats when n > 256, else >= 256*256 + 64)
        const size_t bytes = 3 * 512 * sizeof(float) + 3 * 512 * sizeof(int) + 32;
        const LaunchShape shape{dim3(8), dim3(256), bytes, 8, false};
        const cudaError_t e = n <= 256 ? launch(k_eig_shrink_cluster<4>, shape, st, K, ldk, n, do_shrink, delta_rank, keep, Ur, ldu, sigma_out, n_sigma, max_sweeps,
                                                info, Wsplit, ldw, j_pad, work)
                                       : launch(k_eig_shrink_cluster<8>, shape, st, K, ldk, n, do_shrink, delta_rank, keep, Ur, ldu, sigma_out, n_sigma, max_sweeps,
                                                info, Wsplit, ldw, j_pad, work);
        if (e != cudaErrorInvalidClusterSize && e != cudaErrorLaunchOutOfResources) return e;
        (void)cudaGetLastError();          // the one-CTA kernel below serves n <= 512
    }
    const size_t aux = (4 * 512 + 2 * kWarps + 8) * sizeof(float);
    const size_t xbytes = (size_t)n * n * sizeof(float);
    static int max_optin = -1;
    if (max_optin < 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&max_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    }
    const int use_smem = (aux + xbytes + 64 <= (size_t)max_optin) ? 1 : 0;
    const size_t smem = aux + (use_smem ? xbytes : 0) + 64;
    cudaError_t e = cudaFuncSetAttribute(k_eig_shrink, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch(k_eig_shrink, LaunchShape{dim3(1), dim3(kThreads), smem, 1, false}, st, K, ldk, n, do_shrink, delta_rank, keep, Ur, ldu, sigma_out, n_sigma, work,
                  use_smem, max_sweeps, info, Wsplit, ldw, j_pad);
}

}  // namespace sage
