// Internal declarations shared by the host orchestration and the kernel translation units.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <algorithm>
#include <tuple>

#include "sage.h"

namespace sage {

// ---- launches of the shrink cycle ------------------------------------------------------------------------------------
// The kernels of a cycle follow one another on a stream and each is short, so the gaps between them count. They are launched
// with programmatic stream serialisation: a kernel may start, set up its barriers and allocate while its predecessor ends;
// chain_wait() in it returns when every kernel before it on the stream has finished and its results are visible (each kernel
// of the chain waits, so this holds for all of them), and nothing of theirs is touched before. chain_release() lets the next
// one start; kernels that run long call it near their end, so that the next does not sit on an SM for nothing.
// Every launch of a shrink cycle goes through launch(): it enqueues, or adds the launch to the graph that the calling thread is
// putting together (see run_cycle in api.cu).
struct LaunchShape {
    dim3 grid, block;
    size_t smem = 0;
    unsigned cluster = 1;
    bool chained = true;
};
cudaError_t launch_any(const void* kernel, const LaunchShape& shape, void** args, cudaStream_t st);
template <typename... P, typename... A>
cudaError_t launch(void (*kernel)(P...), const LaunchShape& shape, cudaStream_t st, A... a) {
    std::tuple<P...> values(static_cast<P>(a)...);
    return std::apply(
        [&](auto&... v) {
            void* args[] = {&v...};
            return launch_any(reinterpret_cast<const void*>(kernel), shape, args, st);
        },
        values);
}
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... a) {
    return launch(kernel, LaunchShape{grid, block, smem}, st, a...);
}
#ifdef __CUDACC__
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Row of the split rebuild factors [W_hi ; W_lo] that holds output row j: stacked as two blocks of j_pad rows, or, when
// more than 128 output rows are kept, as one such pair per 128 output rows, as k_tc_rebuild_wide reads them.
__device__ __forceinline__ size_t split_row(int j, int j_pad, bool lo) {
    if (j_pad <= 128) return (size_t)(lo ? j_pad + j : j);
    return (size_t)(j >> 7) * 256 + (size_t)(j & 127) + (lo ? 128 : 0);
}
#endif

// Lets a kernel use up to `bytes` of dynamic shared memory; the driver is asked once per kernel and device. regs > 0: the kernel hands
// registers from some of its warps to others and has to be compiled with exactly that many a thread; cudaErrorInvalidKernelImage
// otherwise, which callers report: the launchers' cudaErrorNotSupported, for which they take other kernels, is about operands only.
cudaError_t allow_smem(const void* kernel, int bytes, int regs = 0);

// Device-side flags accumulated in the handle's status word.
constexpr uint32_t kFlagNotConverged = 1u;
constexpr uint32_t kFlagNonFinite = 2u;
constexpr uint32_t kFlagExchangeTimeout = 8u;   // a bounded wait between thread blocks of the eigen-solve ran out (4: tensor-core waits)

// Results of one eigen-solve, written by the eigen kernel and read by later kernels / stats.
struct EigInfo {
    double sum_delta;   // running sum of delta over shrinks
    float delta;        // delta of the most recent shrink
    int sweeps;         // sweeps of the most recent solve
    int max_sweeps;
    int rank;           // numerical rank of the most recent Gram matrix
    unsigned flags;     // kFlag*
    long long shrinks;  // shrinks applied so far
};

// ---- launchers (each enqueues on `st` and returns cudaGetLastError()) -----------------------------

// B[dst_row0 + i, 0:D] = float(rows[i, 0:D]) for i < n; columns D..pitch-1 of those rows are zeroed.
// n2 > 0: the n2 rows after them come from rows2 (same type and pitch).
cudaError_t launch_append(const void* rows, sage_dtype_t dt, int64_t n, int64_t ld, int64_t D, float* B,
                          int64_t pitch, int dst_row0, cudaStream_t st, const void* rows2 = nullptr, int64_t n2 = 0);

// Structured last-layer rows: B[dst_row0 + i, :] = [vec_rowmajor(q_i feat_i^T) ; q_i] for i < n, with q n x C (pitch ldq) and feat
// n x F (pitch ldf) of element type dt; products in fp32 (exact for bf16 factors); columns C F + C .. pitch-1 zeroed. pitch
// must be a multiple of 4.
cudaError_t launch_append_outer(const void* q, int64_t ldq, const void* feat, int64_t ldf, sage_dtype_t dt, int64_t n, int C, int F,
                                float* B, int64_t pitch, int dst_row0, cudaStream_t st, const void* q2 = nullptr, const void* feat2 = nullptr,
                                int64_t n2 = 0);

// Projection of structured rows from per-class planes: with T[c] = feat * S_c^T (n x ell, the sum of pp consecutive planes of
// `planes`, plane_stride floats apart, n x ell each with pitch ell) and S_c the columns [c F, c F + F) of the sketch,
//     Z[i][j] = sum_c q[i][c] * (T[c][i][j] + Sb[j][c]),      Sb = S + C F (the bias columns of the sketch, pitch lds).
// Classes are added in ascending order in fp32. q is n x C of element type dt (pitch ldq); Z is n x ell, pitch ell. biasT:
// scratch of C x ell floats (receives Sb transposed). Two launches.
cudaError_t launch_outer_combine(const void* q, int64_t ldq, sage_dtype_t dt, int C, const float* planes, int pp, int64_t plane_stride,
                                 const float* Sb, int64_t lds, float* biasT, int64_t n, int ell, float* Z, cudaStream_t st);

// C[z][i][j] = sum over the z-th K-slice of A[i][k] * Bm[j][k]   (both operands contiguous along k).
// A is M x K (element type dt, pitch lda), Bm is N x K fp32 (pitch ldb). splits >= 1 slices of k.
// class_F > 0 ("class slices", needs splits * class_F == K): A is M x class_F and slice z contracts ALL of it with the columns
// [z class_F, (z + 1) class_F) of Bm, so C[z] = A * Bm_z^T: the per-class projections of structured rows in one launch.
cudaError_t launch_gemm_nt(const void* A, sage_dtype_t dt, int64_t lda, const float* Bm, int64_t ldb, int M, int N,
                           int64_t K, int splits, float* C, int64_t ldc, int64_t split_stride, cudaStream_t st, int64_t class_F = 0);

// Tensor-core version of launch_gemm_nt (tcgen05 + TMA). Both operands have element type dt (fp32 operands are
// read as tf32) and must satisfy TMA's rules: 16-byte aligned base, pitch a multiple of 16 bytes.
// Returns cudaErrorNotSupported when they do not, so that the caller can take launch_gemm_nt instead.
// fold != 0: Bm holds two stacked operands, rows [0, N) and rows [n_pad, n_pad + N) with n_pad = N rounded up to
// 16, and C receives the sum of both products (a two-term representation of a more precise B); needs 2 n_pad <= 256.
// Without fold N <= 256. *err (device) is set to 1 if a bounded wait inside the kernel ran out.
// mt (1, 2 or 4) row tiles of 128 share each B tile inside one CTA; needs mt * (fold ? 2 n_pad : n_pad) <= 512.
cudaError_t launch_tc_gemm_nt(const void* A, sage_dtype_t dt, int64_t lda, const void* Bm, int64_t ldb, int M, int N, int fold,
                              int mt, int64_t K, int splits, float* C, int64_t ldc, int64_t split_stride, int* err, cudaStream_t st,
                              int64_t class_F = 0);   // class slices as in launch_gemm_nt; needs class_F * element size a multiple of 16

// fp32-faithful tensor-core C[z] = A_z * Bm_z^T for fp32 operands (three tf32 MMAs on hi/lo halves split in shared
// memory, accumulator drained into registers every few K tiles). Same alignment rules and return convention as
// launch_tc_gemm_nt; any N.
// sym == 1 (a Gram matrix of at most 128 rows, A == Bm): two MMAs per K step instead of three; slice z then stores
// T_z = hi*hi^T + 2*hi*lo^T and the Gram matrix is sum_z (T_z + T_z^T)/2: see launch_gram_sym_reduce.
cudaError_t launch_tc_gemm_nt_x3(const float* A, int64_t lda, const float* Bm, int64_t ldb, int M, int N, int64_t K, int splits,
                                 float* C, int64_t ldc, int64_t split_stride, int sym, int* err, cudaStream_t st,
                                 int64_t class_F = 0);   // class slices as in launch_gemm_nt; needs class_F a multiple of 4
// The symmetric form of launch_tc_gemm_nt_x3 (sym = 1) for a buffer whose last n_new rows have not been appended: rows
// 0 .. old_rows - 1 come from Bold (fp32, pitch elements; one more row must be readable), the n_new rows after them are
// bfloat16 rows at src (pitch ld_src). old_rows + n_new <= 128, old_rows + 1 a multiple of 8. Same output as the appended form.
cudaError_t launch_tc_gram_direct(const float* Bold, int64_t pitch, int old_rows, const void* src, int64_t ld_src, int n_new, int64_t D,
                                  int splits, float* C, int64_t ldc, int64_t split_stride, int* err, cudaStream_t st);
// Sums the slices of a Gram matrix in the symmetric form; n_off: slices of the 256 x 256 tile above the diagonal (more than 256 rows).
cudaError_t launch_gram_sym_reduce(const float* parts, int splits, int64_t stride, int r, int64_t ldp, float* out, int64_t ldo,
                                   cudaStream_t st, int n_off = 0);

// Projection of M fp32 rows onto a sketch of ell <= 64 rows (tc_project.cu), given as launch_split_tf32 leaves it: Z as partial planes
// of M x ell floats at out, plane_stride apart, project_planes(M, K, class_F) of them. class_F as in launch_gemm_nt (a multiple of 4).
// cudaErrorNotSupported where launch_tc_gemm_nt_x3 returns it.
inline int64_t project_pairs(int64_t tiles, int64_t nkt) {      // of SMs: one for every 16 K tiles of 256 rows or for every row tile
    return std::min<int64_t>(74, std::max(tiles, tiles * nkt / 16));
}
int project_planes(int64_t M, int64_t K, int64_t class_F);
cudaError_t launch_tc_project(const float* rows, int64_t ld, const float* sk_split, int64_t lds, int64_t M, int ell, int64_t K, int64_t class_F,
                              float* out, int64_t plane_stride, int* err, cudaStream_t st);

// Gram matrix of 129 to 512 rows (tc_gram_pair.cu): partials of K slice z at C + z * split_stride, n_diag slices of the 256 x 256 tiles on
// the diagonal in the symmetric form (launch_gram_sym_reduce), n_off of the one above it (0 without one). ldc a multiple of 4, C
// 16-byte aligned; cudaErrorNotSupported otherwise.
cudaError_t launch_tc_gram_pair(const float* B, int64_t ldb, int r, int64_t K, int n_diag, int n_off, float* C, int64_t ldc, int64_t split_stride, int* err,
                                cudaStream_t st);

// Tensor-core rebuild: Bdst[j][d] = sum_{i<r} W[j][i] * Bsrc[i][d] for j < keep, d < pitch (fp32-faithful, see
// tc_rebuild.cu). Wsplit holds W already split for tf32: rows [0, j_pad) = W rounded to 11 significant bits, rows
// [j_pad, 2 j_pad) = the remainder; row pitch ldw floats, columns i >= r and rows j >= keep zero (rows the eigen-solve
// does not write, up to the next multiple of 128, are read by the MMA and must be finite: the caller zeroes the array
// once). Needs j_pad a multiple of 16 with keep <= j_pad <= 256 and r <= 512;
// returns cudaErrorNotSupported otherwise.
cudaError_t launch_tc_rebuild(const float* Wsplit, int ldw, int j_pad, const float* Bsrc, float* Bdst, int64_t pitch, int64_t D, int r,
                              int keep, int* err, cudaStream_t st);
// The same rebuild for a buffer whose last n_new rows have not been appended: rows 0 .. r - n_new - 1 come from Bsrc (one
// more row must be readable), the n_new rows after them are bfloat16 rows at src (pitch ld_src, D columns). Needs r <= 128,
// r and r - n_new + 1 multiples of 32, and the factors resident (at most 64 output rows); cudaErrorNotSupported otherwise.
cudaError_t launch_tc_rebuild_direct(const float* Wsplit, int ldw, int j_pad, const float* Bsrc, float* Bdst, int64_t pitch, int64_t D,
                                     int r, int keep, const void* src, int64_t ld_src, int n_new, int* err, cudaStream_t st);

// hi[i][0:cols] = bf16(src[i][0:cols]) (round to nearest even) for i < rows; when lo != nullptr also
// lo[i][:] = bf16(src - float(hi)), so that hi + lo carries 16 significant bits of src.
cudaError_t launch_to_bf16(const float* src, int64_t lds, int rows, int64_t cols, __nv_bfloat16* hi, __nv_bfloat16* lo, int64_t ldd,
                           cudaStream_t st);

// out[i][j] = sum_z parts[z][i][j] in ascending z with fp64 accumulation. (M x N, pitches ldp / ldo.)
// out (128 rows, pitch ldo): row j = src row j rounded to 11 significant bits, row 64 + j = the remainder, for
// j < rows <= 64; the other rows are left as they are (zero from allocation).
cudaError_t launch_split_tf32(const float* src, int64_t lds, int rows, int64_t cols, float* out, int64_t ldo, cudaStream_t st);

cudaError_t launch_split_reduce(const float* parts, int splits, int64_t split_stride, int M, int N, int64_t ldp,
                                float* out, int64_t ldo, cudaStream_t st);

// out[j][d] = sum_{i<r} Ur[i*ldu + j] * Bsrc[i*pitch + d] for j < keep; rows keep..m_total-1 of out are zeroed.
cudaError_t launch_rebuild(const float* Ur, int ldu, const float* Bsrc, float* Bdst, int64_t pitch, int64_t D, int r,
                           int keep, int m_total, cudaStream_t st);

// Eigen-decomposition of the symmetric positive semi-definite n x n matrix K (pitch ldk) and the
// Frequent-Directions shrink factors. do_shrink != 0: delta = lambda at 1-indexed rank delta_rank (0 if the
// matrix has fewer eigenvalues), keep = delta_rank-1 columns. do_shrink == 0: delta = 0, keep columns.
// Writes Ur[i*ldu + j] = U[i][j] * sqrt(max(1 - delta/lambda_j, 0)) for j < keep (eigenvalues descending),
// sigma_out[j] = sqrt(max(lambda_j - delta, 0)) for j < n_sigma, and updates *info.
// `work` is scratch of at least eig_work_floats(n) floats. variant 0: the direct solve (eig_tridiag.cu; ldk a multiple of 4),
// 1: the iterative one (eig.cu; max_sweeps bounds its sweeps).
// Wsplit != nullptr: also writes the factors transposed and split for launch_tc_rebuild, rows [0, j_pad) =
// W rounded to 11 significant bits and rows [j_pad, 2 j_pad) = the remainders, W[j][i] = Ur[i][j], pitch ldw >= n,
// zero outside j < keep, i < n.
cudaError_t launch_eig_shrink(const float* K, int ldk, int n, int do_shrink, int delta_rank, int keep, float* Ur,
                              int ldu, float* sigma_out, int n_sigma, float* work, int max_sweeps, EigInfo* info,
                              float* Wsplit, int ldw, int j_pad, int variant, cudaStream_t st);
cudaError_t launch_eig_direct(const float* K, int ldk, int n, int do_shrink, int delta_rank, int keep, float* Ur, int ldu, float* sigma_out,
                              int n_sigma, float* work, EigInfo* info, float* Wsplit, int ldw, int j_pad, cudaStream_t st);
size_t eig_work_floats(int n);             // scratch of either variant
int eig_launches(int n, int variant);      // kernels of one solve

// Z (n x ell, pitch ldz; planes > 1: that many partial planes plane_stride floats apart, summed in plane order with fp64
// accumulation) -> zhat rows, ||z|| and per-block partial sums of zhat. zsum (ell doubles, may be null) += the partial sums in
// a fixed order (done by a second, single-block kernel).
cudaError_t launch_normalise(const float* Z, int planes, int64_t plane_stride, int64_t ldz, int64_t n, int ell, float* zhat,
                             float* znorm, float* partials, double* zsum, unsigned* flags, cudaStream_t st);

// u = zsum/||zsum|| (0 if zsum = 0); scores[i] = <zhat_i, u>.
cudaError_t launch_consensus_score(const double* zsum, const float* zhat, int64_t N, int ell, float* u, float* scores,
                                   cudaStream_t st);

// Class-balanced variant. U (C x ell) receives the unit centroids, counts (C) the class sizes, scores (N) the
// per-class agreement scores; labels outside [0, C) score 0. scratch: class_scratch_bytes (may be none).
size_t class_scratch_bytes(int64_t N, int ell, int C);
int class_score_launches(int64_t N, int ell, int C);
cudaError_t launch_class_scores(const float* zhat, const int* labels, int64_t N, int ell, int C, float* U, int* counts, float* scores,
                                void* scratch, cudaStream_t st);
// Rows grouped by class, ascending index inside a class, rows without a class last: order (N); starts (C + 1): first place of
// each class. scratch: select_scratch_bytes.
cudaError_t launch_class_order(const int* labels, int64_t N, int C, void* scratch, unsigned* order, unsigned* starts, cudaStream_t st);
int class_order_launches(int64_t N, int C);
// starts as above; counts (C, may be null): class sizes.
cudaError_t launch_class_starts(const int* labels, int64_t N, int C, unsigned* starts, unsigned* counts, cudaStream_t st);
// Per-class top-k_c. One launch, quotas included, where class_select_in_one says so: kc receives the C quotas and their sum.
bool class_select_in_one(int64_t N, int C);
cudaError_t launch_class_select(const float* scores, const int* labels, int64_t N, int C, double keep_rate, void* scratch, int64_t* idx,
                                long long* kc, cudaStream_t st);
// Otherwise with given quotas: idx[offs[c] + r] = the r-th best example of class c, r < kc[c]. class_pick_launches: with launch_class_starts.
int class_pick_launches(int64_t N, int C);
cudaError_t launch_class_pick(const float* scores, const int* labels, int64_t N, int C, void* scratch, const unsigned* starts, const long long* kc,
                              const long long* offs, int64_t* idx, cudaStream_t st);

// Top-k by (score desc, index asc). scratch: select_scratch_bytes. Returns through idx (device).
cudaError_t select_scratch_bytes(int64_t N, size_t* bytes);
int select_launches(int64_t N, int64_t k);
cudaError_t launch_select(const float* scores, int64_t N, int64_t k, int64_t* idx, void* scratch, cudaStream_t st);

// ---- blocks of shrink cycles (block_kernels.cu, tc_gram_block.cu, tc_rebuild_block.cu) -------------------------------------------
// A block holds the rows of several shrink cycles: logical rows 0 .. s_rows - 1 are the sketch as it stood when the block began, the
// rows given since follow. Each is kept as planes of bfloat16 that add up to it exactly, one plane after the other: 3 for rows of the
// sketch, np for rows in the store, 1 for bfloat16 rows that stay where the caller holds them. The planes of the three places lie
// behind one another in the order of the logical rows, each place rounded up to 32 planes (the surplus reads as zero).
struct BlockMap {
    int s_rows, np, n_store, n_in;
    int oR, oI, P;                 // where the planes of the store begin, those in place, and the end
};
struct BlockSource {
    const __nv_bfloat16 *S, *R;
    int64_t pitch;                 // of S and R: values, a multiple of 64
    const void* in_place;
    int64_t ld_in;
};
#ifdef __CUDACC__
#define SAGE_HD __host__ __device__
#else
#define SAGE_HD
#endif
SAGE_HD inline int block_rows(const BlockMap& m) { return m.s_rows + m.n_store + m.n_in; }
SAGE_HD inline int block_phys(const BlockMap& m, int i) {         // the first plane of logical row i
    const int r = i - m.s_rows;
    return r < 0 ? 3 * i : r < m.n_store ? m.oR + m.np * r : m.oI + (r - m.n_store);
}
SAGE_HD inline int block_planes(const BlockMap& m, int i) { return i < m.s_rows ? 3 : i < m.s_rows + m.n_store ? m.np : 1; }
inline BlockMap block_map(int s_rows, int np, int n_store, int n_in) {
    auto up = [](int x) { return (x + 31) & ~31; };
    const int oR = up(3 * s_rows), oI = oR + up(np * n_store);
    return {s_rows, np, n_store, n_in, oR, oI, oI + up(n_in)};
}
// Tiles of 256 x 256 planes on and above the diagonal whose column block is `first` or later.
inline int block_tiles(const BlockMap& m, int first) {
    const int nb = (m.P + 255) / 256;
    return nb * (nb + 1) / 2 - first * (first + 1) / 2;
}
#ifndef SAGE_OPTIONAL
#define SAGE_OPTIONAL __attribute__((weak))      // a library linked without the block kernels does without blocks
#endif
// Between the two calls this thread may wait for streams while a stream is being captured somewhere.
void allow_work_beside_capture(bool on) SAGE_OPTIONAL;
// Planes of n rows (dense: rows, pitch ld; or factors) to rows row0 .. of the store: np planes a row, zero beyond D.
cudaError_t launch_block_append(const void* rows, sage_dtype_t dt, int64_t n, int64_t ld, int64_t D, __nv_bfloat16* R, int64_t pitch, int np,
                                int64_t row0, cudaStream_t st) SAGE_OPTIONAL;
cudaError_t launch_block_append_outer(const void* q, int64_t ldq, const void* feat, int64_t ldf, sage_dtype_t dt, int64_t n, int C, int F,
                                      __nv_bfloat16* R, int64_t pitch, int np, int64_t row0, cudaStream_t st) SAGE_OPTIONAL;
// out[i] = the sum of the np planes of row i, i < n (fp32, pitch ldo, zero beyond D up to ldo).
cudaError_t launch_block_unpack(const __nv_bfloat16* R, int64_t pitch, int np, int n, int64_t D, float* out, int64_t ldo, cudaStream_t st) SAGE_OPTIONAL;
// Inner products of planes, as partial tiles: see tc_gram_block.cu. Tiles that hold a row from logical row first_new on;
// block_tiles(map, block_phys(map, first_new) / 256) * slices of 65,536 floats at parts.
cudaError_t launch_block_gram(const BlockSource& src, const BlockMap& map, int first_new, int64_t D, int slices, float* parts, int* err,
                              cudaStream_t st) SAGE_OPTIONAL;
// P[i][j] and P[j][i] (pitch ldP) for j >= first_new, i <= j: the sums over planes and slices, fp64.
cudaError_t launch_block_gram_reduce(const float* parts, const BlockMap& map, int first_new, int slices, float* P, int ldP, cudaStream_t st) SAGE_OPTIONAL;
// The inner products of a block seen from its cycle c: the kept rows of cycle c are combinations of logical rows before
// b_c = keep + c step, its window is them and logical rows b_c .. b_c + step - 1. U[k] (m x keep, pitch ldu, U_stride floats apart): the
// factors that cycle k's solve left. C (keep x columns, pitch ldP): inner products of the kept rows with logical rows b_c on.
struct BlockSmall {
    int m, keep, step;
    const float* P;
    int ldP;
    float* C;
    const float* U;
    int ldu;
    int64_t U_stride;
    float* K;                      // the window's matrix of a cycle c > 0 (that of cycle 0 is P): K + (c & 1) * K_stride, pitch ldk
    int64_t K_stride;
    int ldk;
    float* Y;                      // scratch, m x keep, pitch ldu
};
inline int block_step_launches(int m, bool inner) { return inner && m > 128 ? 2 : 1; }
// Columns [col0, col1) of C from cycle c0's to cycle c1's (c0 = 0: from P), those of [col1, late1) from cycle 0's, and what they give of
// window c1; inner: c1 = c0 + 1, also the inner products of the kept rows with each other, from window c0 (and, without late columns,
// the launch follows window c0's solve).
cudaError_t launch_block_step(const BlockSmall& b, int c0, int c1, int col0, int col1, int late1, bool inner, cudaStream_t st) SAGE_OPTIONAL;
// The kept rows after ncyc cycles as combinations of planes: T[t][j][p], t < 3, j < j_pad (the planes of the coefficients, pitch ldT), for
// p < P rounded up to 64; carried: the cycles behind which launch_block_step has been. The last cycle's factors have keep_last columns and its window r_last rows.
cudaError_t launch_block_factors(const BlockSmall& b, const BlockMap& map, int carried, int ncyc, int r_last, int keep_last, __nv_bfloat16* T, int j_pad, int64_t ldT,
                                 cudaStream_t st) SAGE_OPTIONAL;
// out[j] = sum_p (T[0] + T[1] + T[2])[j][p] plane_p for j < keep: as three planes a row (planes, pitch of the source) or in fp32
// (rows, pitch ldo, d < ldo).
cudaError_t launch_block_rebuild(const BlockSource& src, const BlockMap& map, int64_t D, const __nv_bfloat16* T, int j_pad, int64_t ldT, int keep,
                                 __nv_bfloat16* planes, float* rows, int64_t ldo, int* err, cudaStream_t st) SAGE_OPTIONAL;

// Hooks into the C ABI's bookkeeping for entry points defined outside api.cu.
void set_error_message(const char* msg);   // becomes the calling thread's sage_last_error()
void count_launches(int k);                // adds to sage_launch_count()

}  // namespace sage
