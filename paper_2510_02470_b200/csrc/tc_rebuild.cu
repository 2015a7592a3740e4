// Tensor-core rebuild of the sketch buffer (Method, first paragraph: the sketch is rebuilt from the shrunk singular values and the right factor).
// With B B^T = U Lambda U^T, Sigma' V^T = diag(sigma'_j / sigma_j) U^T B, i.e.
//     out[j][d] = sum_i W[j][i] * B[i][d],   W[j][i] = U[i][j] * sqrt(max(1 - delta/lambda_j, 0)).
// The buffer is the streamed operand: a CTA walks 128-column tiles of it, and for each tile accumulates over
// chunks of 32 buffer rows   D[d][j] += B[i][d] * W[j][i]   with d on the 128 TMEM lanes (the buffer tile is the
// "A" operand, stored with d contiguous = MN-major), so the epilogue writes out[j][d0..d0+127] as full lines.
//
// fp32 fidelity as in the Gram kernel: the tensor cores read a buffer value as hi (its low 13 bits ignored),
// the split warps write lo = x - hi into a second buffer; W arrives already split from global memory as two stacked operands [W_hi; W_lo],
// so one MMA of width 2*j_pad gives hi*W_hi and hi*W_lo side by side and a second one adds lo*W_hi; the
// epilogue adds the two halves. One TMEM accumulator takes at most 8 chunks (256 buffer rows) this way; more than 256 buffer rows
// or more than 128 output rows go to k_tc_rebuild_wide, factors that fit shared memory as a whole to k_tc_rebuild_narrow. Here:
//
//   warp 0    TMA producer: per chunk 4 boxes of [32 rows][32 columns] of the buffer (128-byte swizzle with
//             32-byte atoms, the only layout the tensor cores take for 32-bit MN-major operands) and one box of W,
//   warp 1    TMEM allocation, MMA issue into two ping-pong accumulators (one per column tile),
//   warps 2-5 write the lo part of the buffer tile of each landed stage,
//   warps 6-9 epilogue: TMEM -> registers -> out.
#include "sage_internal.h"
#include "tc05.cuh"

namespace sage {
namespace tc {
namespace {

constexpr int kThreads = 320;
constexpr int kSplitThreads = 128;
constexpr int kEpiThreads = 128;
constexpr int kTileD = 128;                 // buffer columns per tile (MMA M)
constexpr int kChunkRows = 32;              // buffer rows per stage (MMA K = 4 x 8)
constexpr int kBufBytes = kChunkRows * kTileD * 4;   // 16 KB: 4 spans of [32 rows][128 bytes]
constexpr int kSpanBytes = kChunkRows * 128;         // 4 KB

// The remainders of a landed chunk, by kSplitThreads threads.
__device__ __forceinline__ void split_chunk(const uint4* hi, uint4* lo, int t) {
#pragma unroll
    for (int cc = 0; cc < kBufBytes / 16 / kSplitThreads; ++cc) lo[t + cc * kSplitThreads] = remainder_tf32(hi[t + cc * kSplitThreads]);
}

__global__ void __launch_bounds__(kThreads, 1)
k_tc_rebuild(const __grid_constant__ CUtensorMap tmBuf, const __grid_constant__ CUtensorMap tmW, int r, int keep, int j_pad,
             long long pitch, long long num_tiles, float* __restrict__ out, int stages, int* __restrict__ err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    // stage layout: [buffer hi 16 KB][buffer lo 16 KB][W_hi ; W_lo: 2*j_pad rows of 128 bytes]
    const int w_bytes = 2 * j_pad * 128, stage_bytes = 2 * kBufBytes + w_bytes;
    const int nchunk = (r + kChunkRows - 1) / kChunkRows;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)stages * stage_bytes);
    uint64_t* split_done = full + stages;
    uint64_t* empty = split_done + stages;
    uint64_t* acc_full = empty + stages;                   // [2]
    uint64_t* acc_empty = acc_full + 2;                    // [2]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_mma = 2 * j_pad;                           // <= 256
    uint32_t tmem_cols = 32;
    while (tmem_cols < (uint32_t)(2 * n_mma)) tmem_cols <<= 1;
    // tiles of this CTA: blockIdx.x, blockIdx.x + gridDim.x, ...
    const long long my_tiles = num_tiles > blockIdx.x ? (num_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&split_done[s], kSplitThreads);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], kEpiThreads);
        }
        *abort = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmBuf);
        tma_prefetch_desc(&tmW);
    }
    if (warp == 1) tmem_alloc(tmem_slot, tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    chain_wait();

    if (warp == 0) {
        if (lane == 0) {
            long long issued = 0;
            bool alive = true;
            int s = 0;
            uint32_t ph = 1;                                // parity of the empty-barrier phase to wait for
            uint8_t* st = smem;
            for (long long lt = 0; lt < my_tiles && alive; ++lt) {
                const int d0 = (int)((blockIdx.x + lt * gridDim.x) * kTileD);
                for (int c = 0; c < nchunk; ++c) {
                    if (!mbar_wait(&empty[s], ph, abort)) { alive = false; break; }
                    mbar_expect_tx(&full[s], (uint32_t)(kBufBytes + w_bytes));
#pragma unroll
                    for (int sp = 0; sp < 4; ++sp) tma_load_2d(st + sp * kSpanBytes, &tmBuf, &full[s], d0 + 32 * sp, c * kChunkRows);
                    tma_load_2d(st + 2 * kBufBytes, &tmW, &full[s], c * kChunkRows, 0);
                    ++issued;
                    if (++s == stages) { s = 0; ph ^= 1u; st = smem; } else { st += stage_bytes; }
                }
            }
            if (*abort) {
                for (long long k = issued > stages ? issued - stages : 0; k < issued; ++k)
                    mbar_wait_quiet(&full[k % stages], (uint32_t)(k / stages) & 1u, 20000000ll);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc_fold = instr_desc(2, kTileD, n_mma, 1, 0);   // A (buffer) MN-major, B (W) K-major
            const uint32_t idesc_half = instr_desc(2, kTileD, j_pad, 1, 0);
            // running stage / phase counters and descriptors advanced by a constant per stage: the loop of the single issuing
            // thread bounds the kernel, so it holds no division and builds no descriptor from scratch
            const uint64_t desc_w = smem_desc_k_sw128(0), desc_buf = smem_desc_mn_sw128_atom32(0, kSpanBytes);
            const uint32_t st0 = smem_u32(smem);
            bool alive = true;
            int s = 0;
            uint32_t ph = 0, st = st0;
            for (long long lt = 0; lt < my_tiles && alive; ++lt) {
                const int b = (int)(lt & 1);
                const uint32_t par = (uint32_t)(lt >> 1);
                alive = mbar_wait(&acc_empty[b], (par & 1u) ^ 1u, abort);
                if (!alive) break;
                for (int c = 0; c < nchunk; ++c) {
                    const uint32_t acc = tmem_base + (uint32_t)(b * n_mma);
                    if (!mbar_wait(&split_done[s], ph, abort)) { alive = false; break; }
                    tc_fence_after();
                    const uint64_t d_w = desc_w | ((st + 2 * kBufBytes) >> 4);
                    const uint64_t d_hi = desc_buf | (st >> 4), d_lo = desc_buf | ((st + kBufBytes) >> 4);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {          // 8 buffer rows per MMA: one 1024-byte row group (64 descriptor units)
                        mma_tf32(acc, d_hi + 64 * k, d_w + 2 * k, idesc_fold, (c | k) != 0);   // hi*W_hi | hi*W_lo
                        mma_tf32(acc, d_lo + 64 * k, d_w + 2 * k, idesc_half, 1);     // + lo*W_hi
                    }
                    mma_commit(&empty[s]);
                    if (++s == stages) { s = 0; ph ^= 1u; st = st0; } else { st += (uint32_t)stage_bytes; }
                }
                if (alive) mma_commit(&acc_full[b]);
            }
        }
    } else if (warp < 6) {
        const int t = threadIdx.x - 64;
        const long long total = my_tiles * nchunk;
        int s = 0;
        uint32_t ph = 0;
        for (long long q = 0; q < total; ++q) {
            if (!mbar_wait(&full[s], ph, abort)) break;
            uint4* hi = reinterpret_cast<uint4*>(smem + (size_t)s * stage_bytes);
            split_chunk(hi, hi + kBufBytes / 16, t);
            fence_proxy_async_smem();
            mbar_arrive(&split_done[s]);
            if (++s == stages) { s = 0; ph ^= 1u; }
        }
    } else {
        const int quarter = warp & 3;
        const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        for (long long lt = 0; lt < my_tiles; ++lt) {
            const int b = (int)(lt & 1);
            const uint32_t par = (uint32_t)(lt >> 1);
            bool ok = mbar_wait(&acc_full[b], par & 1u, abort);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            if (lt == my_tiles - 1) chain_release();
            const long long d = (blockIdx.x + lt * gridDim.x) * kTileD + quarter * 32 + lane;
            const uint32_t acc = lane_base + (uint32_t)(b * n_mma);
            for (int j0 = 0; j0 < j_pad; j0 += 32) {
                // four TMEM loads in flight per wait (hi*W_hi | hi*W_lo halves of two groups of 16 output rows)
                const bool second = j0 + 16 < j_pad;
                uint32_t v0[16], w0[16], v1[16], w1[16];
                tmem_ld16_issue(acc + (uint32_t)j0, v0);
                tmem_ld16_issue(acc + (uint32_t)(j_pad + j0), w0);
                if (second) {
                    tmem_ld16_issue(acc + (uint32_t)(j0 + 16), v1);
                    tmem_ld16_issue(acc + (uint32_t)(j_pad + j0 + 16), w1);
                }
                tmem_ld_wait();
                tmem_ld_use(v0);
                tmem_ld_use(w0);
                float a0[16], a1[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) a0[j] = __uint_as_float(v0[j]) + __uint_as_float(w0[j]);
                if (second) {
                    tmem_ld_use(v1);
                    tmem_ld_use(w1);
#pragma unroll
                    for (int j = 0; j < 16; ++j) a1[j] = __uint_as_float(v1[j]) + __uint_as_float(w1[j]);
                }
                if (d < pitch) {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (j0 + j < keep) out[(long long)(j0 + j) * pitch + d] = a0[j];
                    if (second) {
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (j0 + 16 + j < keep) out[(long long)(j0 + 16 + j) * pitch + d] = a1[j];
                    }
                }
            }
            tc_fence_before();
            mbar_arrive(&acc_empty[b]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        if (my_tiles > 0 && !*abort)
            mbar_wait_quiet(&acc_full[(my_tiles - 1) & 1], (uint32_t)((my_tiles - 1) >> 1) & 1u, kWaitLimitCycles);
        tc_fence_after();
        tmem_dealloc(tmem_base, tmem_cols);
    }
    if (threadIdx.x == 0 && *abort) atomicExch(err, 1);
}

// Up to 64 output rows whose factors, all chunks of them, take 64 KB (up to 128 buffer rows): they are loaded once and stay, and the
// remainders go to TMEM, as the A operand of the second product, instead of shared memory: no store and no proxy fence for the split,
// and a stage is the landed chunk alone, so that eight are in flight.
// direct_new > 0: the last direct_new of the r rows are bfloat16 rows in the caller's memory. Row r - direct_new is the last row of its
// chunk (cb), which gets one bfloat16 row (tmSrc1) in place of a placeholder; the chunks after it are 32 of them each (tmSrc). These
// go to TMEM as they are: their remainders are zero, one product is all.
//   warp 0 loads, warp 1 issues MMAs, warps 2-9 write remainders in two groups in turn (thread = buffer column), warps 10-13 are the epilogue.
// 128 rows of 11.2 M columns onto 63, half of them read in place: 1,600 -> 1,533 us against remainders in shared memory and four chunks in
// flight; of 262,144 columns 49 -> 47 us; short rows equal. That is 7.1 GB at 4.6 TB/s, 0.70 of the copy rate, and nothing on the
// chip is near its limit (tensor pipe 28 %, shared memory 31 %, DRAM 50 % of nominal): what holds it there is not known.
constexpr int kNarrowThreads = 448;
constexpr int kSlots = 8;                   // chunks in shared memory and, their remainders, in TMEM
constexpr int kSlotBytes = kBufBytes + 1024;          // 16 KB of fp32 rows or 8 KB of bfloat16 rows, and the one bfloat16 row of chunk cb
constexpr int kResidentBytes = 64 * 1024;
constexpr uint32_t kLoCols = 256;           // TMEM: two accumulators of up to 128 columns, then the remainders, 32 columns each
constexpr size_t kNarrowSmem = 1024 + (size_t)kSlots * kSlotBytes + kResidentBytes + (3 * kSlots + 5) * 8 + 16;

__global__ void __launch_bounds__(kNarrowThreads, 1)
k_tc_rebuild_narrow(const __grid_constant__ CUtensorMap tmBuf, const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmSrc,
                    const __grid_constant__ CUtensorMap tmSrc1, int direct_new, int r, int keep, int j_pad, long long pitch, long long num_tiles,
                    float* __restrict__ out, int* __restrict__ err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint8_t* wres = smem + kSlots * kSlotBytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(wres + kResidentBytes);
    uint64_t* split_done = full + kSlots;
    uint64_t* empty = split_done + kSlots;
    uint64_t* acc_full = empty + kSlots;                   // [2]
    uint64_t* acc_empty = acc_full + 2;                    // [2]
    uint64_t* w_full = acc_empty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(w_full + 1);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int w_bytes = 2 * j_pad * 128, n_mma = 2 * j_pad;           // n_mma <= 128
    const int nchunk = (r + kChunkRows - 1) / kChunkRows;
    const int cb = direct_new ? (r - direct_new) / kChunkRows : 1 << 30;
    const long long my_tiles = num_tiles > blockIdx.x ? (num_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kSlots; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&split_done[s], 4);
            mbar_init(&empty[s], 1);
        }
        mbar_init(w_full, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], kEpiThreads);
        }
        *abort = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmBuf);
        tma_prefetch_desc(&tmW);
    }
    if (warp == 1) tmem_alloc(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    chain_wait();

    if (warp == 0) {
        if (lane == 0) {
            long long issued = 0;
            bool alive = true;
            int s = 0;
            uint32_t ph = 1;
            mbar_expect_tx(w_full, (uint32_t)(nchunk * w_bytes));
            for (int c = 0; c < nchunk; ++c) tma_load_2d(wres + (size_t)c * w_bytes, &tmW, w_full, c * kChunkRows, 0);
            for (long long lt = 0; lt < my_tiles && alive; ++lt) {
                const int d0 = (int)((blockIdx.x + lt * gridDim.x) * kTileD);
                for (int c = 0; c < nchunk; ++c) {
                    if (!mbar_wait(&empty[s], ph, abort)) { alive = false; break; }
                    uint8_t* st = smem + (size_t)s * kSlotBytes;
                    if (c > cb) {                               // caller's rows only
                        mbar_expect_tx(&full[s], 8192u);
                        tma_load_2d(st, &tmSrc, &full[s], d0, 1 + (c - cb - 1) * kChunkRows);
                    } else {
                        mbar_expect_tx(&full[s], (uint32_t)(c == cb ? kBufBytes + 256 : kBufBytes));
#pragma unroll
                        for (int sp = 0; sp < 4; ++sp) tma_load_2d(st + sp * kSpanBytes, &tmBuf, &full[s], d0 + 32 * sp, c * kChunkRows);
                        if (c == cb) tma_load_2d(st + kBufBytes, &tmSrc1, &full[s], d0, 0);
                    }
                    ++issued;
                    if (++s == kSlots) { s = 0; ph ^= 1u; }
                }
            }
            if (*abort) {
                mbar_wait_quiet(w_full, 0, 20000000ll);
                for (long long k = issued > kSlots ? issued - kSlots : 0; k < issued; ++k)
                    mbar_wait_quiet(&full[k % kSlots], (uint32_t)(k / kSlots) & 1u, 20000000ll);
            }
        }
    } else if (warp == 1) {
        const uint32_t idesc_hi = instr_desc(2, kTileD, n_mma, 1, 0), idesc_lo = instr_desc(2, kTileD, j_pad, 0, 0);
        const uint32_t idesc_new = instr_desc(2, kTileD, n_mma, 0, 0);
        const uint64_t desc_w = smem_desc_k_sw128(0), desc_buf = smem_desc_mn_sw128_atom32(0, kSpanBytes);
        const uint32_t st0 = smem_u32(smem), w0 = smem_u32(wres);
        int s = 0;
        uint32_t ph = 0;
        bool alive = __all_sync(0xffffffffu, mbar_wait(w_full, 0, abort));
        for (long long lt = 0; lt < my_tiles && alive; ++lt) {
            const uint32_t b = (uint32_t)(lt & 1), acc = tmem_base + b * 128u;
            alive = __all_sync(0xffffffffu, mbar_wait(&acc_empty[b], ((uint32_t)(lt >> 1) & 1u) ^ 1u, abort));
            for (int c = 0; c < nchunk && alive; ++c) {
                alive = __all_sync(0xffffffffu, mbar_wait(&split_done[s], ph, abort));
                if (!alive) break;
                tc_fence_after();
                const uint64_t d_w = desc_w | ((w0 + (uint32_t)(c * w_bytes)) >> 4), d_hi = desc_buf | ((st0 + (uint32_t)(s * kSlotBytes)) >> 4);
                const uint32_t lo = tmem_base + kLoCols + (uint32_t)(s * 32);
                if (elect_one()) {
                    if (c > cb) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) mma_tf32_ts(acc, lo + 8 * k, d_w + 2 * k, idesc_new, 1);
                    } else {
#pragma unroll
                        for (int k = 0; k < 4; ++k) {      // 8 buffer rows per MMA: one 1024-byte row group (64 descriptor units)
                            mma_tf32(acc, d_hi + 64 * k, d_w + 2 * k, idesc_hi, (c | k) != 0);        // hi*W_hi | hi*W_lo
                            mma_tf32_ts(acc, lo + 8 * k, d_w + 2 * k, idesc_lo, 1);                    // + lo*W_hi
                        }
                    }
                    mma_commit(&empty[s]);
                    if (c == nchunk - 1) mma_commit(&acc_full[b]);
                }
                __syncwarp();
                if (++s == kSlots) { s = 0; ph ^= 1u; }
            }
        }
    } else if (warp < 10) {
        const int quarter = warp & 3, grp = (warp - 2) >> 2;
        const uint32_t dst = tmem_base + kLoCols + (static_cast<uint32_t>(quarter * 32) << 16);
        const int span = quarter * kSpanBytes;                              // this warp's 32 columns of a chunk of fp32 rows
        const int piece = lane >> 3, in_piece = lane & 7;                   // 32-byte piece of a row (permuted by the row), float in it
        const long long total = my_tiles * nchunk;
        int c = grp % nchunk;
        for (long long g = grp; g < total; g += 2) {                        // kSlots is even: a group sees every phase of its slots
            const int s = (int)(g % kSlots);
            bool ok = mbar_wait(&full[s], (uint32_t)(g / kSlots) & 1u, abort);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();                   // loaded after the MMAs of eight chunks ago: the columns of its remainders are free, too
            uint8_t* st = smem + (size_t)s * kSlotBytes;
            uint32_t v[32];
            if (c > cb) {
                const uint16_t* src = reinterpret_cast<const uint16_t*>(st) + quarter * 32 + lane;
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = (uint32_t)src[i * kTileD] << 16;
            } else {
                float* hi = reinterpret_cast<float*>(st + span);
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = remainder_tf32(__float_as_uint(hi[i * 32 + ((piece ^ (i & 3)) << 3) + in_piece]));
                if (c == cb) {                  // the caller's first row takes the placeholder's place
                    const uint32_t x = (uint32_t)reinterpret_cast<const uint16_t*>(st + kBufBytes)[quarter * 32 + lane] << 16;
                    hi[31 * 32 + ((piece ^ 3) << 3) + in_piece] = __uint_as_float(x);
                    v[31] = 0u;
                    fence_proxy_async_smem();
                }
            }
            tmem_st32(dst + (uint32_t)(s * 32), v);
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&split_done[s]);
            c += 2;
            while (c >= nchunk) c -= nchunk;
        }
    } else {
        const int quarter = warp & 3;
        const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        for (long long lt = 0; lt < my_tiles; ++lt) {
            const uint32_t b = (uint32_t)(lt & 1);
            const bool ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[b], (uint32_t)(lt >> 1) & 1u, abort));
            if (!ok) break;
            tc_fence_after();
            if (lt == my_tiles - 1) chain_release();
            const long long d = (blockIdx.x + lt * gridDim.x) * kTileD + quarter * 32 + lane;
            const uint32_t acc = lane_base + b * 128u;
            for (int j0 = 0; j0 < j_pad; j0 += 16) {
                uint32_t v0[16], w0[16];
                tmem_ld16_issue(acc + (uint32_t)j0, v0);
                tmem_ld16_issue(acc + (uint32_t)(j_pad + j0), w0);
                tmem_ld_wait();
                tmem_ld_use(v0);
                tmem_ld_use(w0);
                if (d < pitch) {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (j0 + j < keep) out[(long long)(j0 + j) * pitch + d] = __uint_as_float(v0[j]) + __uint_as_float(w0[j]);
                }
            }
            tc_fence_before();
            mbar_arrive(&acc_empty[b]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        if (my_tiles > 0 && !*abort)
            mbar_wait_quiet(&acc_full[(my_tiles - 1) & 1], (uint32_t)((my_tiles - 1) >> 1) & 1u, kWaitLimitCycles);
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
    if (threadIdx.x == 0 && *abort) atomicExch(err, 1);
}

// More than 256 buffer rows or more than 128 output rows (up to 512 onto 256): a tile's buffer data is loaded once for all output
// rows. A chunk costs 12 MMAs of width j_pad (hi*W_hi, lo*W_hi and hi*W_lo for its 4 steps of 8 rows) that add into ONE accumulator
// of j_pad columns, so that two of them fit TMEM and one is drained while the other fills. A run of kRunChunks chunks makes 60
// additions to an accumulator, where the narrow kernel makes 64; the epilogue keeps the sums of a tile's runs in registers
// (128 a thread, hence the register split below).
// A chunk's factors are four times its buffer data, and come out of the L2 cache: they have a ring of their own, whose slots (hi
// and lo apart) are shorter-lived than the buffer's, and whose loads do not wait for buffer data.
//   warp 0 loads buffer chunks, warp 1 issues MMAs, warp 2 loads factors, warps 4-7 write the lo parts, warps 8-15 are the
//   epilogue (8-11: output rows 0-127, 12-15: the others).
// 512 rows onto 255, 262,144 columns: 422 -> 282 us (two launches of the narrow kernel, each over the whole buffer, before: their
// loads and hand-offs alone took 344 us). The tensor pipe is busy 80 % of that; loads (80 KB a chunk, 34 bytes a cycle) and shared
// memory (60 %) are not far behind.
constexpr int kWideThreads = 512;
constexpr int kWideRegs = 128;              // what every thread is launched with: the sum of the shares below is 4 x 128 x 128
constexpr int kBufStages = 3, kWSlots = 4;
constexpr int kWSlotBytes = 256 * 128;      // [256 output rows][32 buffer rows] of W_hi or W_lo
constexpr int kRunChunks = 5;
constexpr size_t kWideSmem = 1024 + (size_t)kBufStages * 2 * kBufBytes + (size_t)kWSlots * kWSlotBytes + (3 * kBufStages + 2 * kWSlots + 4) * 8 + 16;

__global__ void __launch_bounds__(kWideThreads, 1)
k_tc_rebuild_wide(const __grid_constant__ CUtensorMap tmBuf, const __grid_constant__ CUtensorMap tmW, int r, int keep, int j_pad, int lo_row,
                  long long pitch, long long num_tiles, float* __restrict__ out, int* __restrict__ err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint8_t* wring = smem + kBufStages * 2 * kBufBytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(wring + kWSlots * kWSlotBytes);
    uint64_t* split_done = full + kBufStages;
    uint64_t* empty = split_done + kBufStages;
    uint64_t* w_full = empty + kBufStages;
    uint64_t* w_empty = w_full + kWSlots;
    uint64_t* acc_full = w_empty + kWSlots;                // [2]
    uint64_t* acc_empty = acc_full + 2;                    // [2]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int halves = j_pad > 128 ? 2 : 1;
    const int nchunk = (r + kChunkRows - 1) / kChunkRows;
    const int nruns = (nchunk + kRunChunks - 1) / kRunChunks, run_len = (nchunk + nruns - 1) / nruns;
    // every run has at least one chunk: nchunk <= 16 gives runs of 1 to 5, ceil(nchunk / run_len) == nruns for all of them
    const long long my_tiles = num_tiles > blockIdx.x ? (num_tiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kBufStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&split_done[s], kSplitThreads);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < kWSlots; ++s) {
            mbar_init(&w_full[s], 1);
            mbar_init(&w_empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 128 * halves);
        }
        *abort = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmBuf);
        tma_prefetch_desc(&tmW);
    }
    if (warp == 1) tmem_alloc(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    chain_wait();

    if (warp < 8) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
        if (warp == 0) {
            if (lane == 0) {
                long long issued = 0;
                bool alive = true;
                int s = 0;
                uint32_t ph = 1;
                for (long long lt = 0; lt < my_tiles && alive; ++lt) {
                    const int d0 = (int)((blockIdx.x + lt * gridDim.x) * kTileD);
                    for (int c = 0; c < nchunk; ++c) {
                        if (!mbar_wait(&empty[s], ph, abort)) { alive = false; break; }
                        uint8_t* st = smem + (size_t)s * 2 * kBufBytes;
                        mbar_expect_tx(&full[s], (uint32_t)kBufBytes);
#pragma unroll
                        for (int sp = 0; sp < 4; ++sp) tma_load_2d(st + sp * kSpanBytes, &tmBuf, &full[s], d0 + 32 * sp, c * kChunkRows);
                        ++issued;
                        if (++s == kBufStages) { s = 0; ph ^= 1u; }
                    }
                }
                if (*abort)
                    for (long long k = issued > kBufStages ? issued - kBufStages : 0; k < issued; ++k)
                        mbar_wait_quiet(&full[k % kBufStages], (uint32_t)(k / kBufStages) & 1u, 20000000ll);
            }
        } else if (warp == 2) {
            if (lane == 0) {
                long long issued = 0;
                bool alive = true;
                int s = 0;
                uint32_t ph = 1;
                for (long long lt = 0; lt < my_tiles && alive; ++lt)
                    for (int c = 0; c < nchunk && alive; ++c)
                        for (int part = 0; part < 2; ++part) {
                            if (!mbar_wait(&w_empty[s], ph, abort)) { alive = false; break; }
                            uint8_t* dst = wring + (size_t)s * kWSlotBytes;
                            mbar_expect_tx(&w_full[s], (uint32_t)(halves * 128 * 128));
                            for (int q = 0; q < halves; ++q)
                                tma_load_2d(dst + q * 128 * 128, &tmW, &w_full[s], c * kChunkRows, q * 256 + part * lo_row);
                            ++issued;
                            if (++s == kWSlots) { s = 0; ph ^= 1u; }
                        }
                if (*abort)
                    for (long long k = issued > kWSlots ? issued - kWSlots : 0; k < issued; ++k)
                        mbar_wait_quiet(&w_full[k % kWSlots], (uint32_t)(k / kWSlots) & 1u, 20000000ll);
            }
        } else if (warp == 1) {
            if (lane == 0) {
                const uint32_t idesc = instr_desc(2, kTileD, j_pad, 1, 0);                // A (buffer) MN-major, B (W) K-major
                const uint64_t desc_w = smem_desc_k_sw128(0), desc_buf = smem_desc_mn_sw128_atom32(0, kSpanBytes);
                const uint32_t st0 = smem_u32(smem), w0 = smem_u32(wring);
                bool alive = true;
                int s = 0, ws = 0;
                uint32_t ph = 0, wph = 0, run = 0;
                for (long long lt = 0; lt < my_tiles && alive; ++lt) {
                    for (int c0 = 0; c0 < nchunk && alive; c0 += run_len, ++run) {
                        const int c1 = c0 + run_len < nchunk ? c0 + run_len : nchunk;
                        const uint32_t b = run & 1u, acc = tmem_base + b * 256u;
                        alive = mbar_wait(&acc_empty[b], ((run >> 1) & 1u) ^ 1u, abort);
                        for (int c = c0; c < c1 && alive; ++c) {
                            alive = mbar_wait(&w_full[ws], wph, abort) && mbar_wait(&split_done[s], ph, abort);
                            if (!alive) break;
                            tc_fence_after();
                            const uint32_t st = st0 + (uint32_t)(s * 2 * kBufBytes);
                            const uint64_t d_hi = desc_buf | (st >> 4), d_lo = desc_buf | ((st + kBufBytes) >> 4);
                            uint64_t d_w = desc_w | ((w0 + (uint32_t)(ws * kWSlotBytes)) >> 4);
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                mma_tf32(acc, d_hi + 64 * k, d_w + 2 * k, idesc, c != c0 || k != 0);
                                mma_tf32(acc, d_lo + 64 * k, d_w + 2 * k, idesc, 1);
                            }
                            mma_commit(&w_empty[ws]);
                            if (++ws == kWSlots) { ws = 0; wph ^= 1u; }
                            alive = mbar_wait(&w_full[ws], wph, abort);
                            if (!alive) break;
                            tc_fence_after();
                            d_w = desc_w | ((w0 + (uint32_t)(ws * kWSlotBytes)) >> 4);
#pragma unroll
                            for (int k = 0; k < 4; ++k) mma_tf32(acc, d_hi + 64 * k, d_w + 2 * k, idesc, 1);
                            mma_commit(&w_empty[ws]);
                            mma_commit(&empty[s]);
                            if (++ws == kWSlots) { ws = 0; wph ^= 1u; }
                            if (++s == kBufStages) { s = 0; ph ^= 1u; }
                        }
                        if (alive) mma_commit(&acc_full[b]);
                    }
                }
            }
        } else if (warp >= 4) {
            const int t = threadIdx.x - 128;
            const long long total = my_tiles * nchunk;
            int s = 0;
            uint32_t ph = 0;
            for (long long q = 0; q < total; ++q) {
                if (!mbar_wait(&full[s], ph, abort)) break;
                uint4* hi = reinterpret_cast<uint4*>(smem + (size_t)s * 2 * kBufBytes);
                split_chunk(hi, hi + kBufBytes / 16, t);
                fence_proxy_async_smem();
                mbar_arrive(&split_done[s]);
                if (++s == kBufStages) { s = 0; ph ^= 1u; }
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 184;");
        const int quarter = warp & 3, half = (warp - 8) >> 2;
        if (half < halves) {
            const int j_n = j_pad - half * 128 < 128 ? j_pad - half * 128 : 128;         // output rows of this half, a multiple of 16
            const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + (uint32_t)(half * 128);
            uint32_t run = 0;
            bool ok = true;
            for (long long lt = 0; lt < my_tiles && ok; ++lt) {
                float sum[128];
#pragma unroll
                for (int j = 0; j < 128; ++j) sum[j] = 0.f;
                for (int g = 0; g < nruns; ++g, ++run) {
                    const uint32_t b = run & 1u;
                    ok = mbar_wait(&acc_full[b], (run >> 1) & 1u, abort);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    tc_fence_after();
                    if (lt == my_tiles - 1 && g == nruns - 1) chain_release();
#pragma unroll
                    for (int j0 = 0; j0 < 128; j0 += 32) {
                        if (j0 < j_n) {                     // the upper 16 columns of the last group may lie beyond j_n: added, never stored
                            uint32_t v0[16], v1[16];
                            tmem_ld16_issue(lane_base + b * 256u + (uint32_t)j0, v0);
                            tmem_ld16_issue(lane_base + b * 256u + (uint32_t)(j0 + 16), v1);
                            tmem_ld_wait();
                            tmem_ld_use(v0);
                            tmem_ld_use(v1);
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                sum[j0 + j] += __uint_as_float(v0[j]);
                                sum[j0 + 16 + j] += __uint_as_float(v1[j]);
                            }
                        }
                    }
                    tc_fence_before();
                    mbar_arrive(&acc_empty[b]);
                }
                const long long d = (blockIdx.x + lt * gridDim.x) * kTileD + quarter * 32 + lane;
                if (ok && d < pitch) {
                    float* o = out + (long long)(half * 128) * pitch + d;
#pragma unroll
                    for (int j = 0; j < 128; ++j, o += pitch)
                        if (half * 128 + j < keep) *o = sum[j];
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        if (my_tiles > 0 && !*abort) {
            const long long last = my_tiles * nruns - 1;
            mbar_wait_quiet(&acc_full[last & 1], (uint32_t)(last >> 1) & 1u, kWaitLimitCycles);
        }
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
    if (threadIdx.x == 0 && *abort) atomicExch(err, 1);
}

}  // namespace
}  // namespace tc

// See sage_internal.h.
static cudaError_t launch_tc_rebuild_part(const float* Wsplit, int ldw, int j_pad, const float* Bsrc, float* Bdst, int64_t pitch, int r,
                                          int keep, int* err, cudaStream_t st, const void* src = nullptr, int64_t ld_src = 0, int n_new = 0,
                                          int64_t D = 0) {
    if (keep <= 0 || r <= 0) return cudaSuccess;
    if (j_pad < 16 || j_pad > 128 || (j_pad & 15) || keep > j_pad || r > 256) return cudaErrorNotSupported;
    CUtensorMap tmBuf, tmW;
    // buffer: columns beyond D up to the pitch are zero and are rebuilt as zero, so the map spans the pitch
    // direct form (src != nullptr): only the rows that are in the buffer, plus the placeholder row, are addressable
    if (!tc::make_tmap_2d(&tmBuf, Bsrc, 4, (uint64_t)(src ? r - n_new + 1 : r), (uint64_t)pitch, (uint64_t)pitch, tc::kChunkRows, 1))
        return cudaErrorNotSupported;
    const int kcols = ((r + tc::kChunkRows - 1) / tc::kChunkRows) * tc::kChunkRows;
    if (kcols > ldw) return cudaErrorNotSupported;
    if (!tc::make_tmap_2d(&tmW, Wsplit, 4, (uint64_t)(2 * j_pad), (uint64_t)kcols, (uint64_t)ldw, (uint32_t)(2 * j_pad)))
        return cudaErrorNotSupported;
    const long long num_tiles = (pitch + tc::kTileD - 1) / tc::kTileD;
    const int grid = (int)(num_tiles < 148 ? num_tiles : 148);
    const int nchunk = kcols / tc::kChunkRows;
    if (j_pad <= 64 && nchunk * 2 * j_pad * 128 <= tc::kResidentBytes) {
        CUtensorMap tmSrc = tmW, tmSrc1 = tmW;
        if (src) {
            if (n_new < 2 || n_new >= r || (r - n_new + 1) % tc::kChunkRows != 0 || r % tc::kChunkRows != 0) return cudaErrorNotSupported;
            if (!tc::make_tmap_2d_plain(&tmSrc, src, 2, (uint64_t)n_new, (uint64_t)D, (uint64_t)ld_src, 128, (uint32_t)tc::kChunkRows) ||
                !tc::make_tmap_2d_plain(&tmSrc1, src, 2, (uint64_t)n_new, (uint64_t)D, (uint64_t)ld_src, 128, 1))
                return cudaErrorNotSupported;
        }
        cudaError_t e = allow_smem((const void*)tc::k_tc_rebuild_narrow, 227 * 1024);
        if (e != cudaSuccess) return e;
        return launch_chained(tc::k_tc_rebuild_narrow, dim3(grid), dim3(tc::kNarrowThreads), tc::kNarrowSmem, st, tmBuf, tmW, tmSrc, tmSrc1,
                              src ? n_new : 0, r, keep, j_pad, pitch, num_tiles, Bdst, err);
    }
    if (src) return cudaErrorNotSupported;
    const int stage_bytes = 2 * tc::kBufBytes + 2 * j_pad * 128;
    int stages = (227 * 1024 - 1536) / stage_bytes;
    if (stages > 8) stages = 8;
    const size_t smem = (size_t)stages * stage_bytes + 1024 + (3 * stages + 4) * 8 + 16;
    cudaError_t e = allow_smem((const void*)tc::k_tc_rebuild, 227 * 1024);
    if (e != cudaSuccess) return e;
    return launch_chained(tc::k_tc_rebuild, dim3(grid), dim3(tc::kThreads), smem, st, tmBuf, tmW, r, keep, j_pad, pitch, num_tiles, Bdst, stages, err);
}

static cudaError_t launch_tc_rebuild_wide(const float* Wsplit, int ldw, int j_pad, const float* Bsrc, float* Bdst, int64_t pitch, int r, int keep,
                                          int* err, cudaStream_t st) {
    const int kcols = ((r + tc::kChunkRows - 1) / tc::kChunkRows) * tc::kChunkRows;
    const int rows = j_pad > 128 ? 512 : 256;              // W rows: [hi ; lo] of 128 output rows, twice, or of j_pad <= 128
    if (kcols > ldw || rows > ldw) return cudaErrorNotSupported;
    CUtensorMap tmBuf, tmW;
    if (!tc::make_tmap_2d(&tmBuf, Bsrc, 4, (uint64_t)r, (uint64_t)pitch, (uint64_t)pitch, tc::kChunkRows, 1) ||
        !tc::make_tmap_2d(&tmW, Wsplit, 4, (uint64_t)rows, (uint64_t)kcols, (uint64_t)ldw, 128))
        return cudaErrorNotSupported;
    const cudaError_t e = allow_smem((const void*)tc::k_tc_rebuild_wide, 227 * 1024, tc::kWideRegs);
    if (e != cudaSuccess) return e;
    const long long num_tiles = (pitch + tc::kTileD - 1) / tc::kTileD;
    return launch_chained(tc::k_tc_rebuild_wide, dim3((int)(num_tiles < 148 ? num_tiles : 148)), dim3(tc::kWideThreads), tc::kWideSmem, st, tmBuf, tmW,
                          r, keep, j_pad, j_pad > 128 ? 128 : j_pad, pitch, num_tiles, Bdst, err);
}

// See sage_internal.h.
cudaError_t launch_tc_rebuild(const float* Wsplit, int ldw, int j_pad, const float* Bsrc, float* Bdst, int64_t pitch, int64_t D, int r,
                              int keep, int* err, cudaStream_t st) {
    (void)D;
    if (keep <= 0 || r <= 0) return cudaSuccess;
    if (j_pad < 16 || j_pad > 256 || (j_pad & 15) || keep > j_pad || r > 512) return cudaErrorNotSupported;
    if (r > 256 || j_pad > 128) return launch_tc_rebuild_wide(Wsplit, ldw, j_pad, Bsrc, Bdst, pitch, r, keep, err, st);
    return launch_tc_rebuild_part(Wsplit, ldw, j_pad, Bsrc, Bdst, pitch, r, keep, err, st);
}

// See sage_internal.h.
cudaError_t launch_tc_rebuild_direct(const float* Wsplit, int ldw, int j_pad, const float* Bsrc, float* Bdst, int64_t pitch, int64_t D,
                                     int r, int keep, const void* src, int64_t ld_src, int n_new, int* err, cudaStream_t st) {
    if (keep <= 0 || r <= 0 || !src) return cudaErrorNotSupported;
    if (j_pad < 16 || j_pad > 128 || (j_pad & 15) || keep > j_pad || r > 128) return cudaErrorNotSupported;
    return launch_tc_rebuild_part(Wsplit, ldw, j_pad, Bsrc, Bdst, pitch, r, keep, err, st, src, ld_src, n_new, D);
}

}  // namespace sage
