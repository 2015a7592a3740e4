// Gram matrix K = B B^T of a buffer of more than 128 rows (up to 512) on pairs of SMs: the same fp32-faithful contraction as
// tc_gemm_x3.cu (hi = x read with its low 13 bits ignored, lo = the remainder; hi*hi + hi*lo + lo*hi, an accumulator drained every
// kRunTiles K tiles into registers), with 256 x 256 output tiles on and above the diagonal. On the diagonal a tile holds
// T = hi*hi + hi*(2 lo), two products of the three: (T + T^T) / 2, formed by the reduction, is the sum of all (the doubling is exact).
// A 128 x 128 MMA of one SM reads 64 bytes of shared memory per cycle and operand, all that shared memory can give, and every
// K tile has to be written and split besides: that bounded the kernel. Of a pair's 256 x 256 x 8 MMA each SM holds half of the
// A rows and half of the B rows, reads 64 bytes per cycle in all, and splits what it holds; on diagonal tiles the two halves are the
// same rows. Per K tile and SM: 64 KB (diagonal) or 96 KB read by MMAs, 48 or 96 KB by loads and split, in the 1,020 or 1,540 cycles
// that its 8 or 12 MMAs take at the nominal rate.
// Measured (this kernel alone, against 128 x 128 tiles on single SMs): 512 rows of 262,144 columns 628 -> 310 us, 256 of them
// 239 -> 104 us, 256 rows of 51,300 columns 60 -> 35 us. 6 and 3 % of that are the release at cluster scope behind CTA 1's remainders
// (two warps in turn pass them on; one warp: 12 %). The MMAs bound it: the tensor pipe is busy 82 % of the time (512 rows).
// One cluster of two CTAs owns a tile and a K slice. CTA q: rows q*128 .. of the tile's row block (A, and its rows of the output) and
// rows q*128 .. of its column block (B).
//   warp 0     TMA loads of this CTA's rows (128-byte swizzle),
//   warp 1     TMEM allocation; in CTA 0 the MMAs of both, into two accumulators of 256 columns in turn,
//   warps 2, 3 of CTA 1 pass on to CTA 0 which remainders are written,
//   warps 4-11 write the remainders of landed stages; between stages they drain this CTA's accumulator rows
//              (4-7: columns 0-127, 8-11: the others) into 128 sums a thread, and store them at the end.
#include "sage_internal.h"
#include "tc05.cuh"

namespace sage {
namespace tc {
namespace {

constexpr int kPairThreads = 384;
constexpr int kPairRegs = 168;              // what every thread is launched with: the shares below add up to 3 x 128 x 168
constexpr int kPairWorkers = 8;             // warps
constexpr int kOpBytes = 128 * 128;         // 128 rows of one K tile (32 floats)
constexpr int kPairBK = 32;
constexpr int kRunTiles = 8;                // as tc_gemm_x3.cu: 96 additions between drains
// Two rings of operand tiles: landed data (hi) is held from the request of a load to the MMAs, remainders (lo) only from the split on. A
// stage is one tile on diagonal tiles, [A][B] elsewhere: 8 and 6 stages there, 4 and 3 here. The workers take diagonal stages in two
// groups in turn, others together: 8 pieces of 16 bytes a thread either way, all in flight at once.
constexpr int kHiTiles = 8, kLoTiles = 6;
constexpr size_t kPairSmem = 1024 + (size_t)(kHiTiles + kLoTiles) * kOpBytes + (2 * kHiTiles + 2 * kLoTiles + 4) * 8 + 16;

__global__ void __launch_bounds__(kPairThreads, 1)
k_tc_gram_pair(const __grid_constant__ CUtensorMap tm, int r, long long K, int n_diag, int n_off, float* __restrict__ C, long long ldc,
               long long split_stride, int* __restrict__ err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int q = blockIdx.x & 1, pair = blockIdx.x >> 1;           // CTA of the pair, and which pair: the slices of tile (0,1), then
    const bool diag = pair >= n_off;                                // those of (0,0) and, with it, of (1,1) in turn
    const int slice = diag ? (n_off ? (pair - n_off) >> 1 : pair) : pair;
    const int n0 = !diag || (n_off && ((pair - n_off) & 1)) ? 256 : 0, m0 = diag ? n0 : 0;
    const int stage_bytes = diag ? kOpBytes : 2 * kOpBytes;
    const int n_hi = diag ? kHiTiles : kHiTiles / 2, n_lo = diag ? kLoTiles : kLoTiles / 2, groups = diag ? 2 : 1;
    uint8_t* lo_ring = smem + kHiTiles * kOpBytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(lo_ring + kLoTiles * kOpBytes);   // [kHiTiles], local
    uint64_t* empty = full + kHiTiles;                                  // [kHiTiles], both CTAs': the MMA thread's commits go to both
    uint64_t* split_done = empty + kHiTiles;                            // [kLoTiles], local
    uint64_t* peer_split = split_done + kLoTiles;                       // [kLoTiles], CTA 0's: CTA 1's split_done, passed on
    uint64_t* acc_full = peer_split + kLoTiles;                         // [2], both CTAs'
    uint64_t* acc_empty = acc_full + 2;                                 // [2], CTA 0's: arrivals from both CTAs
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long kt_all = (K + kPairBK - 1) / kPairBK, n_slices = diag ? n_diag : n_off;
    const long long k_begin = kt_all * slice / n_slices * kPairBK;
    const int nkt = (int)(kt_all * (slice + 1) / n_slices - kt_all * slice / n_slices);
    const int nruns = (nkt + kRunTiles - 1) / kRunTiles;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kHiTiles; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < kLoTiles; ++s) {
            mbar_init(&split_done[s], kPairWorkers / groups);
            mbar_init(&peer_split[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 2 * kPairWorkers);
        }
        *abort = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tm);
    }
    if (warp == 1) tmem_alloc_pair(tmem_slot, 512);
    tc_fence_before();
    cluster_barrier();                          // the other CTA's barriers are set up, too
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    chain_wait();

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
        if (warp == 0) {
            if (lane == 0) {
                int issued = 0, s = 0, x = (int)k_begin;
                uint32_t ph = 1;
                for (int kt = 0; kt < nkt; ++kt, x += kPairBK) {
                    if (!mbar_wait(&empty[s], ph, abort)) break;
                    uint8_t* st = smem + (size_t)s * stage_bytes;
                    mbar_expect_tx(&full[s], (uint32_t)stage_bytes);
                    tma_load_2d(st, &tm, &full[s], x, m0 + q * 128);
                    if (!diag) tma_load_2d(st + kOpBytes, &tm, &full[s], x, n0 + q * 128);
                    issued = kt + 1;
                    if (++s == n_hi) { s = 0; ph ^= 1u; }
                }
                if (*abort)
                    for (int kt = issued > n_hi ? issued - n_hi : 0; kt < issued; ++kt)
                        mbar_wait_quiet(&full[kt % n_hi], (uint32_t)(kt / n_hi) & 1u, 20000000ll);
            }
        } else if (warp == 1) {
            if (q == 0) {                                   // the whole warp walks the loop, so that its values stay in uniform registers
                const uint32_t idesc = instr_desc(2, 256, 256, 0, 0);
                const uint64_t desc = smem_desc_k_sw128(0);
                const uint32_t hi0 = smem_u32(smem), lo0 = smem_u32(lo_ring), b_off = diag ? 0u : (uint32_t)kOpBytes;
                bool alive = true;
                int s = 0, ls = 0;
                uint32_t ph = 0;                            // a K tile's remainders are there: so is its data
                for (int kt = 0, run = 0; kt < nkt && alive; ++run) {
                    const int kt_end = kt + kRunTiles < nkt ? kt + kRunTiles : nkt;
                    const uint32_t b = (uint32_t)run & 1u, acc = tmem_base + b * 256u;
                    alive = __all_sync(0xffffffffu, mbar_wait_cluster<false>(&acc_empty[b], (((uint32_t)run >> 1) & 1u) ^ 1u, abort));
                    for (int k0 = kt; kt < kt_end && alive; ++kt) {
                        alive = __all_sync(0xffffffffu, mbar_wait(&split_done[ls], ph, abort) && mbar_wait_cluster<true>(&peer_split[ls], ph, abort));
                        if (!alive) break;
                        tc_fence_after();
                        const uint32_t hi = hi0 + (uint32_t)(s * stage_bytes), lo = lo0 + (uint32_t)(ls * stage_bytes);
                        const uint64_t a_hi = desc | (hi >> 4), b_hi = desc | ((hi + b_off) >> 4);
                        const uint64_t a_lo = desc | (lo >> 4), b_lo = desc | ((lo + b_off) >> 4);
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                mma_tf32_pair(acc, a_hi + 2 * k, b_hi + 2 * k, idesc, kt != k0 || k != 0);
                                mma_tf32_pair(acc, a_hi + 2 * k, b_lo + 2 * k, idesc, 1);
                                if (!diag) mma_tf32_pair(acc, a_lo + 2 * k, b_hi + 2 * k, idesc, 1);
                            }
                            mma_commit_pair(&empty[s]);
                            if (kt == kt_end - 1) mma_commit_pair(&acc_full[b]);
                        }
                        __syncwarp();
                        if (++s == n_hi) s = 0;
                        if (++ls == n_lo) { ls = 0; ph ^= 1u; }
                    }
                }
            }
        } else if (q == 1 && lane == 0) {
            // CTA 1's remainders are handed to the MMAs. On the diagonal a warp passes on every round of its slots (a ring of 6). Off it
            // (a ring of 3) the two take a slot's rounds in turn, and a round is not mistaken for the one two before: all workers
            // split every K tile there, so that K tile kt - 2, which this warp has seen done, was done after kt - 3.
            for (int kt = warp - 2; kt < nkt; kt += 2) {
                const int ls = kt % n_lo;
                if (!mbar_wait(&split_done[ls], (uint32_t)(kt / n_lo) & 1u, abort)) break;
                mbar_arrive_cluster(&peer_split[ls], 0);
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 200;");
        const int quarter = warp & 3, half = (warp - 4) >> 2;
        const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + (uint32_t)(half * 128);
        float sum[128];
#pragma unroll
        for (int j = 0; j < 128; ++j) sum[j] = 0.f;
        bool ok = true;
        auto drain = [&](int run) {
            const uint32_t b = (uint32_t)run & 1u;
            bool w = mbar_wait(&acc_full[b], ((uint32_t)run >> 1) & 1u, abort);
            w = __all_sync(0xffffffffu, w);
            if (!w) { ok = false; return; }
            tc_fence_after();
#pragma unroll
            for (int j0 = 0; j0 < 128; j0 += 32) {
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
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster_relaxed(&acc_empty[b], 0);
        };
        // A group sees every phase of its slots: both rings are multiples of the number of groups.
        const int grp = diag ? half : 0, nt = 32 * kPairWorkers / groups, t = (threadIdx.x - 128) & (nt - 1);
        const float scale = diag ? 2.f : 1.f;
        int s = grp, ls = grp, es = n_hi - n_lo + grp, drained = 0;     // es: the slot of hi that K tile kt - n_lo had
        uint32_t ph = 0, eph = 1;
        for (int kt = grp; kt < nkt && ok; kt += groups) {
            bool w = mbar_wait(&full[s], ph, abort) && (kt < n_lo || mbar_wait(&empty[es], eph, abort));
            w = __all_sync(0xffffffffu, w);
            if (!w) { ok = false; break; }
            const uint4* hi = reinterpret_cast<const uint4*>(smem + (size_t)s * stage_bytes) + t;
            uint4* lo = reinterpret_cast<uint4*>(lo_ring + (size_t)ls * stage_bytes) + t;
            for (int h = 0; h < 2; ++h, hi += 4 * nt, lo += 4 * nt) {
                uint4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = hi[u * nt];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    lo[u * nt] = make_uint4(remainder_tf32(v[u].x, scale), remainder_tf32(v[u].y, scale), remainder_tf32(v[u].z, scale), remainder_tf32(v[u].w, scale));
            }
            fence_proxy_async_smem();                       // the tensor cores read these writes
            __syncwarp();
            if (lane == 0) mbar_arrive(&split_done[ls]);
            s += groups;
            if (s >= n_hi) { s -= n_hi; ph ^= 1u; }
            ls += groups;
            if (ls >= n_lo) ls -= n_lo;
            es += groups;
            if (es >= n_hi) { es -= n_hi; eph ^= 1u; }
            // run d is drained once K tile 8 (d + 1) + n_lo has been split: its slot was free, so the run's MMAs are done (no waiting),
            // and the MMAs that need its accumulator again start 8 - n_lo K tiles later at the earliest
            while (ok && drained < nruns && (drained + 1) * kRunTiles + n_lo <= kt) drain(drained++);
        }
        while (ok && drained < nruns) drain(drained++);
        chain_release();
        const int row = m0 + q * 128 + quarter * 32 + lane, col = n0 + half * 128;
        if (ok && row < r) {
            float* o = C + (long long)slice * split_stride + (long long)row * ldc + col;
#pragma unroll
            for (int j = 0; j < 128; j += 4)                // ldc is r rounded up to a multiple of 4
                if (col + j < r) *reinterpret_cast<float4*>(o + j) = make_float4(sum[j], sum[j + 1], sum[j + 2], sum[j + 3]);
        }
    }
    // no MMA may be in flight when TMEM is freed, and no barrier of a CTA may go while the other still arrives on it
    if (warp == 1 && nruns > 0 && !*abort) mbar_wait_quiet(&acc_full[(nruns - 1) & 1], ((uint32_t)(nruns - 1) >> 1) & 1u, kWaitLimitCycles);
    tc_fence_before();
    __syncthreads();
    cluster_barrier();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, 512);
    }
    if (threadIdx.x == 0 && *abort) atomicExch(err, 1);
}

}  // namespace
}  // namespace tc

// See sage_internal.h.
cudaError_t launch_tc_gram_pair(const float* B, int64_t ldb, int r, int64_t K, int n_diag, int n_off, float* C, int64_t ldc, int64_t split_stride, int* err,
                                cudaStream_t st) {
    if (r <= 128 || r > 512 || K <= 0 || n_diag < 1 || (r > 256) != (n_off > 0)) return cudaErrorNotSupported;
    if (ldc % 4 || ldc < r || split_stride % 4 || (reinterpret_cast<uintptr_t>(C) & 15u)) return cudaErrorNotSupported;
    CUtensorMap tm;
    if (!tc::make_tmap_2d(&tm, B, 4, (uint64_t)r, (uint64_t)K, (uint64_t)ldb, 128)) return cudaErrorNotSupported;
    const cudaError_t e = allow_smem((const void*)tc::k_tc_gram_pair, 227 * 1024, tc::kPairRegs);
    if (e != cudaSuccess) return e;
    const unsigned pairs = (unsigned)(n_off ? n_off + 2 * n_diag : n_diag);
    return launch(tc::k_tc_gram_pair, LaunchShape{dim3(2 * pairs), dim3(tc::kPairThreads), tc::kPairSmem, 2}, st, tm, r, K, n_diag, n_off, C, ldc, split_stride, err);
}

}  // namespace sage
