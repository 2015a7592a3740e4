// Projection of fp32 rows onto a sketch of at most 64 rows, fp32-faithful on the tensor cores: Z = G S^T with both operands split into
// hi (the value read with its low 13 bits ignored, as kind::tf32 does) and lo (the remainder, rounded to 11 bits), all four
// products taken, an accumulator drained every kRunTiles K tiles into registers (it truncates at every addition).
// The data rows are the A operand: hi from shared memory, exactly as TMA left it, lo from TMEM, where the workers put it, so that the
// split costs no shared-memory store and no proxy fence; the sketch, split once into [hi (64 rows) ; lo (64 rows)] when it was
// frozen, is one 128-row B operand. Accumulator column j and 64 + j belong to output j.
// A pair of SMs works on 256 rows (cta_group::2), so that each loads half of the sketch's tile, the hi rows or the lo rows, next to its
// 128 rows: 24 KB a K tile, 700 cycles, as long as the rows take from memory at the copy rate; the MMAs take 512. What bounds it is how
// long a slot lives: load, hand-over to CTA 0, MMAs, eight slots in all (tensor pipe 56 %, DRAM 49 % of nominal, shared memory 31 %
// busy). CTA 1's landed data is released at cluster scope, 2,000 cycles or so under load, beside the split; remainders and drained
// accumulators are in tensor memory, where relaxed arrivals between tcgen05 fences do. (With default arrivals, which order nothing between two
// CTAs: 214 and 333 us where it takes 245 and 366. The release behind the split: 263 and 392; one warp that passes all on: 503.)
// Measured (against single SMs with 128-row tiles that loaded the whole sketch tile, remainders in shared memory, a block per tile and
// K slice): 50,000 rows of 5,130 onto 64 365 -> 245 us (1.03 GB: 159 us at the copy rate), 20,000 of 20,000 546 -> 366 us (245), 512 of 5,130
// 57 -> 19 us. On single SMs, the whole sketch tile loaded: 264 and 389 us.
// Pairs take equal shares of all K tiles of all row tiles, in order: a row tile may be cut, and part i of it goes to plane i. With
// classes (structured rows) every class is a slice of its own plane and nothing is cut.
//   warp 0     TMA loads (128-byte swizzle), warp 1 TMEM allocation and, in CTA 0, the MMAs of both,
//   warps 12-15 of CTA 1 tell CTA 0 what has landed there,
//   warps 4-11 remainders of landed K tiles in two groups in turn (a thread has one row), reported to CTA 0; between them they drain:
//              thread = row, 32 outputs each.
#include "sage_internal.h"
#include "tc05.cuh"

namespace sage {
namespace tc {
namespace {

constexpr int kProjThreads = 512;
constexpr int kProjRegs = 128;               // what every thread is launched with: the sum of the shares below is 4 x 128 x 128
constexpr int kRowBytes = 128 * 128;        // 128 rows of one K tile (32 floats)
constexpr int kStageBytes = kRowBytes + 64 * 128;     // and half of the sketch's
constexpr int kProjBK = 32;
constexpr int kStages = 8;                  // K tiles in flight, in shared memory and, their remainders, in TMEM
constexpr int kRunTiles = 3;                // K tiles, 24 additions, between drains of an accumulator
constexpr int kGroupWarps = 4;
// Warps that tell CTA 0 what has landed in CTA 1: a release at cluster scope takes as long as three K tiles. A forwarder has waited
// for a slot's round before the next one itself, so that the two are never mistaken for one another.
constexpr int kForwards = 4;
static_assert(kStages % kForwards == 0, "");
constexpr uint32_t kLoCol = 256;            // TMEM: two accumulators of 128 columns, then the remainders, 32 columns each
constexpr size_t kProjSmem = 1024 + (size_t)kStages * kStageBytes + (4 * kStages + 4) * 8 + 16;

struct ProjRange {                          // the K tiles of one row tile (and class) that a pair takes
    int tile, slice, part, k0, k1;
};
// Unit u of a launch: K tile u % nkt of item u / nkt; items are row tiles, or (row tile, class) pairs, which are not cut.
__device__ __forceinline__ ProjRange proj_range(long long u, long long u_end, int nkt, int slices, long long units) {
    ProjRange p;
    const long long item = u / nkt;
    p.tile = (int)(item / slices);
    p.slice = (int)(item - (long long)p.tile * slices);
    p.k0 = (int)(u - item * nkt);
    p.k1 = u_end - u < nkt - p.k0 ? p.k0 + (int)(u_end - u) : nkt;
    // the pair that took the item's first unit x: the largest b with units * b / pairs <= x
    const long long x = item * nkt;
    p.part = slices > 1 ? 0 : (int)((blockIdx.x >> 1) - (((x + 1) * (gridDim.x >> 1) + units - 1) / units - 1));
    return p;
}

__global__ void __launch_bounds__(kProjThreads, 1)
k_tc_project(const __grid_constant__ CUtensorMap tmRows, const __grid_constant__ CUtensorMap tmSk, int M, int ell, int nkt, int slices,
             long long slice_cols, long long units, int planes, float* __restrict__ out, long long plane_stride, int* __restrict__ err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)kStages * kStageBytes);   // local
    uint64_t* peer_full = full + kStages;                  // CTA 0's: CTA 1's full, passed on
    uint64_t* split_done = peer_full + kStages;            // CTA 0's: arrivals from both CTAs
    uint64_t* empty = split_done + kStages;                // both CTAs': the MMA thread's commits go to both
    uint64_t* acc_full = empty + kStages;                  // [2], likewise
    uint64_t* acc_empty = acc_full + 2;                    // [2], CTA 0's: arrivals from both CTAs
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = blockIdx.x & 1;
    const long long pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    long long u_begin, u_end;
    if (slices > 1) {
        const long long items = units / nkt;
        u_begin = items * pair / pairs * nkt;
        u_end = items * (pair + 1) / pairs * nkt;
    } else {
        u_begin = units * pair / pairs;
        u_end = units * (pair + 1) / pairs;
    }

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&peer_full[s], 1);
            mbar_init(&split_done[s], 2 * kGroupWarps);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 4 * kGroupWarps);
        }
        *abort = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmRows);
        tma_prefetch_desc(&tmSk);
    }
    if (warp == 1) tmem_alloc_pair(tmem_slot, 512);
    tc_fence_before();
    cluster_barrier();                          // the other CTA's barriers are set up, too
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    chain_wait();

    long long runs = 0;                                    // accumulator runs of this pair (every role counts them alike)
    for (long long u = u_begin; u < u_end;) {
        const ProjRange p = proj_range(u, u_end, nkt, slices, units);
        runs += (p.k1 - p.k0 + kRunTiles - 1) / kRunTiles;
        u += p.k1 - p.k0;
    }

    if (warp < 4 || warp >= 12) asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
    else asm volatile("setmaxnreg.inc.sync.aligned.u32 152;");
    if (warp == 0) {
        if (lane == 0) {
            long long g = 0;                               // K tiles of this pair so far
            bool alive = true;
            for (long long u = u_begin; u < u_end && alive;) {
                const ProjRange p = proj_range(u, u_end, nkt, slices, units);
                for (int kt = p.k0; kt < p.k1; ++kt, ++g) {
                    const int s = (int)(g % kStages);
                    if (!mbar_wait(&empty[s], ((uint32_t)(g / kStages) & 1u) ^ 1u, abort)) { alive = false; break; }
                    uint8_t* st = smem + (size_t)s * kStageBytes;
                    mbar_expect_tx(&full[s], (uint32_t)kStageBytes);
                    tma_load_2d(st, &tmRows, &full[s], kt * kProjBK, p.tile * 256 + q * 128);            // classes share the rows' columns
                    tma_load_2d(st + kRowBytes, &tmSk, &full[s], (int)(p.slice * slice_cols) + kt * kProjBK, q * 64);
                }
                u += p.k1 - p.k0;
            }
            if (*abort)
                for (long long k = g > kStages ? g - kStages : 0; k < g; ++k)
                    mbar_wait_quiet(&full[k % kStages], (uint32_t)(k / kStages) & 1u, 20000000ll);
        }
    } else if (warp == 1) {
        if (q == 0) {
            // the whole warp walks the loop, so that its values stay in uniform registers; one lane issues
            const uint32_t idesc = instr_desc(2, 256, 128, 0, 0);
            const uint64_t desc = smem_desc_k_sw128(0);
            const uint32_t st0 = smem_u32(smem);
            bool alive = true;
            int s = 0;
            uint32_t ph = 0, run = 0;
            for (long long u = u_begin; u < u_end && alive;) {
                const ProjRange p = proj_range(u, u_end, nkt, slices, units);
                for (int kt = p.k0; kt < p.k1 && alive; ++run) {
                    const int kt_end = kt + kRunTiles < p.k1 ? kt + kRunTiles : p.k1;
                    const uint32_t b = run & 1u, acc = tmem_base + b * 128u;
                    alive = __all_sync(0xffffffffu, mbar_wait_cluster<false>(&acc_empty[b], ((run >> 1) & 1u) ^ 1u, abort));
                    for (const int k0 = kt; kt < kt_end && alive; ++kt) {
                        alive = __all_sync(0xffffffffu, mbar_wait(&full[s], ph, abort) && mbar_wait_cluster<true>(&peer_full[s], ph, abort) && mbar_wait_cluster<false>(&split_done[s], ph, abort));
                        if (!alive) break;
                        tc_fence_after();
                        const uint32_t st = st0 + (uint32_t)(s * kStageBytes);
                        const uint64_t d_hi = desc | (st >> 4), d_sk = desc | ((st + kRowBytes) >> 4);
                        const uint32_t lo = tmem_base + kLoCol + (uint32_t)(s * 32);
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                mma_tf32_pair(acc, d_hi + 2 * k, d_sk + 2 * k, idesc, kt != k0 || k != 0);
                                mma_tf32_ts_pair(acc, lo + 8 * k, d_sk + 2 * k, idesc, 1);
                            }
                            mma_commit_pair(&empty[s]);
                            if (kt == kt_end - 1) mma_commit_pair(&acc_full[b]);
                        }
                        __syncwarp();
                        if (++s == kStages) { s = 0; ph ^= 1u; }
                    }
                }
                u += p.k1 - p.k0;
            }
        }
    } else if (warp >= 12) {
        if (q == 1 && lane == 0) {                          // what has landed in CTA 1 is the MMAs' to read
            for (long long g = warp - 12; g < u_end - u_begin; g += kForwards) {
                const int s = (int)(g % kStages);
                if (!mbar_wait(&full[s], (uint32_t)(g / kStages) & 1u, abort)) break;
                mbar_arrive_cluster(&peer_full[s], 0);
            }
        }
    } else if (warp >= 4) {
        const int quarter = warp & 3, grp = (warp - 4) >> 2, row_in = quarter * 32 + lane;
        const uint32_t lanes = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        float sum[32];
        bool ok = true;
        uint32_t run = 0;                                   // next run to drain
        auto drain = [&] {
            const uint32_t b = run & 1u;
            ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[b], (run >> 1) & 1u, abort));
            if (!ok) return;
            tc_fence_after();
            const uint32_t a = lanes + b * 128u + (uint32_t)(grp * 32);
#pragma unroll
            for (int j0 = 0; j0 < 32; j0 += 16) {
                uint32_t v0[16], v1[16];
                tmem_ld16_issue(a + (uint32_t)j0, v0);
                tmem_ld16_issue(a + (uint32_t)(64 + j0), v1);
                tmem_ld_wait();
                tmem_ld_use(v0);
                tmem_ld_use(v1);
#pragma unroll
                for (int j = 0; j < 16; ++j) sum[j0 + j] += __uint_as_float(v0[j]) + __uint_as_float(v1[j]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster_relaxed(&acc_empty[b], 0);
            ++run;
        };
        long long g0 = 0;                                   // K tiles of this pair before the current range
        for (long long u = u_begin; u < u_end && ok;) {
            const ProjRange p = proj_range(u, u_end, nkt, slices, units);
            const int n = p.k1 - p.k0, n_runs = (n + kRunTiles - 1) / kRunTiles;
            const uint32_t run0 = run;
#pragma unroll
            for (int j = 0; j < 32; ++j) sum[j] = 0.f;
            // K tile g of the pair belongs to group g & 1 (kStages is even: a group sees every phase of its slots)
            for (int i = (int)((g0 ^ grp) & 1); i < n && ok; i += 2) {
                const long long g = g0 + i;
                const int s = (int)(g % kStages);
                ok = __all_sync(0xffffffffu, mbar_wait(&full[s], (uint32_t)(g / kStages) & 1u, abort));
                if (!ok) break;
                // K tile g was loaded after the MMAs of K tile g - kStages: the columns of its remainders are free, too
                tc_fence_after();
                const uint4* src = reinterpret_cast<const uint4*>(smem + (size_t)s * kStageBytes) + row_in * 8;
                uint32_t lo[32];
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const uint4 v = src[c ^ (lane & 7)];
                    lo[4 * c] = remainder_tf32(v.x);
                    lo[4 * c + 1] = remainder_tf32(v.y);
                    lo[4 * c + 2] = remainder_tf32(v.z);
                    lo[4 * c + 3] = remainder_tf32(v.w);
                }
                tmem_st32(lanes + kLoCol + (uint32_t)(s * 32), lo);
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster_relaxed(&split_done[s], 0);
                // run d of this range is drained once K tile 3 (d + 1) + 2 has been split, when its MMAs are mostly done; the MMAs that need its
                // accumulator again start one K tile later
                while (ok && (int)(run - run0 + 2) * kRunTiles - 1 <= i) drain();
            }
            while (ok && (int)(run - run0) < n_runs) drain();
            if (!ok) break;
            g0 += n;
            u += n;
            if (u >= u_end) chain_release();
            const int row = p.tile * 256 + q * 128 + row_in, j0 = grp * 32;
            if (row < M && j0 < ell) {
                float* o = out + (long long)(p.slice + p.part) * plane_stride + (long long)row * ell + j0;
                const int last = p.k1 == nkt && slices == 1 ? planes - 1 - p.part : 0;        // planes that no other part of the tile writes
                if (ell % 4 == 0) {
#pragma unroll
                    for (int j = 0; j < 32; j += 4)
                        if (j0 + j < ell) *reinterpret_cast<float4*>(o + j) = make_float4(sum[j], sum[j + 1], sum[j + 2], sum[j + 3]);
                    for (int z = 1; z <= last; ++z)
#pragma unroll
                        for (int j = 0; j < 32; j += 4)
                            if (j0 + j < ell) *reinterpret_cast<float4*>(o + z * plane_stride + j) = make_float4(0.f, 0.f, 0.f, 0.f);
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (j0 + j < ell) o[j] = sum[j];
                    for (int z = 1; z <= last; ++z)
                        for (int j = 0; j < 32; ++j)
                            if (j0 + j < ell) o[z * plane_stride + j] = 0.f;
                }
            }
        }
    }
    // no MMA may be in flight when TMEM is freed, and no barrier of a CTA may go while the other still arrives on it
    if (warp == 1 && runs > 0 && !*abort) mbar_wait_quiet(&acc_full[(runs - 1) & 1], (uint32_t)((runs - 1) >> 1) & 1u, kWaitLimitCycles);
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
int project_planes(int64_t M, int64_t K, int64_t class_F) {
    if (class_F > 0 && class_F < K) return (int)(K / class_F);       // one plane per class
    const int64_t tiles = (M + 255) / 256, nkt = (K + tc::kProjBK - 1) / tc::kProjBK, units = tiles * nkt;
    const int64_t pairs = project_pairs(tiles, nkt);
    if (tiles % pairs == 0) return 1;
    const int64_t q = units / pairs;                       // K tiles of a pair, or one more
    return (int)((nkt - 2 + q) / q + 1);                   // parts that nkt consecutive ones fall into, at most
}

cudaError_t launch_tc_project(const float* rows, int64_t ld, const float* sk_split, int64_t lds, int64_t M, int ell, int64_t K, int64_t class_F,
                              float* out, int64_t plane_stride, int* err, cudaStream_t st) {
    if (M <= 0 || K <= 0) return cudaSuccess;
    if (ell < 1 || ell > 64 || M > (1 << 30)) return cudaErrorNotSupported;
    if (class_F > 0 && (class_F % 4 != 0 || K % class_F != 0)) return cudaErrorNotSupported;
    const int slices = class_F > 0 ? (int)(K / class_F) : 1;
    const int64_t cols = class_F > 0 ? class_F : K;
    CUtensorMap tmRows, tmSk;
    if (!tc::make_tmap_2d(&tmRows, rows, 4, (uint64_t)M, (uint64_t)cols, (uint64_t)ld, 128) ||
        !tc::make_tmap_2d(&tmSk, sk_split, 4, 128, (uint64_t)K, (uint64_t)lds, 64))
        return cudaErrorNotSupported;
    const int64_t tiles = (M + 255) / 256, nkt = (cols + tc::kProjBK - 1) / tc::kProjBK;
    const int64_t pairs = slices > 1 ? std::min<int64_t>(74, tiles * slices) : project_pairs(tiles, nkt);
    const int planes = project_planes(M, K, class_F);
    const cudaError_t e = allow_smem((const void*)tc::k_tc_project, 227 * 1024, tc::kProjRegs);
    if (e != cudaSuccess) return e;
    return launch(tc::k_tc_project, LaunchShape{dim3((unsigned)(2 * pairs)), dim3(tc::kProjThreads), tc::kProjSmem, 2}, st, tmRows, tmSk, (int)M, ell, (int)nkt, slices,
                  class_F, tiles * slices * nkt, planes, out, plane_stride, err);
}

}  // namespace sage
