// Inner products of the rows of a block (several shrink cycles' rows, see block_kernels.cu) on pairs of SMs. A row is held as one to
// three bfloat16 planes that add up to it exactly (x = hi + mid + lo, 8 significant bits each), a plane is a row of this kernel's
// operand, and the inner product of two rows is the sum over their planes, formed by launch_block_gram_reduce. Products of bfloat16
// values are exact in fp32 and no element is split on the way: TMA feeds the MMAs directly. The accumulator rounds toward zero, so it
// is drained into registers every kRunTiles K tiles (32 additions).
// Every element is the sum over the same K slices and runs whatever tile of whatever launch it is computed in: rows may arrive in any
// number of calls, the inner products do not depend on it.
// One cluster of two CTAs works on 256 x 256 tiles on and above the diagonal, one K slice at a time; tiles without a new row are left
// out. CTA q holds rows q*128 .. of both operands (on the diagonal they are the same rows).
//   warp 0     TMA loads of this CTA's rows, in boxes of 32 rows (where each comes from: BlockMap),
//   warp 1     TMEM; in CTA 0 the MMAs of both, into two accumulators of 256 columns in turn,
//   warps 4-11 drain this CTA's accumulator rows (4-7: columns 0-127, 8-11: the others).
// Both CTAs' loads report to CTA 0's barriers.
// What bounds it: bytes in flight. A K tile's 512 cycles of MMAs need 32 KB of each SM, and a load takes 2.6 us (4.6 us on rows 22 MB
// apart) when all SMs load: seven stages of 32 KB, of which six are on their way. 1,793 planes of 262,144 values: 920 us, with six stages 940.
// Boxes of two K tiles (256 bytes a row, as k_tc_rebuild_block loads them) make three stages of 64 KB: 1,410 us.
#include "block.cuh"

namespace sage {
namespace tc {
namespace {

constexpr int kThreads = 384;
constexpr int kRegs = 168;                  // what every thread is launched with: the shares below add up to 3 x 128 x 168
constexpr int kOpBytes = 128 * 128;         // 128 rows of one K tile (64 values)
constexpr int kBK = 64;
constexpr int kRunTiles = 8;
constexpr int kStages = 7;
struct PlaceTmaps {
    CUtensorMap place[3];
};
constexpr int kDrainWarps = 8;
constexpr size_t kSmem = 1024 + (size_t)kStages * 2 * kOpBytes + (2 * kStages + 4) * 8 + 16;

__global__ void __launch_bounds__(kThreads, 1)
k_tc_gram_block(const __grid_constant__ PlaceTmaps tm, BlockMap map, int first_blk, int tiles, int slices, int nkt_all, float* __restrict__ parts, int* __restrict__ err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + kStages * 2 * kOpBytes);   // [kStages], CTA 0's: bytes of both CTAs
    uint64_t* empty = full + kStages;                                   // [kStages], both CTAs'
    uint64_t* acc_full = empty + kStages;                               // [2], both CTAs'
    uint64_t* acc_empty = acc_full + 2;                                 // [2], CTA 0's: arrivals from both CTAs
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int q = blockIdx.x & 1, pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int items = tiles * slices;

    // item -> (K tiles [k0, k1), row blocks a <= b); items of one slice follow one another, so that pairs share its rows in L2
    auto item_of = [&](int item, int& k0, int& k1, int& a, int& b) {
        const int s = item / tiles;
        int t = item - s * tiles;
        k0 = (int)((long long)nkt_all * s / slices);
        k1 = (int)((long long)nkt_all * (s + 1) / slices);
        b = first_blk;
        while (t > b) t -= ++b;
        a = t;
    };

    // columns of row block b: the last one's planes in steps of 64, of which each CTA holds half
    auto cols_of = [&](int b) { return min(256, (map.P - b * 256 + 63) & ~63); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 2 * kDrainWarps);
        }
        *abort = 0;
        mbar_fence_init();
        for (int i = 0; i < 3; ++i) tma_prefetch_desc(&tm.place[i]);
    }
    if (warp == 1) tmem_alloc_pair(tmem_slot, 512);
    tc_fence_before();
    cluster_barrier();                          // the other CTA's barriers are set up, too
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    chain_wait();

    uint32_t last_run = 0;                      // accumulator runs of this pair in all (warp 1)
    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
        if (warp == 0) {
            if (lane == 0) {
                int issued = 0, s = 0;
                uint32_t ph = 1;
                bool alive = true;
                for (int item = pair; item < items && alive; item += pairs) {
                    int k0, k1, a, b;
                    item_of(item, k0, k1, a, b);
                    const int n = cols_of(b);
                    const bool diag = a == b && n == 256;
                    const uint32_t bytes = diag ? kOpBytes : kOpBytes + n * 64;
                    const CUtensorMap* from[8];
                    int y[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int p = (i < 4 ? a * 256 + q * 128 : b * 256 + q * (n / 2)) + (i & 3) * 32, place = block_place(map, p);
                        from[i] = &tm.place[place];
                        y[i] = block_place_row(map, p, place);
                    }
                    for (int kt = k0; kt < k1; ++kt) {
                        if (!mbar_wait(&empty[s], ph, abort)) { alive = false; break; }
                        uint8_t* st = smem + (size_t)s * 2 * kOpBytes;
                        if (q == 0) mbar_expect_tx(&full[s], 2 * bytes);
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if (i < 4 || (!diag && (i - 4) * 64 < n)) tma_load_2d_pair(st + i * 4096, from[i], &full[s], kt * kBK, y[i]);
                        ++issued;
                        if (++s == kStages) { s = 0; ph ^= 1u; }
                    }
                }
                if (q == 0 && *abort)
                    for (int k = issued > kStages ? issued - kStages : 0; k < issued; ++k)
                        mbar_wait_quiet(&full[k % kStages], (uint32_t)(k / kStages) & 1u, 20000000ll);
            }
        } else if (warp == 1) {
            bool alive = true;
            int s = 0;
            uint32_t ph = 0, run = 0;
            const uint64_t desc = smem_desc_k_sw128(0);
            const uint32_t st0 = smem_u32(smem);
            for (int item = pair; item < items && alive; item += pairs) {
                int k0, k1, a, b;
                item_of(item, k0, k1, a, b);
                if (q == 1) {                               // only counts the runs, for the wait at the end
                    run += (uint32_t)((k1 - k0 + kRunTiles - 1) / kRunTiles);
                    continue;
                }
                const int n = cols_of(b);
                const uint32_t idesc = instr_desc(1, 256, n, 0, 0), b_off = a == b && n == 256 ? 0u : (uint32_t)kOpBytes;
                for (int kt = k0; kt < k1 && alive; ++run) {
                    const int kt_end = kt + kRunTiles < k1 ? kt + kRunTiles : k1;
                    const uint32_t bf = run & 1u, acc = tmem_base + bf * 256u;
                    alive = __all_sync(0xffffffffu, mbar_wait_cluster<false>(&acc_empty[bf], ((run >> 1) & 1u) ^ 1u, abort));
                    for (int kf = kt; kt < kt_end && alive; ++kt) {
                        alive = __all_sync(0xffffffffu, mbar_wait_cluster<true>(&full[s], ph, abort));
                        if (!alive) break;
                        tc_fence_after();
                        const uint32_t st = st0 + (uint32_t)(s * 2 * kOpBytes);
                        const uint64_t da = desc | (st >> 4), db = desc | ((st + b_off) >> 4);
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) mma_bf16_pair(acc, da + 2 * k, db + 2 * k, idesc, kt != kf || k != 0);
                            mma_commit_pair(&empty[s]);
                            if (kt == kt_end - 1) mma_commit_pair(&acc_full[bf]);
                        }
                        __syncwarp();
                        if (++s == kStages) { s = 0; ph ^= 1u; }
                    }
                }
            }
            last_run = run;
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 200;");
        const int quarter = warp & 3, half = (warp - 4) >> 2;
        const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + (uint32_t)(half * 128);
        uint32_t run = 0;
        bool ok = true;
        for (int item = pair; item < items && ok; item += pairs) {
            int k0, k1, a, b;
            item_of(item, k0, k1, a, b);
            const int n = cols_of(b);
            float sum[128];
#pragma unroll
            for (int j = 0; j < 128; ++j) sum[j] = 0.f;
            for (int kt = k0; kt < k1; kt += kRunTiles, ++run) {
                const uint32_t bf = run & 1u;
                ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[bf], (run >> 1) & 1u, abort));
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int j0 = 0; j0 < 128; j0 += 32) {
                    if (half * 128 + j0 >= n) continue;
                    uint32_t v0[16], v1[16];
                    tmem_ld16_issue(lane_base + bf * 256u + (uint32_t)j0, v0);
                    tmem_ld16_issue(lane_base + bf * 256u + (uint32_t)(j0 + 16), v1);
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
                if (lane == 0) mbar_arrive_cluster_relaxed(&acc_empty[bf], 0);
            }
            const int row = q * 128 + quarter * 32 + lane, col = half * 128;
            if (ok && a * 256 + row < map.P) {
                float* o = parts + (size_t)item * 65536 + (size_t)row * 256 + col;
#pragma unroll
                for (int j = 0; j < 128; j += 4)
                    if (b * 256 + col + j < map.P) *reinterpret_cast<float4*>(o + j) = make_float4(sum[j], sum[j + 1], sum[j + 2], sum[j + 3]);
            }
        }
        chain_release();
    }
    // no MMA may be in flight when TMEM is freed, and no barrier of a CTA may go while the other still arrives on it
    if (warp == 1 && last_run > 0 && !*abort) mbar_wait_quiet(&acc_full[(last_run - 1) & 1], ((last_run - 1) >> 1) & 1u, kWaitLimitCycles);
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
cudaError_t launch_block_gram(const BlockSource& src, const BlockMap& map, int first_new, int64_t D, int slices, float* parts, int* err,
                              cudaStream_t st) {
    tc::PlaceTmaps tm;
    const tc::Place places[3] = {tc::place_of(src, map, 0), tc::place_of(src, map, 1), tc::place_of(src, map, 2)};
    for (int i = 0; i < 3; ++i)
        if (!tc::make_tmap_2d(&tm.place[i], places[i].base, 2, (uint64_t)std::max(places[i].rows, 1), (uint64_t)D, (uint64_t)places[i].ld, 32)) return cudaErrorInvalidValue;
    const int nkt = (int)((D + tc::kBK - 1) / tc::kBK);
    if (slices < 1 || slices > nkt || map.P < 1) return cudaErrorInvalidValue;
    const int first = block_phys(map, first_new) >> 8, tiles = block_tiles(map, first);
    const cudaError_t e = allow_smem((const void*)tc::k_tc_gram_block, 227 * 1024, tc::kRegs);
    if (e != cudaSuccess) return e;
    const int pairs = std::min(74, tiles * slices);
    return launch(tc::k_tc_gram_block, LaunchShape{dim3(2 * pairs), dim3(tc::kThreads), tc::kSmem, 2}, st, tm, map, first, tiles, slices, nkt,
                  parts, err);
}

}  // namespace sage
