// The kept rows at the end of a block from its planes: out[j][d] = sum_p T[j][p] plane_p[d] (see block_kernels.cu for T). The planes are
// the MMA's M side, 128 values d of a row on the lanes of TMEM, contiguous in memory (MN-major); T, itself as three bfloat16 planes
// that add up to it exactly, is the N side. Three MMAs (T's planes) per 16 planes of the block add into one accumulator.
// One pair of SMs per tile of 256 DS values, each with half of the values and half of T's rows: the tile's planes are read once, T (out of
// L2) once per tile.
//   warp 0 loads, warp 1 of CTA 0 issues the MMAs of both, warps 4-11 are the epilogue and drain (two accumulators in turn).
// Both CTAs' loads report to CTA 0's barriers.
// The result is written as three planes a row again, or in fp32 at the freeze.
#include "block.cuh"

namespace sage {
namespace tc {
namespace {

// Planes are loaded 32 at a time, 128 values of each: 256 consecutive bytes at every visit of a row. On rows megabytes apart each visit is
// another page, and what a stream of loads reaches depends on the bytes per visit (see make_tmap_4d_ktiles): 544 planes of 11.2 M values
// 3.74 ms with boxes of 128 bytes a row, 3.06 ms so. In shared memory: [group of 8 planes][128-byte half][8 planes][128 bytes], each half of a
// group in the 128-byte swizzle.
constexpr int kBoxPlanes = 32, kBoxCols = 128, kBoxBytes = kBoxPlanes * kBoxCols * 2, kGroupBytes = 2048;

// The three places: whole boxes, and boxes of 8 planes x 64 values for what is not whole (a place's last planes, a row's end).
struct BlockTmaps {
    CUtensorMap box[3], piece[3];
    int rows[3];                   // planes of each place
    int whole_cols;                // values of a row that whole boxes reach
};
bool block_tmaps(const BlockSource& src, const BlockMap& map, int64_t D, BlockTmaps* out) {
    out->whole_cols = (int)(D / 64 * 64);
    for (int i = 0; i < 3; ++i) {
        const auto [base, ld, rows] = place_of(src, map, i);
        out->rows[i] = rows;
        if (!make_tmap_2d(&out->piece[i], base, 2, (uint64_t)std::max(rows, 1), (uint64_t)D, (uint64_t)ld, 8)) return false;
        out->box[i] = out->piece[i];               // stays so, unused, where no box is whole
        if (D < 64) continue;
        // (a place without 8 planes has no whole box either: its map only answers "past the end")
        if (!make_tmap_4d_ktiles(&out->box[i], base, 2, (uint64_t)std::max(rows / 8 * 8, 8), (uint64_t)out->whole_cols, (uint64_t)ld, kBoxPlanes, 2)) return false;
    }
    return true;
}

// One box: planes p .. p + 31 of the block (p a multiple of 32; zeros past its end), values x .. x + 127 (zeros past the row's end). Reports
// kBoxBytes to the barrier of CTA 0.
__device__ __forceinline__ void load_block_box(uint8_t* dst, const BlockTmaps& tm, const BlockMap& m, uint64_t* bar, int p, int x) {
    const int place = block_place(m, p), row = block_place_row(m, p, place), rows = tm.rows[place];
    if (x + kBoxCols <= tm.whole_cols && (row + kBoxPlanes <= rows || row >= rows)) {
        tma_load_4d_pair(dst, &tm.box[place], bar, 0, 0, x >> 6, row >= rows ? 1 << 20 : row >> 3);
    } else {
#pragma unroll
        for (int g = 0; g < 4; ++g)
#pragma unroll
            for (int h = 0; h < 2; ++h) tma_load_2d_pair(dst + g * kGroupBytes + h * 1024, &tm.piece[place], bar, x + 64 * h, row + 8 * g);
    }
}

constexpr int kThreads = 384;
constexpr int kChunk = 64;                  // planes per stage
constexpr int kTileBytes = kChunk * 256;    // 64 planes x 128 values

__host__ __device__ constexpr int stage_bytes(int ds, int j_pad) { return ds * kTileBytes + 3 * (j_pad / 2) * 128; }   // of one CTA
__host__ __device__ constexpr int stage_count(int ds, int j_pad) {
    const int n = (227 * 1024 - 2048) / stage_bytes(ds, j_pad);
    return n > 8 ? 8 : n;
}

__device__ __forceinline__ unsigned short top16(float x) { return (unsigned short)(__float_as_uint(x) >> 16); }

constexpr int kRunChunks = 5;               // 60 additions to an accumulator, which truncates, between drains into registers

template <int DS, int JW>                   // tiles of 128 values; output rows per epilogue warp
__global__ void __launch_bounds__(kThreads, 1)
k_tc_rebuild_block(const __grid_constant__ BlockTmaps tm, const __grid_constant__ CUtensorMap tmT, BlockMap map, int j_pad, int keep, long long num_tiles,
                   unsigned short* __restrict__ planes, float* __restrict__ rows, long long ldo, int* __restrict__ err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    const int sbytes = stage_bytes(DS, j_pad), stages = stage_count(DS, j_pad);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)stages * sbytes);
    uint64_t* empty = full + 8;
    uint64_t* acc_full = empty + 8;             // [2]
    uint64_t* acc_empty = acc_full + 2;         // [2]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nchunk = (map.P + kChunk - 1) / kChunk;
    const int nruns = (nchunk + kRunChunks - 1) / kRunChunks;
    const int q = blockIdx.x & 1;
    const long long pair = blockIdx.x >> 1, pairs = gridDim.x >> 1, my_tiles = num_tiles > pair ? (num_tiles - pair + pairs - 1) / pairs : 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 16);
        }
        *abort = 0;
        mbar_fence_init();
        for (int i = 0; i < 3; ++i) tma_prefetch_desc(&tm.box[i]);
        tma_prefetch_desc(&tmT);
    }
    if (warp == 1) tmem_alloc_pair(tmem_slot, 512);
    tc_fence_before();
    cluster_barrier();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    chain_wait();

    if (warp == 0) {
        if (lane == 0) {
            long long issued = 0;
            bool alive = true;
            int s = 0;
            uint32_t ph = 1;
            for (long long lt = 0; lt < my_tiles && alive; ++lt) {
                const int d0 = (int)((2 * (pair + lt * pairs) + q) * (128 * DS));
                for (int c = 0; c < nchunk; ++c) {
                    if (!mbar_wait(&empty[s], ph, abort)) { alive = false; break; }
                    uint8_t* st = smem + (size_t)s * sbytes;
                    if (q == 0) mbar_expect_tx(&full[s], 2 * (uint32_t)sbytes);
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int x = 0; x < DS; ++x) load_block_box(st + x * kTileBytes + h * kBoxBytes, tm, map, &full[s], c * kChunk + 32 * h, d0 + 128 * x);
                    for (int t = 0; t < 3; ++t)
                        tma_load_2d_pair(st + DS * kTileBytes + t * j_pad * 64, &tmT, &full[s], c * kChunk, t * j_pad + q * (j_pad / 2));
                    ++issued;
                    if (++s == stages) { s = 0; ph ^= 1u; }
                }
            }
            if (q == 0 && *abort)
                for (long long k = issued > stages ? issued - stages : 0; k < issued; ++k)
                    mbar_wait_quiet(&full[k % stages], (uint32_t)(k / stages) & 1u, 20000000ll);
        }
    } else if (warp == 1 && q == 0) {
        const uint32_t idesc = instr_desc(1, 256, j_pad, 1, 0);             // A (planes) MN-major, B (T) K-major
        const uint64_t desc_a = smem_desc_mn_sw128(0, 1024, kGroupBytes), desc_t = smem_desc_k_sw128(0);
        const uint32_t st0 = smem_u32(smem), t_bytes = (uint32_t)j_pad * 64u;
        bool alive = true;
        int s = 0;
        uint32_t ph = 0;
        uint32_t run = 0;
        for (long long lt = 0; lt < my_tiles && alive; ++lt)
            for (int c0 = 0; c0 < nchunk && alive; c0 += kRunChunks, ++run) {
                const int c1 = c0 + kRunChunks < nchunk ? c0 + kRunChunks : nchunk;
                const uint32_t b = run & 1u, acc = tmem_base + b * 256u;
                alive = __all_sync(0xffffffffu, mbar_wait_cluster<false>(&acc_empty[b], ((run >> 1) & 1u) ^ 1u, abort));
                for (int c = c0; c < c1 && alive; ++c) {
                    alive = __all_sync(0xffffffffu, mbar_wait_cluster<true>(&full[s], ph, abort));
                    if (!alive) break;
                    tc_fence_after();
                    const uint32_t st = st0 + (uint32_t)(s * sbytes), tt = st + DS * kTileBytes;
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < 4; ++k)
#pragma unroll
                            for (int x = 0; x < DS; ++x) {
                                const uint64_t da = desc_a | ((st + (uint32_t)(x * kTileBytes + k * 2 * kGroupBytes)) >> 4);
#pragma unroll
                                for (int t = 0; t < 3; ++t)
                                    mma_bf16_pair(acc + (uint32_t)(x * j_pad), da, (desc_t | ((tt + (uint32_t)t * t_bytes) >> 4)) + 2 * k, idesc, c != c0 || k != 0 || t != 0);
                            }
                        mma_commit_pair(&empty[s]);
                        if (c == c1 - 1) mma_commit_pair(&acc_full[b]);
                    }
                    __syncwarp();
                    if (++s == stages) { s = 0; ph ^= 1u; }
                }
            }
    } else if (warp >= 4) {
        const int quarter = warp & 3, half = (warp - 4) >> 2;
        // DS = 2: half of the warps take a tile of 128 values each; DS = 1: half of the output rows
        const int x = DS == 2 ? half : 0, j_half = DS == 2 ? j_pad : (j_pad / 2 + 15) & ~15, j_first = DS == 2 ? 0 : half * j_half;
        const int jn = j_pad - j_first < j_half ? j_pad - j_first : j_half;              // a multiple of 16, at most JW
        const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + (uint32_t)(x * j_pad + j_first);
        uint32_t run = 0;
        bool ok = true;
        for (long long lt = 0; lt < my_tiles && ok; ++lt) {
            float sum[JW];
#pragma unroll
            for (int j = 0; j < JW; ++j) sum[j] = 0.f;
            for (int g = 0; g < nruns; ++g, ++run) {
                const uint32_t b = run & 1u;
                ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[b], (run >> 1) & 1u, abort));
                if (!ok) break;
                tc_fence_after();
                if (lt == my_tiles - 1 && g == nruns - 1) chain_release();
#pragma unroll
                for (int j0 = 0; j0 < JW; j0 += 16)
                    if (j0 < jn) {
                        uint32_t v[16];
                        tmem_ld16_issue(lane_base + b * 256u + (uint32_t)j0, v);
                        tmem_ld_wait();
                        tmem_ld_use(v);
#pragma unroll
                        for (int j = 0; j < 16; ++j) sum[j0 + j] += __uint_as_float(v[j]);
                    }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster_relaxed(&acc_empty[b], 0);
            }
            const long long d = (2 * (pair + lt * pairs) + q) * (128 * DS) + x * 128 + quarter * 32 + lane;
            if (!ok) break;
            if (rows) {
                if (d < ldo)
#pragma unroll
                    for (int j = 0; j < JW; ++j)
                        if (j < jn && j_first + j < keep) rows[(long long)(j_first + j) * ldo + d] = sum[j];
                continue;
            }
            // planes: lanes 2 i and 2 i + 1 exchange a value each, so that every store takes two neighbouring d (ldo is even)
            const bool odd = lane & 1;
#pragma unroll
            for (int j = 0; j < JW; j += 2) {
                const float got = __shfl_xor_sync(0xffffffffu, odd ? sum[j] : sum[j + 1], 1);
                float x0 = odd ? got : sum[j], x1 = odd ? sum[j + 1] : got;       // output row j (even lanes) or j + 1 (odd ones), at d & ~1
                const int row = j_first + j + (odd ? 1 : 0);
                if (j < jn && row < keep && d < ldo) {
                    unsigned short* o = planes + (long long)row * 3 * ldo + (d & ~1ll);
#pragma unroll
                    for (int t = 0; t < 3; ++t, o += ldo) {
                        const unsigned short a = top16(x0), c = top16(x1);
                        *reinterpret_cast<unsigned*>(o) = (unsigned)a | ((unsigned)c << 16);
                        x0 -= __uint_as_float((unsigned)a << 16);
                        x1 -= __uint_as_float((unsigned)c << 16);
                    }
                }
            }
        }
    }
    // no MMA may be in flight when TMEM is freed, and no barrier of a CTA may go while the other still arrives on it
    const long long last = my_tiles * nruns - 1;
    if (warp == 1 && last >= 0 && !*abort) mbar_wait_quiet(&acc_full[last & 1], (uint32_t)(last >> 1) & 1u, kWaitLimitCycles);
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
cudaError_t launch_block_rebuild(const BlockSource& src, const BlockMap& map, int64_t D, const __nv_bfloat16* T, int j_pad, int64_t ldT, int keep,
                                 __nv_bfloat16* planes, float* rows, int64_t ldo, int* err, cudaStream_t st) {
    if (j_pad < 32 || j_pad > 256 || (j_pad & 31) || keep > j_pad || map.P < 1) return cudaErrorInvalidValue;
    tc::BlockTmaps tm;
    CUtensorMap tmT;
    const int64_t k64 = (map.P + 63) / 64 * 64;
    if (k64 > ldT || !tc::block_tmaps(src, map, D, &tm) ||
        !tc::make_tmap_2d(&tmT, T, 2, (uint64_t)(3 * j_pad), (uint64_t)k64, (uint64_t)ldT, (uint32_t)(j_pad / 2)))
        return cudaErrorInvalidValue;
    // two tiles of 128 values share a stage's factors where the rows are long enough to fill the SMs twice that way
    const bool two = j_pad <= 64 && ldo >= (int64_t)148 * 512;
    const long long tiles = (ldo + (two ? 511 : 255)) / (two ? 512 : 256);
    const int pairs = (int)(tiles < 74 ? tiles : 74);
    const int ds = two ? 2 : 1;
    const size_t smem = (size_t)tc::stage_count(ds, j_pad) * tc::stage_bytes(ds, j_pad) + 1024 + 20 * 8 + 16;
    auto kernel = two            ? tc::k_tc_rebuild_block<2, 64>
                  : j_pad <= 64  ? tc::k_tc_rebuild_block<1, 32>
                  : j_pad <= 128 ? tc::k_tc_rebuild_block<1, 64>
                                 : tc::k_tc_rebuild_block<1, 128>;
    const cudaError_t e = allow_smem((const void*)kernel, 227 * 1024);
    if (e != cudaSuccess) return e;
    return launch(kernel, LaunchShape{dim3(2 * pairs), dim3(tc::kThreads), smem, 2}, st, tm, tmT, map, j_pad, keep, tiles,
                          reinterpret_cast<unsigned short*>(planes), rows, ldo, err);
}

}  // namespace sage
