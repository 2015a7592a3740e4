// Top-k selection (Algorithm 1, the top-k step) with a total order: score descending, then index ascending, and the orders by
// class that the class-balanced variant needs. A stable radix sort, 8 bits a pass, least significant digit first: each score
// becomes a 32-bit integer whose ascending order is the descending order of the scores, paired with its row index; rows start
// in index order, so ties stay in it and the index needs no passes of its own. Passes over the label follow where rows are
// grouped by class. Integer work only: results are exact.
//
// Up to kClusterMax rows the whole sort is one launch: a cluster of 8 thread blocks, digit counts exchanged through
// distributed shared memory, keys through L2, two cluster barriers per pass. Such a sort is bound by latency (launches before,
// barriers and shared-memory conflicts now). Beyond, three launches per pass (counts, one block per digit scanning its
// counters, scatter). A selection sorts as little as it can (select_filters). Measured, a call on 50,000 scores, a tenth wanted:
// 149 us (20 launches, all scores sorted, index included) -> 57 us (one cluster sort) -> 32 us (the 5,000 picks ranked).
#include <cooperative_groups.h>

#include <cstdio>
#include <mutex>

#include "sage_internal.h"

namespace sage {
namespace {

namespace cg = cooperative_groups;
using u64 = unsigned long long;

constexpr int kThreads = 256;
constexpr int kItems = 16;
constexpr int kTile = kThreads * kItems;   // keys per block
constexpr int kWarps = kThreads / 32;

__device__ __forceinline__ uint32_t ordered_bits(float f) {
    if (f != f) return 0u;                                   // NaN ranks below everything
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);       // larger float <-> larger integer
}
__device__ __forceinline__ u64 make_key(const float* scores, int64_t i) {
    float s = scores[i];
    if (s == 0.f) s = 0.f;                                   // -0 and +0 compare equal: give them one key
    return ((u64)(~ordered_bits(s)) << 32) | (u64)(uint32_t)i;
}
// Class of a row, labels outside [0, C) as class C.
__device__ __forceinline__ unsigned class_of(const int* labels, u64 key, int C) {
    const int lab = labels[(uint32_t)key];
    return (lab >= 0 && lab < C) ? (unsigned)lab : (unsigned)C;
}

// What a sort is for. by_score: four passes over the score image first; label_passes: 0, 1 or 2 passes over the class.
struct SortArgs {
    const float* scores;
    const int* labels;
    int64_t N;
    int C, by_score, label_passes;
    bool given = false;                                      // the keys are in the first buffer already (one-launch form)
};
__device__ __forceinline__ unsigned digit_of(const SortArgs& a, u64 key, int pass) {
    const int vp = a.by_score ? 4 : 0;
    if (pass < vp) return (unsigned)(key >> (32 + 8 * pass)) & 255u;
    return (class_of(a.labels, key, a.C) >> (8 * (pass - vp))) & 255u;
}

// Lanes that hold the same digit (256: a lane without a key), by a vote per bit: a match instruction takes longer the more values
// there are (2,000 cycles per 32 keys and warp on random digits).
__device__ __forceinline__ unsigned same_digit(unsigned d) {
    const unsigned none = __ballot_sync(0xffffffffu, d == 256u);
    unsigned m = d == 256u ? none : ~none;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const unsigned v = __ballot_sync(0xffffffffu, (d >> b) & 1u);
        m &= (d >> b) & 1u ? v : ~v;
    }
    return m;
}

// ---- one launch: cluster of 8 ------------------------------------------------------------------------------------
constexpr int kClThreads = 1024, kClWarps = 32, kClSize = 8;
constexpr int kClKeys = 16384;                               // most keys per block
// What shared memory holds, and about where eight SMs stop being enough: one launch against three launches a pass on all SMs, whole
// calls, 50,000 and 131,072 rows: all scores sorted 50 against 100 and 92 against 102 us, scores by 10 classes 28 against 69 and 48 against
// 92, by 1,000 classes 77 against 107 and 126 against 121, picks of 10 classes 108 against 191 and 171 against 209.
constexpr int64_t kClusterMax = (int64_t)kClSize * kClKeys;

struct ClusterShared {
    unsigned short cnt[kClWarps][256];
    unsigned short pos[kClKeys];                             // rank of a key among those of its digit before it in its warp's run
    u64 local[kClKeys];                                      // the block's keys by digit, so that they leave in runs
    unsigned hist[256];                                      // this block's counts, read by the others
    unsigned base[256];                                      // where this block's keys of a digit go, minus lexcl
    unsigned lexcl[256];                                     // where they start in `local`
    unsigned excl[257];                                      // where a digit's keys start
    unsigned total[256];
    unsigned wsum[16];
    long long kc[256], rem[256], offs[256];
};

enum Emit { EMIT_TOPK = 0, EMIT_ORDER, EMIT_PICK };
// EMIT_TOPK: idx[p] = row at place p, p < k. EMIT_ORDER: order[p] = row (an even number of passes: order may be b0), starts[c] = first
// place of class c (one label pass: c <= C <= 255). EMIT_PICK (one label pass): the quotas of the classes by largest remainder (sage_select_classes),
// idx = the first kc[c] of class 0, then of class 1, ...; kc_out[0 .. C - 1] the quotas, kc_out[C] their sum.
template <int MODE>
__global__ void __launch_bounds__(kClThreads, 1)
k_sort_cluster(SortArgs a, u64* __restrict__ b0, u64* __restrict__ b1, int64_t k, double keep_rate, int64_t* __restrict__ idx,
               unsigned* __restrict__ order, unsigned* __restrict__ starts, long long* __restrict__ kc_out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ClusterShared& sh = *reinterpret_cast<ClusterShared*>(smem_raw);
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int span = (int)((a.N + kClSize * kClThreads - 1) / (kClSize * kClThreads)) * 32;   // keys per warp, whole slots of 32
    const int64_t base = ((int64_t)rank * kClWarps + warp) * span;
    const int passes = (a.by_score ? 4 : 0) + a.label_passes;
    u64* in = b0;
    u64* out = b1;
    chain_wait();
    for (int pass = 0; pass < passes; ++pass) {
        const bool last = pass == passes - 1;
        auto load = [&](int64_t i) -> u64 {
            if (i >= a.N) return 0ull;
            if (pass > 0 || a.given) return __ldcg(in + i);
            return a.by_score ? make_key(a.scores, i) : (u64)i;
        };
        for (int e = tid; e < kClWarps * 128; e += kClThreads) reinterpret_cast<unsigned*>(&sh.cnt[0][0])[e] = 0u;
        __syncthreads();
        unsigned short* cnt = sh.cnt[warp];
        unsigned short* pos = sh.pos + warp * span;
        for (int s0 = 0; s0 < span; s0 += 128) {             // four slots' loads in flight
            u64 key[4];
            unsigned dig[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) key[u] = load(s0 + 32 * u < span ? base + s0 + 32 * u + lane : a.N);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool live = s0 + 32 * u < span && base + s0 + 32 * u + lane < a.N;
                dig[u] = live ? digit_of(a, key[u], pass) : 256u;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (s0 + 32 * u >= span) break;
                const unsigned peers = same_digit(dig[u]);
                const unsigned r = __popc(peers & ((1u << lane) - 1u));
                const unsigned before = dig[u] < 256u ? cnt[dig[u]] : 0u;
                __syncwarp();
                if (dig[u] < 256u && r == 0) cnt[dig[u]] = (unsigned short)(before + __popc(peers));
                __syncwarp();
                pos[s0 + 32 * u + lane] = (unsigned short)(before + r);
            }
        }
        __syncthreads();
        if (tid < 256) {                                     // counts of the warps before, and of the block
            unsigned run = 0;
#pragma unroll
            for (int w = 0; w < kClWarps; ++w) {
                const unsigned c = sh.cnt[w][tid];
                sh.cnt[w][tid] = (unsigned short)run;
                run += c;
            }
            sh.hist[tid] = run;
        }
        cluster.sync();
        unsigned before = 0, total = 0, x = 0, xl = 0;
        if (tid < 256) {
#pragma unroll
            for (int r = 0; r < kClSize; ++r) {
                const unsigned v = cluster.map_shared_rank(sh.hist, r)[tid];
                if (r < rank) before += v;
                total += v;
            }
            x = total;
            xl = sh.hist[tid];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, x, o), yl = __shfl_up_sync(0xffffffffu, xl, o);
                if (lane >= o) {
                    x += y;
                    xl += yl;
                }
            }
            if (lane == 31) {
                sh.wsum[warp] = x;
                sh.wsum[8 + warp] = xl;
            }
        }
        __syncthreads();
        if (tid < 256) {
            unsigned e = x - total, el = xl - sh.hist[tid];
            for (int w = 0; w < warp; ++w) {
                e += sh.wsum[w];
                el += sh.wsum[8 + w];
            }
            sh.excl[tid] = e;
            if (tid == 255) sh.excl[256] = e + total;
            sh.base[tid] = e + before - el;
            sh.lexcl[tid] = el;
            sh.total[tid] = total;
        }
        __syncthreads();
        if (MODE == EMIT_PICK && last) {
            // quotas: k_c = floor(k n_c / n), the k - sum largest remainders (ties: smaller class) get one more
            const long long n_valid = (long long)sh.excl[a.C];
            double kd = floor(__dadd_rn(__dmul_rn(keep_rate, (double)n_valid), 0.5));     // rounded twice, as sage_select_count does
            kd = kd < 0.0 ? 0.0 : kd > (double)n_valid ? (double)n_valid : kd;
            const long long kk = n_valid > 0 ? (long long)kd : 0;
            if (tid < a.C) {
                const long long num = (long long)sh.total[tid] * kk;
                const long long q = n_valid > 0 ? num / n_valid : 0;
                sh.kc[tid] = q;
                sh.rem[tid] = num - q * n_valid;
            }
            __syncthreads();
            long long mine = 0;
            if (tid < a.C) {
                long long given = 0;
                int larger = 0;
                for (int c = 0; c < a.C; ++c) {
                    given += sh.kc[c];
                    larger += sh.rem[c] > sh.rem[tid] || (sh.rem[c] == sh.rem[tid] && c < tid);
                }
                mine = sh.kc[tid] + (larger < kk - given ? 1 : 0);
            }
            __syncthreads();
            if (tid < a.C) sh.kc[tid] = mine;
            __syncthreads();
            if (tid < a.C) {
                long long o = 0;
                for (int c = 0; c < tid; ++c) o += sh.kc[c];
                sh.offs[tid] = o;
                if (rank == 0) {
                    kc_out[tid] = mine;
                    if (tid == a.C - 1) kc_out[a.C] = o + mine;
                }
            }
            __syncthreads();
        }
        if (MODE == EMIT_ORDER && last && starts && rank == 0 && tid <= a.C) starts[tid] = sh.excl[tid];
        for (int s0 = 0; s0 < span; s0 += 128) {
            u64 key[4];
            unsigned dig[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) key[u] = load(s0 + 32 * u < span ? base + s0 + 32 * u + lane : a.N);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool live = s0 + 32 * u < span && base + s0 + 32 * u + lane < a.N;
                dig[u] = live ? digit_of(a, key[u], pass) : 256u;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (dig[u] < 256u) sh.local[sh.lexcl[dig[u]] + cnt[dig[u]] + pos[s0 + 32 * u + lane]] = key[u];
        }
        __syncthreads();
        const int mine = max((long long)0, min((long long)span * kClWarps, (long long)(a.N - (int64_t)rank * kClWarps * span)));
        for (int i = tid; i < mine; i += kClThreads) {
            const u64 key = sh.local[i];
            const unsigned d = digit_of(a, key, pass), p = sh.base[d] + (unsigned)i;
            if (!last) {
                out[p] = key;
            } else if (MODE == EMIT_TOPK) {
                if ((int64_t)p < k) idx[p] = (int64_t)(uint32_t)key;
            } else if (MODE == EMIT_ORDER) {
                order[p] = (unsigned)(uint32_t)key;
            } else {
                const long long r = (long long)(p - sh.excl[d]);
                if ((int)d < a.C && r < sh.kc[d]) idx[sh.offs[d] + r] = (int64_t)(uint32_t)key;
            }
        }
        cluster.sync();                                      // keys are out, counts may be overwritten
        u64* t = in;
        in = out;
        out = t;
    }
}

template <int MODE>
cudaError_t run_cluster_sort(const SortArgs& a, u64* b0, u64* b1, int64_t k, double keep_rate, int64_t* idx, unsigned* order, unsigned* starts,
                             long long* kc_out, cudaStream_t st) {
    cudaError_t e = allow_smem((const void*)k_sort_cluster<MODE>, (int)sizeof(ClusterShared));
    if (e != cudaSuccess) return e;
    return launch(k_sort_cluster<MODE>, LaunchShape{dim3(kClSize), dim3(kClThreads), sizeof(ClusterShared), (unsigned)kClSize}, st, a, b0, b1, k, keep_rate, idx,
                  order, starts, kc_out);
}

// ---- few picks: the k-th key first, then only the k best are put in order --------------------------------------------
// k_top_keys: one cluster of 8. The k-th smallest score image is found by its digits (11, 11, 10 bits, counts exchanged through
// distributed shared memory), ties at it go to the smaller indices, and the k keys are written in index order. Up to
// kClusterMax rows each block keeps its scores in shared memory; beyond it reads them again (from L2) at every step.
constexpr int64_t kFilterMax = 1 << 18;                     // 500,000 scores, a tenth wanted: 146 us this way, 105 us by sorting on all SMs
constexpr int kBins = 2048;
struct FilterShared {
    unsigned hist[kBins];
    unsigned wsum[kClWarps];
    unsigned nless[kClWarps], neq[kClWarps];
    unsigned cta_less, cta_eq;                               // read by the other blocks
    unsigned digit, below;
    unsigned val[kClKeys];
};
__global__ void __launch_bounds__(kClThreads, 1) k_top_keys(const float* __restrict__ scores, int64_t N, int64_t k, u64* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FilterShared& sh = *reinterpret_cast<FilterShared*>(smem_raw);
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int span = (int)((N + kClSize * kClThreads - 1) / (kClSize * kClThreads)) * 32;     // scores per warp, whole slots of 32
    const int64_t base = ((int64_t)rank * kClWarps + warp) * span;
    const int live = (int)max((int64_t)0, min((int64_t)span, N - base));
    const bool resident = N <= kClusterMax;
    unsigned* vals = sh.val + (resident ? warp * span : 0);
    auto image = [&](int i) -> unsigned { return (unsigned)(make_key(scores, base + i) >> 32); };
    chain_wait();
    chain_release();
    if (resident) {
#pragma unroll 4
        for (int i = lane; i < live; i += 32) vals[i] = image(i);
        __syncwarp();
    }
    auto value = [&](int i) -> unsigned { return resident ? vals[i] : image(i); };
    unsigned prefix = 0, mask = 0, want = (unsigned)k;       // looking for the want-th smallest among values with v & mask == prefix
#pragma unroll 1
    for (int step = 0; step < 3; ++step) {
        const int shift = step == 0 ? 21 : step == 1 ? 10 : 0, bits = step == 2 ? 10 : 11;
        for (int e = tid; e < kBins; e += kClThreads) sh.hist[e] = 0u;
        __syncthreads();
#pragma unroll 4
        for (int s0 = 0; s0 < span; s0 += 32) {
            const int i = s0 + lane;
            const unsigned v = i < live ? value(i) : 0u;
            const bool on = i < live && (v & mask) == prefix;
            const unsigned d = (v >> shift) & ((1u << bits) - 1u);
            const unsigned act = __ballot_sync(0xffffffffu, on);
            if (act == 0u) continue;
            const unsigned d0 = __shfl_sync(0xffffffffu, d, __ffs(act) - 1);
            if (__ballot_sync(0xffffffffu, on && d != d0) == 0u) {         // all alike: one add
                if (lane == 0) atomicAdd(&sh.hist[d0], (unsigned)__popc(act));
            } else if (on) {
                atomicAdd(&sh.hist[d], 1u);
            }
        }
        cluster.sync();
        unsigned h[2] = {0u, 0u};                            // bins 2 tid, 2 tid + 1 over the whole cluster
#pragma unroll
        for (int r = 0; r < kClSize; ++r) {
            const uint2 v = *reinterpret_cast<const uint2*>(cluster.map_shared_rank(sh.hist, r) + 2 * tid);
            h[0] += v.x;
            h[1] += v.y;
        }
        const unsigned mine = h[0] + h[1];
        unsigned x = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) sh.wsum[warp] = x;
        __syncthreads();
        unsigned e = x - mine;
        for (int w = 0; w < warp; ++w) e += sh.wsum[w];
        if (e < want && want <= e + h[0]) { sh.digit = 2 * tid; sh.below = e; }
        if (e + h[0] < want && want <= e + mine) { sh.digit = 2 * tid + 1; sh.below = e + h[0]; }
        cluster.sync();                                      // the counts have been read by everybody
        prefix |= sh.digit << shift;
        mask |= ((1u << bits) - 1u) << shift;
        want -= sh.below;
    }
    // prefix is the k-th value; all smaller ones and the first `want` equal ones are picked
    unsigned nl = 0, ne = 0;
#pragma unroll 4
    for (int i = lane; i < live; i += 32) {
        const unsigned v = value(i);
        nl += v < prefix;
        ne += v == prefix;
    }
    nl = __reduce_add_sync(0xffffffffu, nl);
    ne = __reduce_add_sync(0xffffffffu, ne);
    if (lane == 0) {
        sh.nless[warp] = nl;
        sh.neq[warp] = ne;
    }
    __syncthreads();
    if (warp == 0) {
        const unsigned a = __reduce_add_sync(0xffffffffu, sh.nless[lane]), b = __reduce_add_sync(0xffffffffu, sh.neq[lane]);
        if (lane == 0) {
            sh.cta_less = a;
            sh.cta_eq = b;
        }
    }
    cluster.sync();
    unsigned less = 0, eq = 0;                               // before this warp's run
    for (int r = 0; r < rank; ++r) {
        less += *cluster.map_shared_rank(&sh.cta_less, r);
        eq += *cluster.map_shared_rank(&sh.cta_eq, r);
    }
    for (int w = 0; w < warp; ++w) {
        less += sh.nless[w];
        eq += sh.neq[w];
    }
#pragma unroll 2
    for (int s0 = 0; s0 < span; s0 += 32) {
        const int i = s0 + lane;
        const unsigned v = i < live ? value(i) : 0xffffffffu;
        const bool lt = i < live && v < prefix, same = i < live && v == prefix;
        const unsigned bl = __ballot_sync(0xffffffffu, lt), be = __ballot_sync(0xffffffffu, same), mine = (1u << lane) - 1u;
        const unsigned e = eq + __popc(be & mine);
        if (lt || (same && e < want)) out[less + __popc(bl & mine) + min(e, want)] = ((u64)v << 32) | (u64)(uint32_t)(base + i);
        less += __popc(bl);
        eq += __popc(be);
    }
    cluster.sync();                                          // no block leaves while another reads its counts
}

// Few keys: a key's place is the number of smaller ones. Block: 32 keys (one per lane), each of its 16 warps compares them with a
// sixteenth of all. keys == nullptr: made from the scores. n <= kRankMax: 8,192 keys take 5 us on all SMs, about what the sort
// takes on eight; the work grows with the square.
constexpr int kRankMax = 8192;
constexpr int kRankThreads = 512;
__global__ void __launch_bounds__(kRankThreads) k_rank(const u64* __restrict__ keys, const float* __restrict__ scores, int n, int64_t k,
                                                       int64_t* __restrict__ idx) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    u64* all = reinterpret_cast<u64*>(smem_raw);             // n, rounded up to 32 with keys that no other is larger than
    __shared__ unsigned place[kRankThreads / 32][32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int np = (n + 31) & ~31;
    chain_wait();
#pragma unroll 4
    for (int i = tid; i < np; i += kRankThreads) all[i] = i < n ? (keys ? __ldcg(keys + i) : make_key(scores, i)) : ~0ull;
    __syncthreads();
    const int me = blockIdx.x * 32 + lane;
    const u64 mine = me < np ? all[me] : ~0ull;
    unsigned less = 0;
    const ulonglong2* two = reinterpret_cast<const ulonglong2*>(all);
#pragma unroll 4
    for (int i = warp; i < np / 2; i += kRankThreads / 32) {
        const ulonglong2 o = two[i];
        less += (o.x < mine) + (o.y < mine);
    }
    place[warp][lane] = less;
    __syncthreads();
    if (warp == 0 && me < n) {
        unsigned p = 0;
#pragma unroll
        for (int w = 0; w < kRankThreads / 32; ++w) p += place[w][lane];
        if ((int64_t)p < k) idx[p] = (int64_t)(uint32_t)mine;
    }
}

cudaError_t run_rank(const u64* keys, const float* scores, int n, int64_t k, int64_t* idx, cudaStream_t st) {
    const int np = (n + 31) & ~31;
    cudaError_t e = allow_smem((const void*)k_rank, kRankMax * 8);
    if (e != cudaSuccess) return e;
    return launch_chained(k_rank, dim3((unsigned)(np / 32)), dim3(kRankThreads), (size_t)np * 8, st, keys, scores, n, k, idx);
}

cudaError_t run_top_keys(const float* scores, int64_t N, int64_t k, u64* out, cudaStream_t st) {
    cudaError_t e = allow_smem((const void*)k_top_keys, (int)sizeof(FilterShared));
    if (e != cudaSuccess) return e;
    return launch(k_top_keys, LaunchShape{dim3(kClSize), dim3(kClThreads), sizeof(FilterShared), (unsigned)kClSize}, st, scores, N, k, out);
}

// ---- three launches per pass, any N ------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) k_make_keys(SortArgs a, u64* __restrict__ keys) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i < a.N) keys[i] = a.by_score ? make_key(a.scores, i) : (u64)i;
}

__global__ void __launch_bounds__(kThreads) k_histogram(SortArgs a, const u64* __restrict__ keys, int pass, unsigned* __restrict__ hist,
                                                        int nblocks, unsigned* __restrict__ totals) {
    __shared__ unsigned h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kTile;
#pragma unroll
    for (int s = 0; s < kItems; ++s) {
        const int64_t i = base + s * kThreads + threadIdx.x;
        const unsigned d = i < a.N ? digit_of(a, keys[i], pass) : 256u;
        const unsigned peers = same_digit(d);         // scores share their leading bits: one add per value and warp
        if (d < 256u && (threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&h[d], (unsigned)__popc(peers));
    }
    __syncthreads();
    const unsigned v = h[threadIdx.x];
    hist[(int64_t)threadIdx.x * nblocks + blockIdx.x] = v;
    if (v) atomicAdd(&totals[pass * 256 + threadIdx.x], v);
}

// Block d: exclusive scan of the blocks' counts of digit d, starting at the number of keys with smaller digits.
__global__ void __launch_bounds__(kThreads) k_scan(unsigned* __restrict__ hist, int nblocks, const unsigned* __restrict__ totals) {
    __shared__ unsigned ws[kWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, d = blockIdx.x;
    auto block_sum = [&](unsigned v, unsigned& incl) {       // inclusive scan over the block; returns the block's sum
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += y;
        }
        if (lane == 31) ws[warp] = v;
        __syncthreads();
        unsigned before = 0, sum = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            if (w < warp) before += ws[w];
            sum += ws[w];
        }
        __syncthreads();
        incl = v + before;
        return sum;
    };
    unsigned incl;
    unsigned carry = block_sum(tid < d ? totals[tid] : 0u, incl);
    unsigned* row = hist + (int64_t)d * nblocks;
    for (int b0 = 0; b0 < nblocks; b0 += kThreads) {
        const unsigned v = b0 + tid < nblocks ? row[b0 + tid] : 0u;
        const unsigned sum = block_sum(v, incl);
        if (b0 + tid < nblocks) row[b0 + tid] = carry + incl - v;
        carry += sum;
    }
}

// Stable scatter: warp w of a block owns the contiguous keys [w*512, (w+1)*512) of the tile, walked in
// 16 slots of 32 consecutive keys, so (warp, slot, lane) order is index order. The last pass of a selection (idx != null)
// writes the first k rows in place of the keys.
__global__ void __launch_bounds__(kThreads) k_scatter(SortArgs a, const u64* __restrict__ in, int pass, const unsigned* __restrict__ offsets,
                                                      int nblocks, u64* __restrict__ out, int64_t k, int64_t* __restrict__ idx) {
    __shared__ unsigned cnt[kWarps][256];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int e = tid; e < kWarps * 256; e += kThreads) (&cnt[0][0])[e] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kTile + (int64_t)warp * (kItems * 32);
    u64 key[kItems];
    unsigned short pos[kItems], dig[kItems];
#pragma unroll
    for (int s = 0; s < kItems; ++s) {
        const int64_t i = base + s * 32 + lane;
        key[s] = i < a.N ? in[i] : 0ull;
    }
#pragma unroll
    for (int s = 0; s < kItems; ++s) {
        const bool live = base + s * 32 + lane < a.N;
        const unsigned d = live ? digit_of(a, key[s], pass) : 256u;
        const unsigned peers = same_digit(d);
        const unsigned rank = __popc(peers & ((1u << lane) - 1u));
        unsigned before = 0;
        if (live) before = cnt[warp][d];
        __syncwarp();
        if (live && rank == 0) cnt[warp][d] = before + __popc(peers);
        __syncwarp();
        pos[s] = (unsigned short)(before + rank);
        dig[s] = (unsigned short)d;
    }
    __syncthreads();
    {   // thread d: turn per-warp counts of digit d into start offsets
        unsigned off = offsets[(int64_t)tid * nblocks + blockIdx.x];
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const unsigned c = cnt[w][tid];
            cnt[w][tid] = off;
            off += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < kItems; ++s) {
        if (dig[s] >= 256u) continue;
        const unsigned p = cnt[warp][dig[s]] + pos[s];
        if (!idx) out[p] = key[s];
        else if ((int64_t)p < k) idx[p] = (int64_t)(uint32_t)key[s];
    }
}

inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
constexpr size_t kTotalsBytes = 6 * 256 * 4;

// Sorts as `a` says; returns the buffer that holds the result (a selection writes idx instead).
cudaError_t sort_launches(const SortArgs& a, void* scratch, int64_t k, int64_t* idx, u64** result, cudaStream_t st) {
    const int nblocks = (int)((a.N + kTile - 1) / kTile);
    char* p = static_cast<char*>(scratch);
    u64* in = reinterpret_cast<u64*>(p);
    u64* out = reinterpret_cast<u64*>(p + align256((size_t)a.N * 8));
    unsigned* totals = reinterpret_cast<unsigned*>(p + 2 * align256((size_t)a.N * 8));
    unsigned* hist = totals + kTotalsBytes / 4;
    cudaError_t e = cudaMemsetAsync(totals, 0, kTotalsBytes, st);
    if (e != cudaSuccess) return e;
    k_make_keys<<<(unsigned)((a.N + kThreads - 1) / kThreads), kThreads, 0, st>>>(a, in);
    const int passes = (a.by_score ? 4 : 0) + a.label_passes;
    for (int pass = 0; pass < passes; ++pass) {
        k_histogram<<<nblocks, kThreads, 0, st>>>(a, in, pass, hist, nblocks, totals);
        k_scan<<<256, kThreads, 0, st>>>(hist, nblocks, totals + pass * 256);
        k_scatter<<<nblocks, kThreads, 0, st>>>(a, in, pass, hist, nblocks, out, k, pass == passes - 1 ? idx : nullptr);
        u64* t = in;
        in = out;
        out = t;
    }
    if (result) *result = in;
    return cudaGetLastError();
}

// ---- classes with more than one label pass, or more rows than a cluster takes ------------------------------------------
__global__ void __launch_bounds__(256) k_class_count(const int* __restrict__ labels, int64_t N, int C, unsigned* __restrict__ counts) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= N) return;
    const int lab = labels[i];
    if (lab >= 0 && lab < C) atomicAdd(&counts[lab], 1u);      // integer counts: the result does not depend on order
}

// In place: counts[0 .. C - 1] -> first place of each class, [C] = the number of rows with a class. One block.
__global__ void __launch_bounds__(1024) k_class_starts(unsigned* __restrict__ c, int C) {
    __shared__ unsigned ws[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned carry = 0;
    for (int b0 = 0; b0 <= C; b0 += 1024) {
        const unsigned v = b0 + tid < C ? c[b0 + tid] : 0u;
        unsigned x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) ws[warp] = x;
        __syncthreads();
        unsigned before = 0, sum = 0;
        for (int w = 0; w < 32; ++w) {
            if (w < warp) before += ws[w];
            sum += ws[w];
        }
        if (b0 + tid <= C) c[b0 + tid] = carry + before + x - v;
        carry += sum;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(256) k_order_of_keys(const u64* __restrict__ keys, int64_t N, unsigned* __restrict__ order) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i < N) order[i] = (unsigned)(uint32_t)keys[i];
}

// keys (or rows alone): rows grouped by class, best first; the first kc[c] of class c go to offs[c] ...
template <typename Key>
__global__ void __launch_bounds__(256) k_class_pick(const Key* __restrict__ keys, const int* __restrict__ labels, int64_t N, int C,
                                                    const unsigned* __restrict__ starts, const long long* __restrict__ kc,
                                                    const long long* __restrict__ offs, int64_t* __restrict__ out) {
    chain_wait();
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= N) return;
    const u64 key = keys[i];
    const unsigned c = class_of(labels, key, C);
    if (c >= (unsigned)C) return;
    const long long r = i - (int64_t)starts[c];
    if (r < kc[c]) out[offs[c] + r] = (int64_t)(uint32_t)key;
}

int label_passes_of(int C) { return C <= 255 ? 1 : 2; }

}  // namespace

cudaError_t select_scratch_bytes(int64_t N, size_t* bytes) {
    const int64_t nblocks = (N + kTile - 1) / kTile;
    *bytes = 2 * align256((size_t)N * 8) + kTotalsBytes + align256((size_t)nblocks * 256 * 4) + 256;
    return cudaSuccess;
}

// Few rows: ranked. At most half of them wanted: the k-th key first, then the picks ranked or sorted. Otherwise all are sorted.
static bool select_filters(int64_t N, int64_t k) { return N > kRankMax && N <= kFilterMax && k <= N / 2 && k <= kClusterMax; }

int select_launches(int64_t N, int64_t k) { return N <= kRankMax ? 1 : select_filters(N, k) ? 2 : N <= kClusterMax ? 1 : 1 + 3 * 4; }

cudaError_t launch_select(const float* scores, int64_t N, int64_t k, int64_t* idx, void* scratch, cudaStream_t st) {
    if (N <= 0 || k <= 0) return cudaSuccess;
    if (N <= kRankMax) return run_rank(nullptr, scores, (int)N, k, idx, st);
    SortArgs a = {scores, nullptr, N, 0, 1, 0};
    u64* b0 = static_cast<u64*>(scratch);
    u64* b1 = reinterpret_cast<u64*>(static_cast<char*>(scratch) + align256((size_t)N * 8));
    if (select_filters(N, k)) {
        const cudaError_t e = run_top_keys(scores, N, k, b0, st);
        if (e != cudaSuccess) return e;
        if (k <= kRankMax) return run_rank(b0, nullptr, (int)k, k, idx, st);
        a.N = k;
        a.given = true;
        return run_cluster_sort<EMIT_TOPK>(a, b0, b1, k, 0.0, idx, nullptr, nullptr, nullptr, st);
    }
    if (N <= kClusterMax) return run_cluster_sort<EMIT_TOPK>(a, b0, b1, k, 0.0, idx, nullptr, nullptr, nullptr, st);
    return sort_launches(a, scratch, k, idx, nullptr, st);
}

// Brings every kernel that launch_select can take, whatever its sizes, onto the current device: with lazy loading the first launch of
// a kernel loads it, and its code takes device memory.
static cudaError_t load_selection() {
    cudaError_t e = allow_smem((const void*)k_rank, kRankMax * 8);
    if (e == cudaSuccess) e = allow_smem((const void*)k_top_keys, (int)sizeof(FilterShared));
    if (e == cudaSuccess) e = allow_smem((const void*)k_sort_cluster<EMIT_TOPK>, (int)sizeof(ClusterShared));
    for (const void* kernel : {(const void*)k_rank, (const void*)k_top_keys, (const void*)k_sort_cluster<EMIT_TOPK>, (const void*)k_make_keys, (const void*)k_histogram,
                               (const void*)k_scan, (const void*)k_scatter}) {
        cudaFuncAttributes fa;
        if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernel);
    }
    return e;
}

cudaError_t launch_class_order(const int* labels, int64_t N, int C, void* scratch, unsigned* order, unsigned* starts, cudaStream_t st) {
    const SortArgs a = {nullptr, labels, N, C, 0, label_passes_of(C)};
    cudaError_t e = cudaSuccess;
    if (N <= 0 || C > 255 || N > kClusterMax) {
        e = launch_class_starts(labels, N, C, starts, nullptr, st);
        if (e != cudaSuccess || N <= 0) return e;
    }
    if (N <= kClusterMax) {
        u64* b0 = static_cast<u64*>(scratch);
        u64* b1 = reinterpret_cast<u64*>(static_cast<char*>(scratch) + align256((size_t)N * 8));
        return run_cluster_sort<EMIT_ORDER>(a, b0, b1, 0, 0.0, nullptr, order, C <= 255 ? starts : nullptr, nullptr, st);
    }
    u64* keys = nullptr;
    e = sort_launches(a, scratch, 0, nullptr, &keys, st);
    if (e != cudaSuccess) return e;
    k_order_of_keys<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(keys, N, order);
    return cudaGetLastError();
}

int class_order_launches(int64_t N, int C) {
    return N > kClusterMax ? 2 + 1 + 3 * label_passes_of(C) + 1 : C > 255 ? 3 : 1;
}

cudaError_t launch_class_starts(const int* labels, int64_t N, int C, unsigned* starts, unsigned* counts, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(starts, 0, (size_t)(C + 1) * sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    if (N > 0) k_class_count<<<(unsigned)((N + 255) / 256), 256, 0, st>>>(labels, N, C, starts);
    if (counts && (e = cudaMemcpyAsync(counts, starts, (size_t)C * sizeof(unsigned), cudaMemcpyDeviceToDevice, st)) != cudaSuccess) return e;
    k_class_starts<<<1, 1024, 0, st>>>(starts, C);
    return cudaGetLastError();
}

bool class_select_in_one(int64_t N, int C) { return C <= 255 && N > 0 && N <= kClusterMax; }

cudaError_t launch_class_select(const float* scores, const int* labels, int64_t N, int C, double keep_rate, void* scratch, int64_t* idx,
                                long long* kc, cudaStream_t st) {
    const SortArgs a = {scores, labels, N, C, 1, 1};
    u64* b0 = static_cast<u64*>(scratch);
    u64* b1 = reinterpret_cast<u64*>(static_cast<char*>(scratch) + align256((size_t)N * 8));
    return run_cluster_sort<EMIT_PICK>(a, b0, b1, 0, keep_rate, idx, nullptr, nullptr, kc, st);
}

// More than 255 classes: six passes in one launch, or eighteen launches on all SMs. The whole call, 256 classes: 1,000 rows 108 against
// 198 us, 10,000 120 against 230, 50,000 178 against 247, 100,000 252 against 260, 131,072 287 against 268.
constexpr int64_t kPickClusterMax = 98304;
static bool pick_in_cluster(int64_t N, int C) { return C > 255 && N <= kPickClusterMax; }
int class_pick_launches(int64_t N, int C) { return 3 + (pick_in_cluster(N, C) ? 1 : 1 + 3 * (4 + label_passes_of(C))); }

cudaError_t launch_class_pick(const float* scores, const int* labels, int64_t N, int C, void* scratch, const unsigned* starts, const long long* kc,
                              const long long* offs, int64_t* idx, cudaStream_t st) {
    if (N <= 0) return cudaSuccess;
    const SortArgs a = {scores, labels, N, C, 1, label_passes_of(C)};
    const dim3 grid((unsigned)((N + 255) / 256));
    if (pick_in_cluster(N, C)) {
        u64* b0 = static_cast<u64*>(scratch);
        u64* b1 = reinterpret_cast<u64*>(static_cast<char*>(scratch) + align256((size_t)N * 8));
        unsigned* order = static_cast<unsigned*>(scratch);
        const cudaError_t e = run_cluster_sort<EMIT_ORDER>(a, b0, b1, 0, 0.0, nullptr, order, nullptr, nullptr, st);
        return e != cudaSuccess ? e : launch_chained(k_class_pick<unsigned>, grid, dim3(256), 0, st, order, labels, N, C, starts, kc, offs, idx);
    }
    u64* keys = nullptr;
    cudaError_t e = sort_launches(a, scratch, 0, nullptr, &keys, st);
    if (e != cudaSuccess) return e;
    return launch_chained(k_class_pick<u64>, grid, dim3(256), 0, st, keys, labels, N, C, starts, kc, offs, idx);
}

}  // namespace sage

// ------------------------------------------------------------------------------------------------
// sage_select_static: the same selection for callers that must not allocate.
//
// Some callers run where device allocation is off the table: inside a serving or training loop whose
// memory is handed out once at start-up by a pool they do not own, in a process whose remaining device
// memory is deliberately zero, or on a thread that may not take the allocator's locks. sage_select asks
// the stream-ordered allocator for its O(N) scratch on every call; this variant keeps that scratch in
// the library image instead, in the array below, which every device that loads the library holds
// until the process exits.
//
// The array's name is only a host-side stand-in in host code, so its device address is looked up once
// per device (with that device current) and that address is what the kernels get.
// ------------------------------------------------------------------------------------------------
namespace {

constexpr int64_t kStaticMaxN = 262144;    // largest N served without allocating
constexpr size_t kStaticKeyBytes = (size_t)kStaticMaxN * 8;                          // one key array
constexpr size_t kStaticHistBytes = (size_t)((kStaticMaxN + sage::kTile - 1) / sage::kTile) * 256 * 4;
constexpr size_t kStaticScratchBytes = 2 * kStaticKeyBytes + sage::kTotalsBytes + kStaticHistBytes + 256;  // about 4.07 MiB

static __device__ __align__(256) unsigned char g_select_scratch[kStaticScratchBytes];

constexpr int kMaxDevices = 64;
void* g_scratch_addr[kMaxDevices] = {};    // device address of g_select_scratch, per device ordinal
std::mutex g_scratch_mutex;

}  // namespace

extern "C" sage_status_t sage_select_static(const float* scores, int64_t N, double keep_rate, int64_t* idx, int64_t* k_out,
                                            void* cuda_stream) {
    if (N < 0 || !(keep_rate == keep_rate) || (N > 0 && !scores)) {
        sage::set_error_message("sage_select_static: bad argument (negative N, NaN keep_rate or null scores)");
        return SAGE_ERR_INVALID_ARG;
    }
    if (N > kStaticMaxN) {
        char msg[200];
        snprintf(msg, sizeof msg, "sage_select_static: N=%lld exceeds the built-in scratch (at most %lld scores); use sage_select",
                 (long long)N, (long long)kStaticMaxN);
        sage::set_error_message(msg);
        return SAGE_ERR_UNSUPPORTED;
    }
    const int64_t k = sage_select_count(N, keep_rate);
    if (k > 0 && !idx) {
        sage::set_error_message("sage_select_static: null idx");
        return SAGE_ERR_INVALID_ARG;
    }
    if (k > 0) {
        int dev = -1;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
            sage::set_error_message("sage_select_static: no current CUDA device (or ordinal above 63)");
            return SAGE_ERR_CUDA;
        }
        void* scratch = nullptr;
        {
            std::lock_guard<std::mutex> lock(g_scratch_mutex);
            if (!g_scratch_addr[dev]) {       // first call on this device: resolve the array's device address
                void* p = nullptr;
                e = cudaGetSymbolAddress(&p, g_select_scratch);
                if (e != cudaSuccess || !p) {
                    char msg[200];
                    snprintf(msg, sizeof msg, "sage_select_static: cudaGetSymbolAddress failed on device %d: %s", dev,
                             cudaGetErrorString(e));
                    sage::set_error_message(msg);
                    return SAGE_ERR_CUDA;
                }
                e = sage::load_selection();   // other sizes run other kernels
                if (e != cudaSuccess) {
                    char msg[200];
                    snprintf(msg, sizeof msg, "sage_select_static: loading its kernels failed on device %d: %s", dev, cudaGetErrorString(e));
                    sage::set_error_message(msg);
                    return SAGE_ERR_CUDA;
                }
                g_scratch_addr[dev] = p;
            }
            scratch = g_scratch_addr[dev];
        }
        // Nothing in the scratch has to start at zero: the key arrays are written for every i < N before
        // they are read, and what a radix pass counts in is cleared or rewritten by the call.
        e = sage::launch_select(scores, N, k, idx, scratch, static_cast<cudaStream_t>(cuda_stream));
        if (e != cudaSuccess) {
            char msg[200];
            snprintf(msg, sizeof msg, "sage_select_static: launch failed: %s", cudaGetErrorString(e));
            sage::set_error_message(msg);
            return SAGE_ERR_CUDA;
        }
        sage::count_launches(sage::select_launches(N, k));
    }
    if (k_out) *k_out = k;
    return SAGE_OK;
}
