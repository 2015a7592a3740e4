// Host orchestration behind the C ABI: state machine, buffer management and the launch sequences of
// pass 1 (append -> Gram -> eigen/shrink -> rebuild), freeze, pass 2 (project -> normalise -> consensus
// -> score) and selection. No device->host synchronisation happens inside sage_fd_update.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "sage_internal.h"

using namespace sage;

namespace {

thread_local char g_err[512] = "";
std::atomic<long long> g_launches{0};

void set_err(const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof g_err, fmt, ap);
    va_end(ap);
}

#define CU_TRY(expr)                                                                       \
    do {                                                                                   \
        cudaError_t e__ = (expr);                                                          \
        if (e__ != cudaSuccess) {                                                          \
            set_err("%s failed: %s (%s:%d)", #expr, cudaGetErrorString(e__), __FILE__, __LINE__); \
            return e__ == cudaErrorMemoryAllocation ? SAGE_ERR_ALLOC : SAGE_ERR_CUDA;      \
        }                                                                                  \
    } while (0)

#define ST_TRY(expr)                       \
    do {                                   \
        sage_status_t s__ = (expr);        \
        if (s__ != SAGE_OK) return s__;    \
    } while (0)

struct DeviceGuard {
    int prev = -1;
    bool ok = false;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        ok = cudaSetDevice(dev) == cudaSuccess;
    }
    ~DeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

enum State { SKETCHING = 0, FROZEN = 1, SCORING = 2 };

// Kernel classes for the optional per-kernel timing (sage_fd_profile).
enum KClass { K_APPEND = 0, K_GRAM, K_GRAM_REDUCE, K_EIG, K_REBUILD, K_PROJECT, K_PROJECT_REDUCE, K_NORMALISE, K_SCORE, K_NCLASS };

struct Prof {
    unsigned mask = 0;
    std::vector<cudaEvent_t> pool;
    struct Pending { int cls; cudaEvent_t a, b; };
    std::vector<Pending> pending;
    double ms[K_NCLASS] = {};
    int64_t n[K_NCLASS] = {};
    // Adds the pairs whose second event has completed to the sums and recycles their events.
    void fold_finished() {
        size_t keep = 0;
        for (size_t i = 0; i < pending.size(); ++i) {
            Pending& p = pending[i];
            float t = 0.f;
            if (cudaEventQuery(p.b) == cudaSuccess && cudaEventElapsedTime(&t, p.a, p.b) == cudaSuccess) {
                ms[p.cls] += t;
                n[p.cls] += 1;
                pool.push_back(p.a);
                pool.push_back(p.b);
            } else {
                pending[keep++] = p;
            }
        }
        pending.resize(keep);
    }
    cudaEvent_t get() {
        if (!pool.empty()) { cudaEvent_t e = pool.back(); pool.pop_back(); return e; }
        cudaEvent_t e = nullptr;
        cudaEventCreate(&e);
        return e;
    }
};

size_t elem_size(sage_dtype_t dt) { return dt == SAGE_F32 ? 4 : 2; }

// Stream-ordered scratch of the selection entry points, and all memory of a sage_select_from_host call, comes from a pool of
// the library's own that keeps up to kPoolKeep bytes across synchronisations and gives the rest back (the device's default pool
// gives everything back at every synchronisation, and getting it again costs milliseconds). One pool per device, created on first
// use, kept until the process exits.
constexpr unsigned long long kPoolKeep = 1ull << 30;
cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t st) {
    static cudaMemPool_t pools[64] = {};
    static std::mutex mu;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaMallocAsync(p, bytes, st);
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!pools[dev]) {
            cudaMemPoolProps props = {};
            props.allocType = cudaMemAllocationTypePinned;
            props.handleTypes = cudaMemHandleTypeNone;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            cudaMemPool_t pool = nullptr;
            e = cudaMemPoolCreate(&pool, &props);
            if (e != cudaSuccess) return e;
            unsigned long long keep = kPoolKeep;
            e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
            if (e != cudaSuccess) return e;
            pools[dev] = pool;
        }
    }
    return cudaMallocFromPoolAsync(p, bytes, pools[dev], st);
}

// Where the rows of an update come from: a dense matrix (rows, pitch ld), or the two factors of structured last-layer
// rows (q: pitch ldq, C values per row; feat: pitch ldf, F values per row), expanded on the fly.
struct RowSrc {
    const void* rows = nullptr;
    int64_t ld = 0;
    const void* q = nullptr;
    const void* feat = nullptr;
    int64_t ldq = 0, ldf = 0;
    int C = 0, F = 0;
    sage_dtype_t dt = SAGE_F32;
    bool outer() const { return q != nullptr; }
    RowSrc advanced(int64_t k) const {       // the same source, k rows further on
        RowSrc r = *this;
        const size_t es = elem_size(dt);
        if (rows) r.rows = static_cast<const char*>(rows) + (size_t)k * ld * es;
        if (q) r.q = static_cast<const char*>(q) + (size_t)k * ldq * es;
        if (feat) r.feat = static_cast<const char*>(feat) + (size_t)k * ldf * es;
        return r;
    }
    // `take` rows, followed by the first `take2` rows of `more` (same type, pitches and shape)
    cudaError_t append(int64_t take, int64_t D, float* B, int64_t pitch, int dst_row0, cudaStream_t st, const RowSrc* more = nullptr,
                       int64_t take2 = 0) const {
        if (outer())
            return launch_append_outer(q, ldq, feat, ldf, dt, take, C, F, B, pitch, dst_row0, st, more ? more->q : nullptr, more ? more->feat : nullptr, take2);
        return launch_append(rows, dt, take, ld, D, B, pitch, dst_row0, st, more ? more->rows : nullptr, take2);
    }
};

}  // namespace

struct sage_fd {
    bool pooled = false;           // a handle that lives for one call: its memory comes from the library's pool, ordered on pool_stream
    cudaStream_t pool_stream = nullptr;
    int64_t D = 0;
    int ell = 0, m = 0;
    sage_dtype_t dtype = SAGE_F32;
    int device = 0;
    int64_t pitch = 0;             // floats per buffer row (multiple of 32)
    float* B[2] = {nullptr, nullptr};
    int cur = 0;
    int fill = 0;
    int64_t rows_seen = 0;
    State state = SKETCHING;
    int delta_rank = 0, max_sweeps = 30;
    // Gram / eigen workspaces
    float* gram_parts = nullptr;   // split-K partials of the Gram matrix (gram_part_floats floats)
    size_t gram_part_floats = 0;   // at least kGramPartFloats; 74 or 30 slices of m x m for buffers of more than 128 or 256 rows
    float* Wsplit = nullptr;       // rebuild factors split for the tensor cores: wsplit_ld rows x wsplit_ld floats
    int wsplit_ld = 256;           // 256 (buffers of up to 256 rows) or 512
    float* Kmat = nullptr;         // m x m, pitch ldk
    int ldk = 0;                   // m rounded up to 4: the eigen-solve reads rows as float4
    float* Ur = nullptr;           // m x m
    float* eig_work = nullptr;     // eig_work_floats(m) floats
    float* sigma = nullptr;        // ell
    EigInfo* info = nullptr;       // device
    // scoring
    int64_t N_total = 0, next_row = 0, zcap = 0;
    float* zhat = nullptr;
    float* znorm = nullptr;
    float* zwork = nullptr;
    size_t zwork_bytes = 0;
    float* partials = nullptr;
    size_t partials_bytes = 0;
    double* zsum = nullptr;
    float* u = nullptr;
    bool scored = false;           // a scoring pass over N_total rows has finished: zhat holds their normalised projections
    float* bias_t = nullptr;       // structured rows: the bias block of the sketch transposed (C x ell)
    size_t bias_t_bytes = 0;
    float* zred = nullptr;         // projections of a sub-chunk summed over their K slices (when there are many slices)
    size_t zred_bytes = 0;
    bool direct_rows = true;       // option 9: shrink cycles read bfloat16 rows from the caller's memory where the shapes allow it
    bool strict = false;           // option 8: no N x ell store; scores come from a third pass (sage_score_apply)
    bool scored_strict = false;    // the finished pass ran in strict-memory mode: u is known, zhat is not kept
    float* class_U = nullptr;      // class-balanced variant: unit centroids (class_cap x ell) and class sizes
    int* class_counts = nullptr;
    int class_cap = 0, class_num = 0;
    __nv_bfloat16* P16 = nullptr;  // frozen sketch in bf16 (bf16 handles: tensor-core projection operand); with p16_fold
                                   // rows [0, ell) hold bf16(S) and rows [n_pad, n_pad + ell) hold bf16(S - bf16(S))
    int p16_fold = 0, p16_npad = 0;
    float* S32split = nullptr;     // frozen sketch split into tf32 hi / lo rows (fp32 handles with ell <= 64): 128 x pitch
    cudaStream_t side = nullptr;   // appends of the next shrink cycle run here, beside the eigen-solve of the current one
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    int* tc_err = nullptr;         // set by a tensor-core kernel whose bounded wait ran out
    bool use_tc = true;            // option 4: tensor-core kernels where their alignment rules hold
    int eig_variant = 0;           // option 5: 0 the direct eigen-solve, 1 the iterative one
    int64_t launches = 0;
    int64_t tc_launches = 0;       // how many of them were tensor-core (tcgen05) kernels
    int64_t rows_in_place = 0;     // rows that shrink cycles read where the caller held them (never appended)
    Prof prof;
    // Merged form of pass 1 (option 6): P sketches over interleaved row blocks. This handle is sketch 0; sketches
    // 1..P-1 are handles of their own that only sketch (no scoring state). With P > 1 every sketch runs its
    // Gram / eigen-solve / rebuild chain on a stream of its own, so the chains of different sketches overlap.
    int P = 1;
    int64_t block = 0;             // rows per dealt block
    int64_t dealt = 0;             // rows dealt so far (all sketches)
    std::vector<sage_fd*> kids;
    bool sketch_only = false;      // a sub-sketch: no scoring buffers
    cudaStream_t chain = nullptr;  // P > 1: the stream of this sketch's chain (P == 1: the caller's stream)
    bool app_pending = false;      // appends on `side` that the chain stream has not been made to wait for yet
    int64_t in_epoch = -1;         // the update call whose entry event `side` already waits for
    cudaEvent_t ev_in = nullptr;   // the caller's stream at the entry of an update call (sketch 0 only)
    cudaEvent_t ev_rows = nullptr; // end of the current update call on the stream that reads its rows
    cudaEvent_t ev_done = nullptr; // end of the chain stream (joins)
    RowSrc pend;                   // rows of the current update call that still have to be appended, pend_n of them, to row pend_row
    int64_t pend_n = 0;            // (merged form: the dealt blocks cut a cycle's rows in two; one launch appends both parts)
    int pend_row = 0;
    struct Cycle {                 // merged form: a whole cycle's launches as a graph, one per buffer copy (see run_cycle)
        cudaGraphExec_t exec = nullptr;
        int launches = 0, tc_launches = 0;
    } cycle[2];
    int cycles_run = 0;
    bool cycle_graphs = true;
    cudaStream_t used = nullptr;   // the stream that reads rows of the current update call
    bool sketching_in_blocks = false;  // pass 1 works on `blk`; the buffers B hold the frozen sketch only
    size_t buffer_rows = 0;        // rows that the buffers B are allocated for: m, or ell in B[0] alone
    struct Block {                 // shrink cycles in blocks: see block_kernels.cu
        bool able = false;         // the shapes allow it and the memory is there
        int L = 0, M = 0;          // cycles of a block, logical rows of a full one: m + (L - 1)(ell + 1)
        int ldP = 0, ldu = 0, j_pad = 0, slices = 0;
        int64_t pitch = 0, ldT = 0;
        void *memory = nullptr, *row_memory = nullptr;       // what the arrays below lie in: R, T and parts in the second
        __nv_bfloat16 *S[2] = {nullptr, nullptr}, *R = nullptr, *T = nullptr;
        int R_planes = 0;          // planes a row that R and parts are allocated for
        float *P = nullptr, *C = nullptr, *U = nullptr, *K = nullptr, *parts = nullptr;
        int cur = 0;               // S[cur]: the sketch that the block began with
        int s_rows = 0, n_raw = 0; // its rows, and the rows given since
        int n_gram = 0;            // logical rows whose inner products are in P
        int cycles = 0;            // cycles done
        bool step_due = false;     // window `cycles` has not been begun: that waits for its rows
        int np = 0;                // planes a row of R
    } blk;
};

namespace {

void count(sage_fd* h, int k) {
    if (h) h->launches += k;
    g_launches.fetch_add(k, std::memory_order_relaxed);
}

// Runs one launcher; when the class is selected for timing, brackets it with events on the same stream.
template <typename F>
cudaError_t timed(sage_fd* h, int cls, int nlaunch, cudaStream_t st, F&& f) {
    const bool on = h && (h->prof.mask >> cls) & 1u;
    cudaEvent_t a = nullptr, b = nullptr;
    if (on) {
        a = h->prof.get();
        b = h->prof.get();
        cudaEventRecord(a, st);
    }
    const cudaError_t e = f();
    if (on) {
        cudaEventRecord(b, st);
        h->prof.pending.push_back({cls, a, b});
        if (h->prof.pending.size() >= 65536) h->prof.fold_finished();   // never grows without bound if nobody asks for the profile
    }
    count(h, nlaunch);
    return e;
}

constexpr size_t kBlockBytes = (size_t)40 << 30;              // sketches that would take more work cycle by cycle

constexpr size_t kGramPartFloats = (size_t)148 * 128 * 128;   // >= 296 tiles of 64 x 64

int gram_tiles(int r) {
    const int t = (r + 63) / 64;
    return t * t;
}

int pick_splits(int tiles, int64_t K, int64_t min_k) {
    int64_t s = 296 / (tiles > 0 ? tiles : 1);
    const int64_t cap = (K + min_k - 1) / min_k;
    if (s > cap) s = cap;
    if (s < 1) s = 1;
    return (int)s;
}

// Split count for a grid of `tiles` CTAs per split on 148 SMs: the count (each slice keeping at least
// min_k of the contraction) that wastes the least of the last wave; ties go to fewer splits.
int pick_splits_waves(int tiles, int64_t K, int64_t min_k, int max_splits) {
    int64_t cap = K / min_k;
    if (cap > max_splits) cap = max_splits;
    if (cap < 1) cap = 1;
    int best = 1;
    double best_eff = 0.0;
    for (int s = 1; s <= (int)cap; ++s) {
        const int64_t ctas = (int64_t)tiles * s;
        const double eff = (double)ctas / (double)(((ctas + 147) / 148) * 148);
        if (eff > best_eff + 1e-9) { best_eff = eff; best = s; }
    }
    return best;
}

// K slices of the Gram matrix of up to 128 rows, 256 columns and more; with short rows up to 16 slices of 64 and more: the kernel is
// a chain of K tiles there, while many slices cost the reduction what they save (a cycle on rows of 257, 1,024, 3,001 values:
// 34.9 -> 32.7, 58.7 -> 56.3, 82.3 -> 80.8 us; slices of 64 throughout: 5,130 values 107.9 -> 108.8, 20,000 values 113.7 -> 118.2 us).
int gram_splits(int64_t D, int cap) {
    return pick_splits_waves(1, D, D >= 4096 ? 256 : D >= 1024 ? (D + 15) / 16 : 64, cap);
}

// The same for the 74 pairs of SMs that a buffer of more than 128 rows takes (tc_gram_pair.cu). More than 256 rows: 22 slices of each
// tile on the diagonal (8 MMAs a K tile), 30 of the one above it (12 MMAs): 512 rows of 262,144 columns take 304, 293, 295 us with 21, 22,
// 23 slices of the former. At least 64 columns a slice (256 columns: a Gram matrix of 256 rows of 2,052 columns 29.9 instead of 27.4 us).
constexpr int kDiagSlices = 22, kOffSlices = 74 - 2 * kDiagSlices;
void pair_splits(int r, int64_t D, int cap, int* n_diag, int* n_off) {
    const int64_t most = std::max<int64_t>(1, std::min<int64_t>((D + 63) / 64, cap));
    *n_diag = (int)std::min<int64_t>(r > 256 ? kDiagSlices : 74, most);
    *n_off = r > 256 ? (int)std::min<int64_t>(kOffSlices, most) : 0;
}

// After the sketch is frozen: the bf16 copy the tensor-core projection reads (bf16 handles only).
sage_status_t enqueue_freeze_aux(sage_fd* h, cudaStream_t st) {
    if (h->dtype == SAGE_F32 && h->S32split)
        CU_TRY(timed(h, K_APPEND, 1, st, [&] { return launch_split_tf32(h->B[h->cur], h->pitch, h->ell, h->pitch, h->S32split, h->pitch, st); }));
    if (h->dtype == SAGE_BF16 && h->P16)
        CU_TRY(timed(h, K_APPEND, 1, st, [&] {
            return launch_to_bf16(h->B[h->cur], h->pitch, h->ell, h->pitch, h->P16,
                                  h->p16_fold ? h->P16 + (size_t)h->p16_npad * h->pitch : nullptr, h->pitch, st);
        }));
    return SAGE_OK;
}

// Gram of the first r buffer rows -> Kmat (r x r, pitch ldk).
sage_status_t enqueue_gram(sage_fd* h, int r, cudaStream_t st) {
    float* Bc = h->B[h->cur];
    if (h->use_tc) {
        // tensor cores: one tile, or 256 x 256 tiles on pairs of SMs, in as many K slices as fill the SMs
        const int ldc = ((r + 3) / 4) * 4;
        const int64_t stride = (int64_t)r * ldc;
        int cap = (int)(h->gram_part_floats / (size_t)stride);
        if (cap > 148) cap = 148;
        int splits, n_off = 0;
        if (r > 128) pair_splits(r, h->D, cap, &splits, &n_off);
        else splits = gram_splits(h->D, cap);
        cudaError_t e = timed(h, K_GRAM, 1, st, [&] {
            if (r > 128) return launch_tc_gram_pair(Bc, h->pitch, r, h->D, splits, n_off, h->gram_parts, ldc, stride, h->tc_err, st);
            return launch_tc_gemm_nt_x3(Bc, h->pitch, Bc, h->pitch, r, r, h->D, splits, h->gram_parts, ldc, stride, 1, h->tc_err, st);
        });
        if (e == cudaSuccess) {
            h->tc_launches += 1;
            CU_TRY(timed(h, K_GRAM_REDUCE, 1, st, [&] { return launch_gram_sym_reduce(h->gram_parts, splits, stride, r, ldc, h->Kmat, h->ldk, st, n_off); }));
            return SAGE_OK;
        }
        if (e != cudaErrorNotSupported) CU_TRY(e);
        count(h, -1);
    }
    // splits * tiles <= 296, and the partials are stored compactly (pitch r_pad), so they always fit in
    // the 296 tiles of 64 x 64 floats allocated at create.
    const int splits = pick_splits(gram_tiles(r), h->D, 256);
    const int r_pad = ((r + 63) / 64) * 64;
    const int64_t stride = (int64_t)r_pad * r_pad;
    if (splits == 1) {
        CU_TRY(timed(h, K_GRAM, 1, st, [&] { return launch_gemm_nt(Bc, SAGE_F32, h->pitch, Bc, h->pitch, r, r, h->D, 1, h->Kmat, h->ldk, 0, st); }));
    } else {
        CU_TRY(timed(h, K_GRAM, 1, st, [&] {
            return launch_gemm_nt(Bc, SAGE_F32, h->pitch, Bc, h->pitch, r, r, h->D, splits, h->gram_parts, r_pad, stride, st);
        }));
        CU_TRY(timed(h, K_GRAM_REDUCE, 1, st, [&] { return launch_split_reduce(h->gram_parts, splits, stride, r, r, r_pad, h->Kmat, h->ldk, st); }));
    }
    return SAGE_OK;
}

// The appends of the next cycle may run beside the Gram kernel (they write the other buffer copy) and, unless the buffer is large,
// they do: an event recorded inside the chain would end the overlap of its kernels. A buffer beyond the L2 cache keeps them
// behind the Gram kernel, where they do not take its bandwidth (11 M columns: 3.10 s a pass behind it, 3.33 s beside it).
bool appends_early(const sage_fd* h) { return (size_t)h->m * h->pitch * sizeof(float) <= ((size_t)64 << 20); }

// Factor the first r rows and rebuild `keep` rows into the other buffer; rows keep..zero_to-1 are zeroed.
sage_status_t enqueue_factor(sage_fd* h, int r, int do_shrink, int keep, int zero_to, cudaStream_t st) {
    // where the appends of the next cycle may start: see sketch_feed
    const bool fork = !(h->chain && st == h->chain), early = fork && appends_early(h);
    if (early) CU_TRY(cudaEventRecord(h->ev_fork, st));
    ST_TRY(enqueue_gram(h, r, st));
    if (fork && !early) CU_TRY(cudaEventRecord(h->ev_fork, st));       // from here on HBM is idle until the rebuild
    const int j_pad = ((keep + 15) / 16) * 16;
    const bool tc_rebuild = h->use_tc && h->Wsplit && keep > 0 && j_pad <= h->wsplit_ld / 2 && r <= h->wsplit_ld;
    CU_TRY(timed(h, K_EIG, eig_launches(r, h->eig_variant), st, [&] {
        return launch_eig_shrink(h->Kmat, h->ldk, r, do_shrink, h->delta_rank, keep, h->Ur, h->m, h->sigma, h->ell, h->eig_work,
                                 h->max_sweeps, h->info, tc_rebuild ? h->Wsplit : nullptr, h->wsplit_ld, j_pad, h->eig_variant, st);
    }));
    const int m_total = zero_to > keep ? zero_to : keep;
    bool done = false;
    if (tc_rebuild) {
        cudaError_t e = timed(h, K_REBUILD, 1, st, [&] {
            return launch_tc_rebuild(h->Wsplit, h->wsplit_ld, j_pad, h->B[h->cur], h->B[1 - h->cur], h->pitch, h->D, r, keep, h->tc_err, st);
        });
        if (e == cudaSuccess) {
            done = true;
            h->tc_launches += 1;
            if (m_total > keep)
                CU_TRY(cudaMemsetAsync(h->B[1 - h->cur] + (size_t)keep * h->pitch, 0, (size_t)(m_total - keep) * h->pitch * sizeof(float), st));
        } else if (e != cudaErrorNotSupported) {
            CU_TRY(e);
        } else {
            count(h, -1);
        }
    }
    if (!done)
        CU_TRY(timed(h, K_REBUILD, 1, st, [&] {
            return launch_rebuild(h->Ur, h->m, h->B[h->cur], h->B[1 - h->cur], h->pitch, h->D, r, keep, m_total, st);
        }));
    h->cur = 1 - h->cur;
    h->fill = keep;
    return SAGE_OK;
}

cudaError_t dev_malloc(const sage_fd* h, void** p, size_t bytes) {
    return h->pooled ? scratch_alloc(p, bytes, h->pool_stream) : cudaMalloc(p, bytes);
}
cudaError_t dev_free(const sage_fd* h, void* p) {
    if (!p) return cudaSuccess;
    return h->pooled ? cudaFreeAsync(p, h->pool_stream) : cudaFree(p);
}

sage_status_t ensure(const sage_fd* h, float** p, size_t* have, size_t need) {
    if (*have >= need) return SAGE_OK;
    if (*p) CU_TRY(dev_free(h, *p));
    *p = nullptr;
    *have = 0;
    CU_TRY(dev_malloc(h, reinterpret_cast<void**>(p), need));
    *have = need;
    return SAGE_OK;
}

sage_status_t check_handle(const sage_fd* h) {
    if (!h) {
        set_err("null handle");
        return SAGE_ERR_INVALID_ARG;
    }
    return SAGE_OK;
}

}  // namespace

namespace {
// A graph that a thread puts together launch by launch, each behind the one before it: no stream is captured, so that whatever
// other threads do meanwhile (a synchronisation of the device ends every capture that is open in the process) does not concern it.
struct Recorder {
    cudaGraph_t graph = nullptr;
    cudaGraphNode_t last = nullptr;
    int launches = 0;
};
thread_local Recorder* g_recorder = nullptr;
}  // namespace

namespace sage {
cudaError_t launch_any(const void* kernel, const LaunchShape& shape, void** args, cudaStream_t st) {
    if (Recorder* r = g_recorder) {
        cudaGraphNodeParams p = {};
        p.type = cudaGraphNodeTypeKernel;
        p.kernel.func = const_cast<void*>(kernel);
        p.kernel.gridDim = shape.grid;
        p.kernel.blockDim = shape.block;
        p.kernel.sharedMemBytes = (unsigned)shape.smem;
        p.kernel.kernelParams = args;
        cudaGraphEdgeData edge = {};
        if (shape.chained) {
            edge.from_port = cudaGraphKernelNodePortProgrammatic;
            edge.type = cudaGraphDependencyTypeProgrammatic;
        }
        cudaGraphNode_t node = nullptr;
        cudaError_t e = cudaGraphAddNode_v2(&node, r->graph, r->last ? &r->last : nullptr, r->last ? &edge : nullptr, r->last ? 1 : 0, &p);
        if (e == cudaSuccess && shape.cluster > 1) {
            cudaLaunchAttributeValue v = {};
            v.clusterDim.x = shape.cluster;
            v.clusterDim.y = v.clusterDim.z = 1;
            e = cudaGraphKernelNodeSetAttribute(node, cudaLaunchAttributeClusterDimension, &v);
        }
        r->last = node;
        r->launches += 1;
        return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = shape.grid;
    cfg.blockDim = shape.block;
    cfg.dynamicSmemBytes = shape.smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    cfg.attrs = at;
    if (shape.chained) {
        at[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (shape.cluster > 1) {
        at[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        at[cfg.numAttrs].val.clusterDim.x = shape.cluster;
        at[cfg.numAttrs].val.clusterDim.y = 1;
        at[cfg.numAttrs++].val.clusterDim.z = 1;
    }
    return cudaLaunchKernelExC(&cfg, kernel, args);
}
cudaError_t allow_smem(const void* kernel, int bytes, int regs) {
    // set once per kernel and device, which is remembered: an array, as this runs below entry points that must not throw
    struct Seen { const void* kernel; int dev, bytes; };
    static std::mutex mu;
    static Seen seen[256];
    static int n_seen = 0;
    int dev = 0;
    const cudaError_t e0 = cudaGetDevice(&dev);
    if (e0 != cudaSuccess) return e0;
    std::lock_guard<std::mutex> lock(mu);
    for (int i = 0; i < n_seen; ++i)
        if (seen[i].kernel == kernel && seen[i].dev == dev && seen[i].bytes >= bytes) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    if (regs > 0) {
        cudaFuncAttributes fa;
        e = cudaFuncGetAttributes(&fa, kernel);
        if (e != cudaSuccess) return e;
        if (fa.numRegs != regs) return cudaErrorInvalidKernelImage;
    }
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && n_seen < 256) seen[n_seen++] = {kernel, dev, bytes};
    return e;
}
void set_error_message(const char* msg) { set_err("%s", msg); }
void count_launches(int k) { count(nullptr, k); }
}  // namespace sage

extern "C" {

const char* sage_status_string(sage_status_t s) {
    switch (s) {
        case SAGE_OK: return "ok";
        case SAGE_ERR_INVALID_ARG: return "invalid argument";
        case SAGE_ERR_BAD_STATE: return "call not allowed in this state";
        case SAGE_ERR_ALLOC: return "allocation failed";
        case SAGE_ERR_CUDA: return "CUDA error";
        case SAGE_ERR_UNSUPPORTED: return "unsupported size";
        case SAGE_ERR_NOT_CONVERGED: return "eigen-solver did not converge";
        case SAGE_ERR_NONFINITE: return "non-finite input";
    }
    return "unknown status";
}

const char* sage_last_error(void) { return g_err; }
const char* sage_version(void) { return "sage-b200 0.1 (sm_100a)"; }
int64_t sage_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

int64_t sage_select_count(int64_t N, double keep_rate) {
    if (N <= 0 || !(keep_rate == keep_rate)) return 0;
    double k = std::floor(keep_rate * (double)N + 0.5);
    if (k < 0.0) k = 0.0;
    if (k > (double)N) k = (double)N;
    return (int64_t)k;
}

// Forgets the graphs of the cycles, where an option changes that their launches hold (which kernels, delta's rank; the iterative
// solve is not in graphs); waits for the device if there are any.
static void drop_cycles(sage_fd* s) {
    if (s->cycle[0].exec || s->cycle[1].exec) cudaDeviceSynchronize();
    for (sage_fd::Cycle& c : s->cycle) {
        if (c.exec) cudaGraphExecDestroy(c.exec);
        c = sage_fd::Cycle();
    }
    s->cycles_run = 0;
    for (sage_fd* k : s->kids) drop_cycles(k);
}

static bool block_setup(sage_fd* h);
static void block_free(sage_fd* h);
static cudaError_t alloc_buffers(sage_fd* h, size_t rows);
enum Form { BY_OPTIONS, BY_CYCLES, IN_BLOCKS };
static sage_status_t settle_form(sage_fd* h, Form form = BY_OPTIONS);

static sage_status_t create_handle(sage_fd_t** out, int64_t D, int32_t ell, sage_dtype_t row_dtype, int device, bool sketch_only,
                                   bool pooled = false, cudaStream_t pool_stream = nullptr) {
    if (!out || D < 1 || (row_dtype != SAGE_F32 && row_dtype != SAGE_BF16) || device < 0) {
        set_err("sage_fd_create: bad argument (out=%p D=%lld dtype=%d device=%d)", (void*)out, (long long)D, (int)row_dtype, device);
        return SAGE_ERR_INVALID_ARG;
    }
    if (ell < 2 || ell > 256) {
        set_err("sage_fd_create: ell=%d outside [2, 256]", ell);
        return ell < 2 ? SAGE_ERR_INVALID_ARG : SAGE_ERR_UNSUPPORTED;
    }
    DeviceGuard g(device);
    if (!g.ok) {
        set_err("sage_fd_create: cannot select CUDA device %d: %s", device, cudaGetErrorString(cudaGetLastError()));
        return SAGE_ERR_CUDA;
    }
    sage_fd* h = new (std::nothrow) sage_fd();
    if (!h) return SAGE_ERR_ALLOC;
    h->pooled = pooled;
    h->pool_stream = pool_stream;
    h->D = D;
    h->ell = ell;
    h->m = 2 * ell;
    h->dtype = row_dtype;
    h->device = device;
    h->delta_rank = ell;
    h->sketch_only = sketch_only;
    h->block = ell + 1;
    h->pitch = ((D + 31) / 32) * 32;
    h->ldk = (h->m + 3) & ~3;
    const size_t mm = (size_t)h->m * h->ldk * sizeof(float);
    auto fail = [&](cudaError_t e, const char* what) {
        set_err("sage_fd_create: %s failed: %s", what, cudaGetErrorString(e));
        sage_fd_destroy(h);
        return e == cudaErrorMemoryAllocation ? SAGE_ERR_ALLOC : SAGE_ERR_CUDA;
    };
    cudaError_t e;
    h->sketching_in_blocks = block_setup(h);
    if ((e = alloc_buffers(h, h->sketching_in_blocks ? ell : h->m)) != cudaSuccess) return fail(e, "cudaMalloc(buffer)");
    h->gram_part_floats = kGramPartFloats;
    const size_t slices = h->m > 256 ? kOffSlices : h->m > 128 ? 74 : 0;
    if (slices * h->m * ((h->m + 3) / 4 * 4) > h->gram_part_floats) h->gram_part_floats = slices * h->m * ((h->m + 3) / 4 * 4);
    if ((e = dev_malloc(h, (void**)&h->gram_parts, h->gram_part_floats * sizeof(float))) != cudaSuccess) return fail(e, "cudaMalloc(gram)");
    h->wsplit_ld = h->m <= 256 ? 256 : 512;
    if ((e = dev_malloc(h, (void**)&h->Wsplit, (size_t)h->wsplit_ld * h->wsplit_ld * sizeof(float))) != cudaSuccess)
        return fail(e, "cudaMalloc(W)");
    // rows of the split factors beyond the ones an eigen-solve writes are read by the rebuild's MMA (and ignored by its
    // epilogue): they must hold finite values
    if ((e = cudaMemsetAsync(h->Wsplit, 0, (size_t)h->wsplit_ld * h->wsplit_ld * sizeof(float), pool_stream)) != cudaSuccess) return fail(e, "cudaMemset");
    if ((e = dev_malloc(h, (void**)&h->Kmat, mm)) != cudaSuccess) return fail(e, "cudaMalloc(K)");
    if ((e = dev_malloc(h, (void**)&h->Ur, mm)) != cudaSuccess) return fail(e, "cudaMalloc(U)");
    if ((e = dev_malloc(h, (void**)&h->eig_work, eig_work_floats(h->m) * sizeof(float))) != cudaSuccess)
        return fail(e, "cudaMalloc(eig)");
    if ((e = dev_malloc(h, (void**)&h->sigma, ell * sizeof(float))) != cudaSuccess) return fail(e, "cudaMalloc(sigma)");
    if ((e = dev_malloc(h, (void**)&h->info, sizeof(EigInfo))) != cudaSuccess) return fail(e, "cudaMalloc(info)");
    if (!sketch_only) {
        if ((e = dev_malloc(h, (void**)&h->zsum, 256 * sizeof(double))) != cudaSuccess) return fail(e, "cudaMalloc(zsum)");
        if ((e = dev_malloc(h, (void**)&h->u, 256 * sizeof(float))) != cudaSuccess) return fail(e, "cudaMalloc(u)");
    }
    if ((e = dev_malloc(h, (void**)&h->tc_err, sizeof(int))) != cudaSuccess) return fail(e, "cudaMalloc(err)");
    if ((e = cudaStreamCreateWithFlags(&h->side, cudaStreamNonBlocking)) != cudaSuccess) return fail(e, "cudaStreamCreate");
    for (cudaEvent_t* ev : {&h->ev_fork, &h->ev_join, &h->ev_in, &h->ev_rows, &h->ev_done})
        if ((e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming)) != cudaSuccess) return fail(e, "cudaEventCreate");
    if ((e = cudaMemsetAsync(h->tc_err, 0, sizeof(int), pool_stream)) != cudaSuccess) return fail(e, "cudaMemset");
    if (row_dtype == SAGE_BF16 && !sketch_only) {
        // Two-term bf16 sketch (16 significant bits) for short rows, where the rounding errors of a one-term
        // sketch would average over too few terms; long rows take the one-term sketch (half the operand traffic).
        h->p16_npad = ((ell + 15) / 16) * 16;
        h->p16_fold = (2 * h->p16_npad <= 256 && D < 16384) ? 1 : 0;
        const size_t prow = h->p16_fold ? 2 * (size_t)h->p16_npad : (size_t)ell;
        if ((e = dev_malloc(h, (void**)&h->P16, prow * h->pitch * sizeof(__nv_bfloat16))) != cudaSuccess) return fail(e, "cudaMalloc(P16)");
        if ((e = cudaMemsetAsync(h->P16, 0, prow * h->pitch * sizeof(__nv_bfloat16), pool_stream)) != cudaSuccess) return fail(e, "cudaMemset");
    }
    if (row_dtype == SAGE_F32 && ell <= 64 && !sketch_only) {
        // fp32 rows, small sketch: the projection multiplies the rows against the sketch pre-split into tf32 hi / lo rows
        if ((e = dev_malloc(h, (void**)&h->S32split, (size_t)128 * h->pitch * sizeof(float))) != cudaSuccess) return fail(e, "cudaMalloc(S split)");
        if ((e = cudaMemsetAsync(h->S32split, 0, (size_t)128 * h->pitch * sizeof(float), pool_stream)) != cudaSuccess) return fail(e, "cudaMemset");
    }
    if ((e = cudaMemsetAsync(h->info, 0, sizeof(EigInfo), pool_stream)) != cudaSuccess) return fail(e, "cudaMemset");
    if ((e = cudaMemsetAsync(h->sigma, 0, ell * sizeof(float), pool_stream)) != cudaSuccess) return fail(e, "cudaMemset");
    if (!pooled && (e = cudaDeviceSynchronize()) != cudaSuccess) return fail(e, "cudaDeviceSynchronize");
    *out = h;
    return SAGE_OK;
}

sage_status_t sage_fd_create(sage_fd_t** out, int64_t D, int32_t ell, sage_dtype_t row_dtype, int device) {
    return create_handle(out, D, ell, row_dtype, device, false);
}

void sage_fd_destroy(sage_fd_t* h) {
    if (!h) return;
    DeviceGuard g(h->device);
    cudaDeviceSynchronize();
    for (sage_fd* k : h->kids) sage_fd_destroy(k);
    h->kids.clear();
    drop_cycles(h);
    if (h->chain) cudaStreamDestroy(h->chain);
    for (cudaEvent_t ev : {h->ev_in, h->ev_rows, h->ev_done})
        if (ev) cudaEventDestroy(ev);
    void* memory[] = {h->B[0], h->B[1], h->gram_parts, h->Wsplit, h->Kmat, h->Ur, h->eig_work, h->sigma, h->info, h->zhat, h->znorm, h->zwork,
                      h->partials, h->zred, h->bias_t, h->zsum, h->u, h->class_U, h->class_counts, h->P16, h->S32split, h->tc_err};
    for (void* p : memory) dev_free(h, p);
    block_free(h);
    if (h->side) cudaStreamDestroy(h->side);
    if (h->ev_fork) cudaEventDestroy(h->ev_fork);
    if (h->ev_join) cudaEventDestroy(h->ev_join);
    for (auto& p : h->prof.pending) {
        cudaEventDestroy(p.a);
        cudaEventDestroy(p.b);
    }
    for (cudaEvent_t e : h->prof.pool) cudaEventDestroy(e);
    delete h;
}

sage_status_t sage_fd_reset(sage_fd_t* h) {
    ST_TRY(check_handle(h));
    DeviceGuard g(h->device);
    CU_TRY(cudaDeviceSynchronize());
    CU_TRY(cudaMemset(h->info, 0, sizeof(EigInfo)));
    CU_TRY(cudaMemset(h->sigma, 0, h->ell * sizeof(float)));
    CU_TRY(cudaMemset(h->tc_err, 0, sizeof(int)));
    h->fill = 0;
    h->rows_seen = 0;
    h->dealt = 0;
    h->cur = 0;
    h->scored = false;
    h->scored_strict = false;
    h->state = SKETCHING;
    h->launches = 0;
    h->tc_launches = 0;
    h->rows_in_place = 0;
    h->app_pending = false;
    h->in_epoch = -1;
    h->pend = RowSrc();
    h->pend_n = 0;
    h->used = nullptr;
    h->blk.s_rows = h->blk.n_raw = h->blk.n_gram = h->blk.cycles = 0;
    h->blk.step_due = false;
    h->blk.np = h->dtype == SAGE_F32 ? 3 : 1;
    for (sage_fd* k : h->kids) ST_TRY(sage_fd_reset(k));
    return settle_form(h);
}

sage_status_t sage_fd_set_option(sage_fd_t* h, int key, double value) {
    ST_TRY(check_handle(h));
    if (key == 3) {                          // per-kernel event timing mask: allowed at any time
        h->prof.mask = (unsigned)value & ((1u << K_NCLASS) - 1u);
        for (sage_fd* k : h->kids) k->prof.mask = h->prof.mask;
        return SAGE_OK;
    }
    if (key == 4) {                          // 0: CUDA-core kernels only, 1: tensor-core kernels where possible
        DeviceGuard g(h->device);
        if (h->use_tc != (value != 0.0)) drop_cycles(h);
        h->use_tc = value != 0.0;
        for (sage_fd* k : h->kids) k->use_tc = h->use_tc;
        return h->state == SKETCHING ? settle_form(h) : SAGE_OK;
    }
    if (key == 9) {                          // 1: whole shrink cycles read their new rows in place (no append), 0: always append
        h->direct_rows = value != 0.0;
        for (sage_fd* k : h->kids) k->direct_rows = h->direct_rows;
        return SAGE_OK;
    }
    if (key == 8) {                          // strict-memory scoring: no N x ell store, scores from a third pass
        if (h->state == SCORING) {
            set_err("sage_fd_set_option: a scoring pass is open");
            return SAGE_ERR_BAD_STATE;
        }
        h->strict = value != 0.0;
        return SAGE_OK;
    }
    if (key == 5) {                          // eigen-solve kernel family (same algorithm, same results up to rounding order)
        h->eig_variant = value != 0.0 ? 1 : 0;
        for (sage_fd* k : h->kids) k->eig_variant = h->eig_variant;
        return SAGE_OK;
    }
    if (h->dealt != 0 || h->state != SKETCHING) {
        set_err("sage_fd_set_option: options must be set before the first update");
        return SAGE_ERR_BAD_STATE;
    }
    const int v = (int)value;
    if (key == 1 && v >= 2 && v <= h->m - 1) {
        DeviceGuard g(h->device);
        if (h->delta_rank != v) drop_cycles(h);
        h->delta_rank = v;
        for (sage_fd* k : h->kids) k->delta_rank = v;
        return settle_form(h);
    }
    if (key == 2 && v >= 1 && v <= 1000) {
        h->max_sweeps = v;
        for (sage_fd* k : h->kids) k->max_sweeps = v;
        return SAGE_OK;
    }
    if (key == 6 && v >= 1 && v <= 64 && (double)v == value) {      // number of sketches of the merged form of pass 1
        if (v != h->P) {
            DeviceGuard g(h->device);
            cudaDeviceSynchronize();
            for (sage_fd* k : h->kids) sage_fd_destroy(k);
            h->kids.clear();
            if (v == 1 && h->chain) {
                cudaStreamDestroy(h->chain);
                h->chain = nullptr;
            }
        }
        h->P = v;
        return settle_form(h);
    }
    if (key == 7 && v >= 1 && v <= (1 << 20) && (double)v == value) { // rows per dealt block of the merged form
        h->block = v;
        return SAGE_OK;
    }
    set_err("sage_fd_set_option: unknown key %d or value %g out of range", key, value);
    return SAGE_ERR_INVALID_ARG;
}

// ---- shrink cycles in blocks (block_kernels.cu) ----------------------------------------------------------------
//
// A block's rows are read twice, for their inner products and when the kept rows are formed at its end; the solves in between run on
// small matrices. Where a block ends depends on the number of rows given since the reset only, and every product is formed in the same
// order whenever its rows came: the sketch does not depend on how the rows are cut into calls, to the bit. Rows of a block that is not
// complete when an update returns stay in the store (as rows of an incomplete cycle stay in the buffer otherwise).

// Cycles of a block: as many as make 352 new rows, at least 4. Per cycle the kernels that read the rows cost 1 / L of a launch that takes
// little longer for more rows; beyond that the inner products among a block's rows, which grow with the square, take over: 4 cycles where
// rows are long (ell 64, 11.2 M values: 5 cycles are 544 planes and a third block of 256 of them, 2.3 ms of Gram and rebuild a cycle; 4: 2.0). The
// first block ends with the first shrink.
static int block_cycles(int64_t D, int ell) { return D >= ((int64_t)1 << 18) ? 4 : std::max(4, 352 / (ell + 1)); }
static int block_cycles_now(const sage_fd* h) { return h->blk.s_rows < h->ell - 1 ? 1 : h->blk.L; }

static BlockMap block_full_map(const sage_fd* h, int np, bool first) {
    const int s_rows = first ? 0 : h->ell - 1;
    BlockMap m = block_map(s_rows, np, (first ? h->m : h->blk.M) - s_rows, 0);
    m.P += 64;                                     // a part of the rows in place: two places' surplus more
    return m;
}
static int block_most_tiles(const sage_fd* h, int np) {
    return std::max(block_tiles(block_full_map(h, np, false), 0), block_tiles(block_full_map(h, np, true), 0));
}
// K slices of a block's inner products: fixed for a handle, as the sums must not depend on how many rows a launch has. The number with
// which the tiles of a full block end soonest on 74 pairs of SMs, and to a quarter those of a launch with an eighth of them (the first block,
// the freeze, rows of short calls); a slice costs 6 K tiles besides its own, and a partial tile 0.35 in the reduction. Measured, Gram +
// reduction of a full block and of the first one, us: 262,144 values, ell 256: 2 slices 919 + 200, 875; 8 (taken) 939 + 227, 238;
// 20: 961 + 317, 109. 51,300 values, ell 128: 2: 195 + 80, 187; 6: 83 + 83, 76 (7 taken); 20: 83 + 106, 37. 5,130 fp32 values, ell 64:
// 1: 52 + 59, 50; 4 (taken): 27 + 61, 25; 12: 38 + 75, 24.
static int block_slices(int64_t D, int tiles) {
    const int nkt = (int)((D + 63) / 64);
    int best = 1;
    double best_cost = 1e300;
    for (int s = 1; s <= std::min(nkt, 74); ++s) {
        const double each = (double)((nkt + s - 1) / s) + 6.0;
        const double cost = ((tiles * s + 73) / 74 + 0.25 * ((std::max(1, tiles / 8) * s + 73) / 74)) * each + 0.35 * tiles * s;
        if (cost < best_cost) { best_cost = cost; best = s; }
    }
    return best;
}

static void block_free(sage_fd* h) {
    auto& k = h->blk;
    dev_free(h, k.memory);
    dev_free(h, k.row_memory);
    k = sage_fd::Block();
}

// One allocation for several arrays, each on a 1,024-byte boundary.
struct Arena {
    struct Part {
        void** at;
        size_t begin;
    } part[8];
    int n = 0;
    size_t bytes = 0;
    void add(void* at, size_t size) {              // at: the address of the array's pointer
        part[n++] = {static_cast<void**>(at), bytes};
        bytes += (size + 1023) & ~(size_t)1023;
    }
    cudaError_t allocate(sage_fd* h, void** memory) {
        const cudaError_t e = dev_malloc(h, memory, bytes);
        for (int i = 0; i < n && e == cudaSuccess; ++i) *part[i].at = static_cast<char*>(*memory) + part[i].begin;
        return e;
    }
};

// Memory of the rows' planes, of what multiplies them and of their partial inner products, for np planes a row.
static cudaError_t block_alloc_rows(sage_fd* h, int np) {
    auto& k = h->blk;
    k.ldT = (std::max(block_full_map(h, np, false).P, block_full_map(h, np, true).P) + 63) / 64 * 64;
    k.R_planes = np;
    Arena a;
    a.add(&k.R, (size_t)np * k.M * k.pitch * sizeof(__nv_bfloat16));
    a.add(&k.T, (size_t)3 * k.j_pad * k.ldT * sizeof(__nv_bfloat16));
    a.add(&k.parts, (size_t)block_most_tiles(h, np) * k.slices * 65536 * sizeof(float));
    return a.allocate(h, &k.row_memory);
}

static sage_fd::Block block_shape(const sage_fd* h) {
    sage_fd::Block k;
    k.L = block_cycles(h->D, h->ell);
    k.M = h->m + (k.L - 1) * (h->ell + 1);
    k.ldP = (k.M + 3) & ~3;
    k.ldu = (h->m + 3) & ~3;
    k.j_pad = (h->ell + 31) / 32 * 32;
    k.pitch = (h->D + 63) / 64 * 64;
    k.np = h->dtype == SAGE_F32 ? 3 : 1;
    return k;
}

// Sets blk up; false where blocks do not apply (then nothing is allocated).
static bool block_setup(sage_fd* h) {
    if (!launch_block_gram || h->sketch_only) return false;
    auto& k = h->blk;
    k = block_shape(h);
    const int np = k.np;
    k.slices = block_slices(h->D, block_tiles(block_full_map(h, np, false), 0));
    const size_t s_bytes = (size_t)3 * (h->ell - 1) * k.pitch * sizeof(__nv_bfloat16);
    const size_t bytes = 2 * s_bytes + (size_t)np * k.M * k.pitch * sizeof(__nv_bfloat16) + (size_t)block_most_tiles(h, np) * k.slices * 65536 * sizeof(float);
    cudaError_t e = bytes <= kBlockBytes ? cudaSuccess : cudaErrorMemoryAllocation;
    Arena a;
    a.add(&k.S[0], s_bytes);
    a.add(&k.S[1], s_bytes);
    a.add(&k.P, (size_t)k.M * k.ldP * sizeof(float));
    a.add(&k.C, (size_t)h->ell * k.ldP * sizeof(float));
    a.add(&k.U, (size_t)(k.L + 1) * h->m * k.ldu * sizeof(float));
    a.add(&k.K, (size_t)2 * h->m * h->ldk * sizeof(float));
    if (e == cudaSuccess) e = a.allocate(h, &k.memory);
    // (rows of bfloat16 handles may be products of two factors: room for two planes at once, unless they are very long)
    if (e == cudaSuccess) e = block_alloc_rows(h, bytes <= kBlockBytes / 64 ? std::max(np, 2) : np);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        block_free(h);
        return false;
    }
    k.able = true;
    return true;
}

static BlockSmall block_small(const sage_fd* h) {
    const auto& k = h->blk;
    return {h->m, h->ell - 1, h->ell + 1, k.P, k.ldP, k.C, k.U, k.ldu, (int64_t)h->m * k.ldu, k.K, (int64_t)h->m * h->ldk, h->ldk, k.U + (size_t)k.L * h->m * k.ldu};
}
static BlockSource block_source(const sage_fd* h, const void* in_place, int64_t ld) {
    return {h->blk.S[h->blk.cur], h->blk.R, h->blk.pitch, in_place, ld};
}

// The rows of R with np planes each from here on (structured rows of a bfloat16 handle are products: two planes).
static sage_status_t block_widen(sage_fd* h, int np, cudaStream_t st) {
    auto& k = h->blk;
    if (k.np >= np) return SAGE_OK;
    if (k.R_planes < np || k.n_raw > 0) {                  // new memory, as rows that are there move apart
        __nv_bfloat16* old = k.R;
        void* old_memory = k.row_memory;
        const int have = k.np;
        k.row_memory = nullptr;
        k.R = k.T = nullptr;
        k.parts = nullptr;
        CU_TRY(cudaStreamSynchronize(st));
        const cudaError_t e = block_alloc_rows(h, np);
        if (e == cudaSuccess && k.n_raw > 0) {
            CU_TRY(cudaMemsetAsync(k.R, 0, (size_t)np * k.n_raw * k.pitch * 2, st));
            for (int i = 0; i < k.n_raw; ++i)
                CU_TRY(cudaMemcpyAsync(k.R + (size_t)i * np * k.pitch, old + (size_t)i * have * k.pitch, (size_t)have * k.pitch * 2, cudaMemcpyDeviceToDevice, st));
        }
        CU_TRY(cudaStreamSynchronize(st));
        CU_TRY(dev_free(h, old_memory));
        CU_TRY(e);
    }
    k.np = np;
    return SAGE_OK;
}

static sage_status_t block_gram(sage_fd* h, const BlockMap& map, const BlockSource& src, cudaStream_t st) {
    auto& k = h->blk;
    const int first = k.n_gram, nl = block_rows(map);
    if (first >= nl) return SAGE_OK;
    CU_TRY(timed(h, K_GRAM, 1, st, [&] { return launch_block_gram(src, map, first, h->D, k.slices, k.parts, h->tc_err, st); }));
    h->tc_launches += 1;
    CU_TRY(timed(h, K_GRAM_REDUCE, 1, st, [&] { return launch_block_gram_reduce(k.parts, map, first, k.slices, k.P, k.ldP, st); }));
    k.n_gram = nl;
    return SAGE_OK;
}

static sage_status_t block_solve(sage_fd* h, int r, int do_shrink, int keep, cudaStream_t st) {
    auto& k = h->blk;
    const int c = k.cycles;
    const float* K = c == 0 ? k.P : k.K + (size_t)(c & 1) * h->m * h->ldk;
    CU_TRY(timed(h, K_EIG, eig_launches(r, h->eig_variant), st, [&] {
        return launch_eig_shrink(K, c == 0 ? k.ldP : h->ldk, r, do_shrink, h->delta_rank, keep, k.U + (size_t)c * h->m * k.ldu, k.ldu, h->sigma, h->ell, h->eig_work,
                                 h->max_sweeps, h->info, nullptr, 0, 0, h->eig_variant, st);
    }));
    return SAGE_OK;
}

// The kept rows after ncyc cycles: into the other sketch copy, or in fp32 to rows 0 .. keep - 1 of `rows`.
static sage_status_t block_rebuild(sage_fd* h, const BlockMap& map, const BlockSource& src, int carried, int ncyc, int r_last, int keep, float* rows, cudaStream_t st) {
    auto& k = h->blk;
    CU_TRY(timed(h, K_REBUILD, 2, st, [&] {
        const cudaError_t e = launch_block_factors(block_small(h), map, carried, ncyc, r_last, keep, k.T, k.j_pad, k.ldT, st);
        if (e != cudaSuccess) return e;
        return launch_block_rebuild(src, map, h->D, k.T, k.j_pad, k.ldT, keep, rows ? nullptr : k.S[1 - k.cur], rows, rows ? h->pitch : k.pitch, h->tc_err, st);
    }));
    h->tc_launches += 1;
    return SAGE_OK;
}

// The step into window `cycles`, if it is due; columns from `before` on are new and have all cycles before them.
static sage_status_t block_step(sage_fd* h, int before, cudaStream_t st) {
    auto& k = h->blk;
    const int c = k.cycles;
    if (!k.step_due && (c == 0 || k.n_gram == before)) return SAGE_OK;
    const bool due = k.step_due;
    k.step_due = false;
    CU_TRY(timed(h, K_GRAM_REDUCE, block_step_launches(h->m, due), st, [&] {
        return launch_block_step(block_small(h), due ? c - 1 : 0, c, due ? h->ell - 1 + c * (h->ell + 1) : before, before, k.n_gram, due, st);
    }));
    return SAGE_OK;
}

// Products of the rows that have come since the last cycle, and what they give of the open window. (In one launch with a step that waited
// for them: 6,000 rows of 5,130, ell 64, in calls of 64 rows 12.2 ms with a launch each, 11.8 so.)
static sage_status_t block_catch_up(sage_fd* h, const BlockMap& map, const BlockSource& src, cudaStream_t st) {
    const int before = h->blk.n_gram;
    ST_TRY(block_gram(h, map, src, st));
    return block_step(h, before, st);
}

// Ends an open block at its last cycle: the kept rows are formed, the rows behind them (fewer than a cycle's) begin the next block.
static sage_status_t block_end_early(sage_fd* h, cudaStream_t st) {
    auto& k = h->blk;
    if (k.cycles == 0) return SAGE_OK;
    const int keep = h->ell - 1, raw = h->m + (k.cycles - 1) * (h->ell + 1) - k.s_rows, rest = k.n_raw - raw;
    const BlockMap map = block_map(k.s_rows, k.np, raw, 0);
    ST_TRY(block_step(h, k.n_gram, st));
    ST_TRY(block_rebuild(h, map, block_source(h, nullptr, 0), k.cycles, k.cycles, h->m, keep, nullptr, st));
    const size_t row = (size_t)k.np * k.pitch;             // (raw >= ell + 1 > rest: the two ranges lie apart)
    if (rest > 0) CU_TRY(cudaMemcpyAsync(k.R, k.R + raw * row, rest * row * sizeof(__nv_bfloat16), cudaMemcpyDeviceToDevice, st));
    k.cur = 1 - k.cur;
    k.s_rows = keep;
    k.n_raw = rest;
    k.n_gram = k.cycles = 0;
    return SAGE_OK;
}

static sage_status_t block_feed(sage_fd* h, RowSrc src, int64_t n, cudaStream_t st) {
    auto& k = h->blk;
    const int keep = h->ell - 1, step = h->ell + 1, m = h->m;
    if (src.outer() && h->dtype == SAGE_BF16) ST_TRY(block_widen(h, 2, st));
    while (n > 0) {
        const int L = block_cycles_now(h), M = m + (L - 1) * step;
        const int nl = k.s_rows + k.n_raw, take = (int)std::min<int64_t>(n, M - nl);
        // Rows that complete a block stay where the caller holds them, from one on whose plane has the place it would have in the store:
        // sums over planes are formed 16 at a time.
        int at = M;                                // the first logical row in place
        if (take == M - nl && h->direct_rows && k.np == 1 && !src.outer() && (reinterpret_cast<uintptr_t>(src.rows) & 15u) == 0 && ((src.ld * 2) & 15) == 0) {
            at = std::min(M, k.s_rows + (k.n_raw + 31) / 32 * 32);
            if (L > 1) h->rows_in_place += (M - at) / step * step;       // whole cycles
        }
        const int copied = std::min(take, at - nl);
        if (copied > 0)
            CU_TRY(timed(h, K_APPEND, 1, st, [&] {
                if (src.outer()) return launch_block_append_outer(src.q, src.ldq, src.feat, src.ldf, src.dt, copied, src.C, src.F, k.R, k.pitch, k.np, k.n_raw, st);
                return launch_block_append(src.rows, src.dt, copied, src.ld, h->D, k.R, k.pitch, k.np, k.n_raw, st);
            }));
        const RowSrc rest = src.advanced(copied);
        const BlockMap map = block_map(k.s_rows, k.np, k.n_raw + copied, take - copied);
        const BlockSource from = block_source(h, rest.rows, rest.ld);
        k.n_raw += take;
        h->rows_seen += take;
        src = src.advanced(take);
        n -= take;
        if (nl + take >= m + k.cycles * step) ST_TRY(block_catch_up(h, map, from, st));
        while (k.cycles < L && nl + take >= m + k.cycles * step) {
            ST_TRY(block_solve(h, m, 1, keep, st));
            const int c = ++k.cycles;
            k.step_due = c < L;
            if (c < L && nl + take >= m + c * step) ST_TRY(block_step(h, k.n_gram, st));
        }
        if (k.cycles == L) {
            ST_TRY(block_rebuild(h, map, from, L - 1, L, m, keep, nullptr, st));
            k.cur = 1 - k.cur;
            k.s_rows = keep;
            k.n_raw = k.n_gram = k.cycles = 0;
            k.step_due = false;
        }
    }
    h->fill = k.s_rows + k.n_raw - k.cycles * step;
    return SAGE_OK;
}

// An update that the caller captures has to leave the handle as it found it where its rows are a number of whole cycles, so that it can
// be replayed: it begins and ends between blocks, with the sketch in the same copy. What is open before it is ended at once, on a
// stream of the library's own, and not by the graph.
static sage_status_t block_feed_captured(sage_fd* h, RowSrc src, int64_t n, cudaStream_t st) {
    auto& k = h->blk;
    if (k.cycles > 0) {
        allow_work_beside_capture(true);
        auto now = [&]() -> sage_status_t {
            CU_TRY(cudaStreamWaitEvent(h->side, h->ev_rows, 0));
            ST_TRY(block_end_early(h, h->side));
            CU_TRY(cudaStreamSynchronize(h->side));
            return SAGE_OK;
        };
        const sage_status_t rc = now();
        allow_work_beside_capture(false);
        ST_TRY(rc);
    }
    const int cur = k.cur;
    ST_TRY(block_feed(h, src, n, st));
    ST_TRY(block_end_early(h, st));
    if (k.cur != cur) {
        CU_TRY(cudaMemcpyAsync(k.S[cur], k.S[k.cur], (size_t)3 * k.s_rows * k.pitch * sizeof(__nv_bfloat16), cudaMemcpyDeviceToDevice, st));
        k.cur = cur;
    }
    return SAGE_OK;
}

// The freeze: one more solve on the open window, its rows straight to the frozen sketch.
static sage_status_t block_freeze(sage_fd* h, cudaStream_t st) {
    auto& k = h->blk;
    const int r = h->fill, ell = h->ell, do_shrink = r > ell ? 1 : 0, keep = do_shrink ? ell - 1 : std::min(r, ell);
    if (r > 0) {
        const BlockMap map = block_map(k.s_rows, k.np, k.n_raw, 0);
        const BlockSource src = block_source(h, nullptr, 0);
        ST_TRY(block_catch_up(h, map, src, st));
        ST_TRY(block_solve(h, r, do_shrink, keep, st));
        ST_TRY(block_rebuild(h, map, src, k.cycles, k.cycles + 1, r, keep, h->B[0], st));
    } else {
        CU_TRY(cudaMemsetAsync(h->sigma, 0, ell * sizeof(float), st));
    }
    if (keep < ell) CU_TRY(cudaMemsetAsync(h->B[0] + (size_t)keep * h->pitch, 0, (size_t)(ell - keep) * h->pitch * sizeof(float), st));
    h->cur = 0;
    h->fill = keep;
    return SAGE_OK;
}

// Buffers of `rows` rows: two of m rows for cycle-by-cycle sketching, or one of ell rows for the frozen sketch.
static cudaError_t alloc_buffers(sage_fd* h, size_t rows) {
    const size_t bytes = rows * h->pitch * sizeof(float);
    cudaError_t e = dev_malloc(h, (void**)&h->B[0], bytes);
    if (e == cudaSuccess && rows == (size_t)h->m) e = dev_malloc(h, (void**)&h->B[1], bytes);
    h->buffer_rows = rows;
    return e;
}

// Rows that B holds become a block's first rows, or the other way round, when an option changes the form of pass 1. Sketching only.
static sage_status_t settle_form(sage_fd* h, Form form) {
    bool want = !h->sketch_only && h->P == 1 && h->use_tc && h->delta_rank == h->ell && launch_block_gram != nullptr;
    if (form != BY_OPTIONS) want = form == IN_BLOCKS;
    if (want == h->sketching_in_blocks) return SAGE_OK;
    DeviceGuard g(h->device);
    CU_TRY(cudaDeviceSynchronize());
    auto& k = h->blk;
    const int keep = h->ell - 1;
    if (want) {
        if (!block_setup(h)) return SAGE_OK;       // cycle by cycle, as before
        k.s_rows = std::min(h->fill, keep);
        const int rest = h->fill - k.s_rows;
        if (rest > 0 && h->dtype == SAGE_BF16) ST_TRY(block_widen(h, 2, nullptr));       // rows of either kind
        CU_TRY(launch_block_append(h->B[h->cur], SAGE_F32, k.s_rows, h->pitch, h->D, k.S[0], k.pitch, 3, 0, nullptr));
        CU_TRY(launch_block_append(h->B[h->cur] + (size_t)k.s_rows * h->pitch, SAGE_F32, rest, h->pitch, h->D, k.R, k.pitch, k.np, 0, nullptr));
        k.n_raw = rest;
        h->sketching_in_blocks = true;
    } else {
        if (h->buffer_rows != (size_t)h->m) {
            for (float*& b : h->B) {
                CU_TRY(dev_free(h, b));
                b = nullptr;
            }
            if (h->fill == 0) block_free(h);       // first, where memory is short
            CU_TRY(alloc_buffers(h, h->m));
        }
        h->cur = 0;
        if (h->fill > 0) {
            ST_TRY(block_end_early(h, nullptr));
            CU_TRY(launch_block_unpack(k.S[k.cur], k.pitch, 3, k.s_rows, h->D, h->B[0], h->pitch, nullptr));
            CU_TRY(launch_block_unpack(k.R, k.pitch, k.np, k.n_raw, h->D, h->B[0] + (size_t)k.s_rows * h->pitch, h->pitch, nullptr));
            CU_TRY(cudaDeviceSynchronize());
        }
        block_free(h);
        h->sketching_in_blocks = false;
    }
    CU_TRY(cudaDeviceSynchronize());
    return SAGE_OK;
}

// ---- one sketch: feed rows, factor, freeze ------------------------------------------------------------------
//
// Streams of a sketch: every append runs on its `side` stream, the Gram / eigen-solve / rebuild chain on `chain` (the
// caller's stream for a single sketch, the sketch's own stream in the merged form). An append writes rows
// [fill, fill + take) of the current buffer copy and touches nothing the eigen-solve or the rebuild of the previous
// shrink reads or writes (the rebuild fills rows [0, keep) of the same copy), so appends run beside the eigen-solve,
// which leaves HBM idle. The side stream starts before the Gram kernel of the previous shrink, or for large buffers
// after it (appends_early): either way after the rebuild before, which read the copy now being filled. The chain waits
// for the appends before the next Gram kernel. In the merged form the appends run on the chain stream itself.

static sage_status_t sketch_join_appends(sage_fd* s, cudaStream_t chain) {
    if (s->app_pending) {
        CU_TRY(cudaEventRecord(s->ev_join, s->side));
        CU_TRY(cudaStreamWaitEvent(chain, s->ev_join, 0));
        s->app_pending = false;
    }
    return SAGE_OK;
}

// A full buffer's cycle in the merged form. Sixteen chains share the device and one host thread enqueues for all of them, so the
// host bounds a pass over short rows: the launches of a cycle (the same every time but for the buffer copy) are put into a graph
// once the sketch has run a few, one host call instead of five. A stream that the caller is capturing takes the launches themselves.
static sage_status_t run_cycle(sage_fd* s, cudaStream_t chain) {
    const int keep = s->delta_rank - 1;
    constexpr int kDirect = 8;                 // cycles before a graph pays
    auto direct = [&] { return enqueue_factor(s, s->m, 1, keep, 0, chain); };
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    CU_TRY(cudaStreamIsCapturing(chain, &capturing));
    if (capturing != cudaStreamCaptureStatusNone || !s->cycle_graphs || s->eig_variant != 0) return direct();
    sage_fd::Cycle& c = s->cycle[s->cur];
    if (!c.exec) {
        if (s->cycles_run < kDirect) {
            ++s->cycles_run;
            return direct();
        }
        const int cur = s->cur, fill = s->fill;
        const int64_t l0 = s->launches, t0 = s->tc_launches;
        Recorder rec;
        cudaError_t e = cudaGraphCreate(&rec.graph, 0);
        sage_status_t rc = SAGE_ERR_CUDA;
        if (e == cudaSuccess) {
            g_recorder = &rec;
            rc = direct();
            g_recorder = nullptr;
            if (rc == SAGE_OK) e = cudaGraphInstantiate(&c.exec, rec.graph, 0);
            cudaGraphDestroy(rec.graph);
        }
        c.launches = rec.launches;
        c.tc_launches = (int)(s->tc_launches - t0);
        g_launches.fetch_sub(s->launches - l0, std::memory_order_relaxed);
        s->cur = cur;                          // nothing has run yet
        s->fill = fill;
        s->launches = l0;
        s->tc_launches = t0;
        if (e != cudaSuccess || rc != SAGE_OK) {
            (void)cudaGetLastError();
            c = sage_fd::Cycle();
            s->cycle_graphs = false;
            return direct();
        }
    }
    CU_TRY(cudaGraphLaunch(c.exec, chain));
    count(s, c.launches);
    s->tc_launches += c.tc_launches;
    s->cur = 1 - s->cur;
    s->fill = keep;
    return SAGE_OK;
}

static sage_status_t sketch_factor(sage_fd* s, int r, int do_shrink, int keep, int zero_to, cudaStream_t chain) {
    ST_TRY(sketch_join_appends(s, chain));
    if (s->chain && chain == s->chain && r == s->m && do_shrink && zero_to == 0 && keep == s->delta_rank - 1 && s->prof.mask == 0)
        return run_cycle(s, chain);
    ST_TRY(enqueue_factor(s, r, do_shrink, keep, zero_to, chain));
    if (!(s->chain && chain == s->chain)) CU_TRY(cudaStreamWaitEvent(s->side, s->ev_fork, 0));
    return SAGE_OK;
}

// A whole shrink cycle whose new rows (m - fill of them, bfloat16, pitch ld) are read where the caller holds them instead of
// being appended first: the Gram and rebuild kernels take rows 0 .. fill - 1 from the buffer and the rest from `rows`
// (same arithmetic, same results as the appended form). *done = false (and nothing enqueued) when the kernels do not
// support the shape: the caller then appends as usual.
static sage_status_t sketch_factor_direct(sage_fd* s, const void* rows, int64_t ld, cudaStream_t chain, bool* done) {
    *done = false;
    const int r = s->m, old_rows = s->fill, n_new = s->m - s->fill, keep = s->delta_rank - 1;
    const int j_pad = ((keep + 15) / 16) * 16;
    if (!s->use_tc || !s->Wsplit || r > 128 || keep != old_rows || keep <= 0 || (old_rows + 1) % 32 != 0 || r % 32 != 0 ||
        j_pad > s->wsplit_ld / 2 || r > s->wsplit_ld || j_pad > 64 || (reinterpret_cast<uintptr_t>(rows) & 15u) || ((ld * 2) & 15))
        return SAGE_OK;
    ST_TRY(sketch_join_appends(s, chain));
    const int ldc = ((r + 3) / 4) * 4;
    const int64_t stride = (int64_t)r * ldc;
    int cap = (int)(s->gram_part_floats / (size_t)stride);
    if (cap > 148) cap = 148;
    const int splits = gram_splits(s->D, cap);
    float* Bc = s->B[s->cur];
    cudaError_t e = timed(s, K_GRAM, 1, chain, [&] {
        return launch_tc_gram_direct(Bc, s->pitch, old_rows, rows, ld, n_new, s->D, splits, s->gram_parts, ldc, stride, s->tc_err, chain);
    });
    if (e == cudaErrorNotSupported) {
        count(s, -1);
        return SAGE_OK;
    }
    CU_TRY(e);
    s->tc_launches += 1;
    CU_TRY(timed(s, K_GRAM_REDUCE, 1, chain, [&] { return launch_gram_sym_reduce(s->gram_parts, splits, stride, r, ldc, s->Kmat, s->ldk, chain); }));
    CU_TRY(cudaEventRecord(s->ev_fork, chain));
    CU_TRY(timed(s, K_EIG, eig_launches(r, s->eig_variant), chain, [&] {
        return launch_eig_shrink(s->Kmat, s->ldk, r, 1, s->delta_rank, keep, s->Ur, s->m, s->sigma, s->ell, s->eig_work, s->max_sweeps, s->info,
                                 s->Wsplit, s->wsplit_ld, j_pad, s->eig_variant, chain);
    }));
    e = timed(s, K_REBUILD, 1, chain, [&] {
        return launch_tc_rebuild_direct(s->Wsplit, s->wsplit_ld, j_pad, Bc, s->B[1 - s->cur], s->pitch, s->D, r, keep, rows, ld, n_new, s->tc_err,
                                        chain);
    });
    if (e == cudaErrorNotSupported) {
        // the factors exist already: bring the rows into the buffer after all and rebuild from there
        count(s, -1);
        CU_TRY(timed(s, K_APPEND, 1, chain, [&] { return launch_append(rows, SAGE_BF16, n_new, ld, s->D, Bc, s->pitch, old_rows, chain); }));
        CU_TRY(timed(s, K_REBUILD, 1, chain, [&] {
            return launch_tc_rebuild(s->Wsplit, s->wsplit_ld, j_pad, Bc, s->B[1 - s->cur], s->pitch, s->D, r, keep, s->tc_err, chain);
        }));
    } else {
        CU_TRY(e);
    }
    s->tc_launches += 1;
    s->cur = 1 - s->cur;
    s->fill = keep;
    CU_TRY(cudaStreamWaitEvent(s->side, s->ev_fork, 0));
    *done = true;
    return SAGE_OK;
}

static sage_status_t flush_pending(sage_fd* s, cudaStream_t as) {
    if (s->pend_n == 0) return SAGE_OK;
    const int64_t n = s->pend_n;
    s->pend_n = 0;
    CU_TRY(timed(s, K_APPEND, 1, as, [&] { return s->pend.append(n, s->D, s->B[s->cur], s->pitch, s->pend_row, as); }));
    return SAGE_OK;
}

// Appends n rows of type dt and shrinks whenever the buffer fills. e_in (may be null): the event after which `rows`
// are valid; epoch identifies the update call it belongs to. on_chain: appends run on the chain stream itself (used
// where the rows to append are produced by that stream). Leaves the stream that reads the rows in s->used.
static sage_status_t sketch_feed(sage_fd* s, RowSrc src, int64_t n, cudaStream_t chain, cudaEvent_t e_in, int64_t epoch, bool on_chain) {
    // merged form: the appends run on the chain stream too (the chains of the other sketches fill the device while this
    // one waits, and half as many streams keep every chain on a hardware queue of its own)
    const bool from_caller = !on_chain;
    if (s->chain && chain == s->chain) on_chain = true;
    cudaStream_t as = on_chain ? chain : s->side;
    if (from_caller && e_in && s->in_epoch != epoch) {
        CU_TRY(cudaStreamWaitEvent(as, e_in, 0));
        s->in_epoch = epoch;
    }
    bool appended = false;
    auto body = [&]() -> sage_status_t {
        while (n > 0) {
            const int64_t room = s->m - s->fill;
            const int64_t take = n < room ? n : room;
            // a whole cycle's rows at hand, bfloat16, on the caller's own stream: no append, the kernels read them in place
            if (s->direct_rows && from_caller && !s->chain && !src.outer() && src.dt == SAGE_BF16 && take == room && s->fill > 0 &&
                s->fill == s->delta_rank - 1) {
                bool direct = false;
                ST_TRY(sketch_factor_direct(s, src.rows, src.ld, chain, &direct));
                if (direct) {
                    s->rows_in_place += take;
                    s->rows_seen += take;
                    src = src.advanced(take);
                    n -= take;
                    continue;
                }
            }
            if (on_chain && from_caller && s->pend_n == 0) {     // appended together with the next part, or by flush_pending
                s->pend = src;
                s->pend_n = take;
                s->pend_row = s->fill;
            } else if (s->pend_n > 0) {
                const int64_t first = s->pend_n;
                s->pend_n = 0;
                CU_TRY(timed(s, K_APPEND, 1, as, [&] { return s->pend.append(first, s->D, s->B[s->cur], s->pitch, s->pend_row, as, &src, take); }));
            } else {
                CU_TRY(timed(s, K_APPEND, 1, as, [&] { return src.append(take, s->D, s->B[s->cur], s->pitch, s->fill, as); }));
            }
            appended = true;
            if (!on_chain) s->app_pending = true;
            s->fill += (int)take;
            s->rows_seen += take;
            src = src.advanced(take);
            n -= take;
            if (s->fill == s->m) ST_TRY(flush_pending(s, as));
            if (s->fill == s->m) ST_TRY(sketch_factor(s, s->m, 1, s->delta_rank - 1, 0, chain));
        }
        return SAGE_OK;
    };
    const sage_status_t rc = body();
    if (appended && from_caller) s->used = as;   // also on the error path: the caller's stream must not run ahead of appends that read `rows`
    return rc;
}

// The freeze of one sketch: orthogonalise what the buffer holds, shrink only if more than ell rows are in use.
// Afterwards s->fill is the number of rows kept (at most ell) and rows up to ell are zero.
static sage_status_t sketch_freeze(sage_fd* s, cudaStream_t chain) {
    ST_TRY(sketch_join_appends(s, chain));
    const int r = s->fill;
    if (r == 0) {
        CU_TRY(cudaMemsetAsync(s->B[s->cur], 0, (size_t)s->ell * s->pitch * sizeof(float), chain));
        CU_TRY(cudaMemsetAsync(s->sigma, 0, s->ell * sizeof(float), chain));
    } else {
        const int do_shrink = r > s->ell ? 1 : 0;
        const int keep = do_shrink ? s->delta_rank - 1 : (r < s->ell ? r : s->ell);
        ST_TRY(sketch_factor(s, r, do_shrink, keep < s->ell ? keep : s->ell, s->ell, chain));
    }
    return SAGE_OK;
}

static sage_fd* sketch_at(sage_fd* h, int p) { return p == 0 ? h : h->kids[(size_t)p - 1]; }

// Creates the sketches 1..P-1 and the chain streams of the merged form (first update after option 6).
static sage_status_t ensure_sketches(sage_fd* h) {
    if (h->P <= 1 || (int)h->kids.size() == h->P - 1) return SAGE_OK;
    for (int p = (int)h->kids.size() + 1; p < h->P; ++p) {
        sage_fd* k = nullptr;
        ST_TRY(create_handle(&k, h->D, h->ell, h->dtype, h->device, true));
        k->delta_rank = h->delta_rank;
        k->max_sweeps = h->max_sweeps;
        k->use_tc = h->use_tc;
        k->eig_variant = h->eig_variant;
        k->prof.mask = h->prof.mask;
        h->kids.push_back(k);
    }
    for (int p = 0; p < h->P; ++p) {
        sage_fd* s = sketch_at(h, p);
        if (!s->chain) CU_TRY(cudaStreamCreateWithFlags(&s->chain, cudaStreamNonBlocking));
    }
    return SAGE_OK;
}

// Algorithm 1, Phase I for n rows from `src` (dense rows or the factors of structured rows): shared by sage_fd_update and
// sage_fd_update_outer.
static sage_status_t update_from(sage_fd* h, RowSrc src, int64_t n, cudaStream_t st) {
    DeviceGuard g(h->device);
    ST_TRY(ensure_sketches(h));
    static std::atomic<long long> epochs{0};
    const int64_t epoch = epochs.fetch_add(1) + 1;
    sage_status_t rc = SAGE_OK;
    if (h->sketching_in_blocks) {
        cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
        CU_TRY(cudaStreamIsCapturing(st, &capturing));
        h->dealt += n;
        if (capturing != cudaStreamCaptureStatusNone) return block_feed_captured(h, src, n, st);
        ST_TRY(block_feed(h, src, n, st));
        CU_TRY(cudaEventRecord(h->ev_rows, st));
        return SAGE_OK;
    }
    CU_TRY(cudaEventRecord(h->ev_in, st));
    if (h->P == 1) {
        rc = sketch_feed(h, src, n, st, h->ev_in, epoch, false);
        h->dealt += n;
    } else {
        // block b of the row stream (counted over all calls) goes to sketch b mod P
        while (n > 0 && rc == SAGE_OK) {
            const int64_t b = h->dealt / h->block;
            const int64_t left_in_block = (b + 1) * h->block - h->dealt;
            const int64_t take = n < left_in_block ? n : left_in_block;
            sage_fd* s = sketch_at(h, (int)(b % h->P));
            rc = sketch_feed(s, src, take, s->chain, h->ev_in, epoch, false);
            h->dealt += take;
            src = src.advanced(take);
            n -= take;
        }
    }
    // the caller's stream continues once every row of this call has been copied into a buffer
    for (int p = 0; p < h->P && p <= (int)h->kids.size(); ++p) {
        sage_fd* s = sketch_at(h, p);
        if (s->used) {
            const sage_status_t fl = flush_pending(s, s->used);
            if (rc == SAGE_OK) rc = fl;
            // every sketch is flushed and joined, whatever failed before: nothing of this call may read its rows later
            auto join = [&]() -> sage_status_t {
                CU_TRY(cudaEventRecord(s->ev_rows, s->used));
                CU_TRY(cudaStreamWaitEvent(st, s->ev_rows, 0));
                return SAGE_OK;
            };
            const sage_status_t jn = join();
            if (rc == SAGE_OK) rc = jn;
            s->used = nullptr;
        }
    }
    return rc;
}

sage_status_t sage_fd_update(sage_fd_t* h, const void* rows, int64_t n, int64_t ld, void* cuda_stream) {
    ST_TRY(check_handle(h));
    if (n < 0 || (n > 0 && (!rows || ld < h->D))) {
        set_err("sage_fd_update: bad argument (rows=%p n=%lld ld=%lld D=%lld)", rows, (long long)n, (long long)ld, (long long)h->D);
        return SAGE_ERR_INVALID_ARG;
    }
    if (h->state != SKETCHING) {
        set_err("sage_fd_update: the sketch is frozen (call sage_fd_reset to start over)");
        return SAGE_ERR_BAD_STATE;
    }
    if (n == 0) return SAGE_OK;
    RowSrc src;
    src.rows = rows;
    src.ld = ld;
    src.dt = h->dtype;
    return update_from(h, src, n, static_cast<cudaStream_t>(cuda_stream));
}

// Checks the arguments of the entry points that take structured last-layer rows.
static sage_status_t check_outer(const sage_fd* h, const char* who, const void* q, int64_t ldq, const void* feat, int64_t ldf, int64_t n,
                                 int32_t C, int32_t F) {
    if (C < 1 || F < 1 || (int64_t)C * F + C != h->D) {
        set_err("%s: C=%d classes x F=%d features + C biases is not the handle's row dimension D=%lld", who, (int)C, (int)F, (long long)h->D);
        return SAGE_ERR_INVALID_ARG;
    }
    if (n < 0 || (n > 0 && (!q || !feat || ldq < C || ldf < F))) {
        set_err("%s: bad argument (q=%p ldq=%lld feat=%p ldf=%lld n=%lld)", who, q, (long long)ldq, feat, (long long)ldf, (long long)n);
        return SAGE_ERR_INVALID_ARG;
    }
    return SAGE_OK;
}

sage_status_t sage_fd_update_outer(sage_fd_t* h, const void* q, int64_t ldq, const void* feat, int64_t ldf, int64_t n, int32_t C, int32_t F,
                                   void* cuda_stream) {
    ST_TRY(check_handle(h));
    ST_TRY(check_outer(h, "sage_fd_update_outer", q, ldq, feat, ldf, n, C, F));
    if (h->state != SKETCHING) {
        set_err("sage_fd_update_outer: the sketch is frozen (call sage_fd_reset to start over)");
        return SAGE_ERR_BAD_STATE;
    }
    if (n == 0) return SAGE_OK;
    RowSrc src;
    src.q = q;
    src.ldq = ldq;
    src.feat = feat;
    src.ldf = ldf;
    src.C = C;
    src.F = F;
    src.dt = h->dtype;
    return update_from(h, src, n, static_cast<cudaStream_t>(cuda_stream));
}

// Makes `cuda_stream` wait for everything the handle has enqueued on streams of its own.
sage_status_t sage_fd_join(sage_fd_t* h, void* cuda_stream) {
    ST_TRY(check_handle(h));
    DeviceGuard g(h->device);
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    for (int p = 0; p <= (int)h->kids.size(); ++p) {
        sage_fd* s = sketch_at(h, p);
        CU_TRY(cudaEventRecord(s->ev_join, s->side));
        CU_TRY(cudaStreamWaitEvent(st, s->ev_join, 0));
        if (s->chain) {
            CU_TRY(cudaEventRecord(s->ev_done, s->chain));
            CU_TRY(cudaStreamWaitEvent(st, s->ev_done, 0));
        }
    }
    return SAGE_OK;
}

sage_status_t sage_fd_finalize(sage_fd_t* h, void* cuda_stream) {
    ST_TRY(check_handle(h));
    if (h->state != SKETCHING) {
        set_err("sage_fd_finalize: already frozen");
        return SAGE_ERR_BAD_STATE;
    }
    DeviceGuard g(h->device);
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const int nsk = (int)h->kids.size() + 1;            // sketches that exist (1 unless the merged form has been fed)
    if (h->sketching_in_blocks) {
        ST_TRY(block_freeze(h, st));
    } else if (nsk == 1) {
        ST_TRY(sketch_freeze(h, (h->P > 1 && h->chain) ? h->chain : st));
    } else {
        // every sketch is frozen on its own, then sketch a absorbs sketch a + s for s = 1, 2, 4, ...: the rows the
        // other one kept are appended to it and it is frozen again (a shrink happens if that fills its buffer)
        for (int p = 0; p < nsk; ++p) ST_TRY(sketch_freeze(sketch_at(h, p), sketch_at(h, p)->chain));
        for (int stride = 1; stride < nsk; stride *= 2)
            for (int a = 0; a + stride < nsk; a += 2 * stride) {
                sage_fd* A = sketch_at(h, a);
                sage_fd* Bs = sketch_at(h, a + stride);
                CU_TRY(cudaEventRecord(Bs->ev_done, Bs->chain));
                CU_TRY(cudaStreamWaitEvent(A->chain, Bs->ev_done, 0));
                if (Bs->fill > 0)
                {
                    RowSrc kept;
                    kept.rows = Bs->B[Bs->cur];
                    kept.ld = Bs->pitch;
                    kept.dt = SAGE_F32;
                    ST_TRY(sketch_feed(A, kept, Bs->fill, A->chain, nullptr, 0, true));
                }
                ST_TRY(sketch_freeze(A, A->chain));
            }
    }
    if (h->P > 1 && h->chain) {                          // merged form: sketch 0 holds the result; back to the caller's stream
        CU_TRY(cudaEventRecord(h->ev_done, h->chain));
        CU_TRY(cudaStreamWaitEvent(st, h->ev_done, 0));
    }
    ST_TRY(enqueue_freeze_aux(h, st));
    h->state = FROZEN;
    EigInfo info;
    int tc_err = 0;
    CU_TRY(cudaMemcpyAsync(&info, h->info, sizeof info, cudaMemcpyDeviceToHost, st));
    CU_TRY(cudaMemcpyAsync(&tc_err, h->tc_err, sizeof tc_err, cudaMemcpyDeviceToHost, st));
    CU_TRY(cudaStreamSynchronize(st));
    for (sage_fd* k : h->kids) {                         // their chains ended before sketch 0's did
        EigInfo ki;
        int kt = 0;
        CU_TRY(cudaMemcpy(&ki, k->info, sizeof ki, cudaMemcpyDeviceToHost));
        CU_TRY(cudaMemcpy(&kt, k->tc_err, sizeof kt, cudaMemcpyDeviceToHost));
        info.flags |= ki.flags;
        tc_err |= kt;
    }
    if (tc_err) {
        set_err("sage_fd_finalize: a tensor-core kernel gave up waiting on its pipeline (results are not valid)");
        return SAGE_ERR_CUDA;
    }
    if (info.flags & kFlagExchangeTimeout) {
        set_err("sage_fd_finalize: an eigen-solve gave up waiting for another thread block of its cluster (results are not valid)");
        return SAGE_ERR_CUDA;
    }
    if (info.flags & kFlagNotConverged) {
        set_err("sage_fd_finalize: an eigen-solve reached the sweep limit (%d)", h->max_sweeps);
        return SAGE_ERR_NOT_CONVERGED;
    }
    if (info.flags & kFlagNonFinite) {
        set_err("sage_fd_finalize: non-finite values were met in the rows of pass 1");
        return SAGE_ERR_NONFINITE;
    }
    return SAGE_OK;
}

sage_status_t sage_fd_sketch(const sage_fd_t* h, const float** S, int64_t* pitch, const float** sigma) {
    ST_TRY(check_handle(h));
    if (h->state == SKETCHING) {
        set_err("sage_fd_sketch: the sketch is not frozen yet");
        return SAGE_ERR_BAD_STATE;
    }
    if (S) *S = h->B[h->cur];
    if (pitch) *pitch = h->pitch;
    if (sigma) *sigma = h->sigma;
    return SAGE_OK;
}

sage_status_t sage_fd_load_sketch(sage_fd_t* h, const float* S, int64_t ld, void* cuda_stream) {
    ST_TRY(check_handle(h));
    if (!S || ld < h->D) {
        set_err("sage_fd_load_sketch: bad argument");
        return SAGE_ERR_INVALID_ARG;
    }
    if (h->state == SCORING) {
        set_err("sage_fd_load_sketch: a scoring pass is open");
        return SAGE_ERR_BAD_STATE;
    }
    DeviceGuard g(h->device);
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    CU_TRY(timed(h, K_APPEND, 1, st, [&] { return launch_append(S, SAGE_F32, h->ell, ld, h->D, h->B[h->cur], h->pitch, 0, st); }));
    CU_TRY(cudaMemsetAsync(h->sigma, 0, h->ell * sizeof(float), st));
    ST_TRY(enqueue_freeze_aux(h, st));
    h->fill = h->ell;
    h->scored = false;
    h->scored_strict = false;
    h->state = FROZEN;
    return SAGE_OK;
}

sage_status_t sage_score_begin(sage_fd_t* h, int64_t N_total, void* cuda_stream) {
    ST_TRY(check_handle(h));
    if (N_total < 0) {
        set_err("sage_score_begin: negative row count");
        return SAGE_ERR_INVALID_ARG;
    }
    if (h->state != FROZEN) {
        set_err("sage_score_begin: needs a frozen sketch and no open scoring pass");
        return SAGE_ERR_BAD_STATE;
    }
    DeviceGuard g(h->device);
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (!h->strict && N_total > h->zcap) {
        CU_TRY(cudaStreamSynchronize(st));
        if (h->zhat) CU_TRY(dev_free(h, h->zhat));
        if (h->znorm) CU_TRY(dev_free(h, h->znorm));
        h->zhat = h->znorm = nullptr;
        h->zcap = 0;
        CU_TRY(dev_malloc(h, (void**)&h->zhat, (size_t)N_total * h->ell * sizeof(float)));
        CU_TRY(dev_malloc(h, (void**)&h->znorm, (size_t)N_total * sizeof(float)));
        h->zcap = N_total;
    }
    CU_TRY(cudaMemsetAsync(h->zsum, 0, 256 * sizeof(double), st));
    h->N_total = N_total;
    h->next_row = 0;
    h->scored = false;
    h->scored_strict = false;
    h->state = SCORING;
    return SAGE_OK;
}

// Projection, normalisation and consensus partials of n rows (sub-chunk by sub-chunk). store_at >= 0: the normalised
// projections go to rows [store_at, store_at + n) of the handle's N x ell store; store_at < 0: to a scratch of one sub-chunk
// (strict-memory mode). accumulate: the rows' sum is added to the consensus sum. scores_out != null (third pass of the
// strict-memory mode): the scores of these rows against the finished consensus are written there.
// Projection, normalisation, consensus partials (and, with scores_out, the scores) of n rows, a sub-chunk at a time.
// Dense rows: `rows` with pitch ld. Structured last-layer rows (outer != nullptr; rows and ld unused): the projection
// factorises over the classes,
//     z_i = S g_i = sum_c q_ic (S_c h_i) + S_b q_i      (S_c: columns [c F, c F + F) of the sketch, S_b: its last C columns),
// so the row g_i is never formed: ONE launch of the projection kernel takes the classes as its K slices (every slice reads
// the same F feature columns, slice c the class block c of the sketch) and leaves the planes T_c = H S_c^T, which a second
// kernel folds with the factors q_ic and the bias block.
static sage_status_t score_rows(sage_fd* h, const void* rows, sage_dtype_t dt, int64_t n, int64_t ld, cudaStream_t st, int64_t store_at,
                                bool accumulate, float* scores_out, const RowSrc* outer = nullptr) {
    const int ell = h->ell;
    const bool structured = outer != nullptr;
    const void* oq = structured ? outer->q : nullptr;
    const int64_t oldq = structured ? outer->ldq : 0;
    const int oC = structured ? outer->C : 0, oF = structured ? outer->F : 0;
    if (structured) {
        rows = outer->feat;
        ld = outer->ldf;
    }
    const int64_t K = structured ? (int64_t)oC * oF : h->D;      // contraction length against the sketch
    const int64_t class_F = structured ? oF : 0;
    int64_t sub_max = 148 * 128;             // one full wave of 128-row tiles
    const char* p = static_cast<const char*>(rows);
    const size_t row_bytes = (size_t)ld * elem_size(dt);
    const float* S = h->B[h->cur];
    // Tensor-core path: bf16 rows against the bf16 copy of the sketch (a one-term bf16 sketch is only used for
    // long rows, where its rounding errors average out).
    const bool tc_ok = h->use_tc && dt == SAGE_BF16 && h->P16 && (h->p16_fold || h->D >= 16384) &&
                       (reinterpret_cast<uintptr_t>(rows) & 15u) == 0 && (row_bytes & 15u) == 0;
    // fp32 rows: the fp32-faithful three-MMA kernel against the fp32 sketch itself (one 128-wide tile of S)
    const bool tc32_ok = h->use_tc && dt == SAGE_F32 && ell <= 128 && (reinterpret_cast<uintptr_t>(rows) & 15u) == 0 &&
                         (row_bytes & 15u) == 0;
    // fp32 rows against a small sketch: the projections of a sub-chunk are small (ell <= 64 floats per row and plane), so
    // up to 8 waves go into one launch (fewer launch-scale overheads per pass)
    if (tc32_ok && h->S32split) sub_max *= 8;
    if (structured) {
        // one plane per class: keep the planes of a sub-chunk within 1 GiB
        const int64_t per_row = (int64_t)oC * ell * (int64_t)sizeof(float);
        int64_t fit = ((int64_t)1 << 30) / per_row / 128 * 128;
        if (fit < 128) fit = 128;
        if (sub_max > fit) sub_max = fit;
    }
    for (int64_t r0 = 0; r0 < n; r0 += sub_max) {
        const int64_t sub = (n - r0 < sub_max) ? n - r0 : sub_max;
        const size_t nb = (size_t)((sub + 63) / 64);
        ST_TRY(ensure(h, &h->partials, &h->partials_bytes, nb * ell * sizeof(float)));
        if (store_at < 0 && sub > h->zcap) {         // strict-memory mode: normalised projections of one sub-chunk only
            CU_TRY(cudaStreamSynchronize(st));
            if (h->zhat) CU_TRY(dev_free(h, h->zhat));
            if (h->znorm) CU_TRY(dev_free(h, h->znorm));
            h->zhat = h->znorm = nullptr;
            h->zcap = 0;
            CU_TRY(dev_malloc(h, (void**)&h->zhat, (size_t)sub * ell * sizeof(float)));
            CU_TRY(dev_malloc(h, (void**)&h->znorm, (size_t)sub * sizeof(float)));
            h->zcap = sub;
        }
        const size_t zred = (size_t)sub * ell * sizeof(float);
        bool done = false;
        const float* Zparts = nullptr;       // the projections of this sub-chunk as nplanes partial planes of sub x ell floats
        int nplanes = 1;
        if (tc32_ok) {
            // sketches of at most 64 rows: a kernel of their own, against the pre-split sketch
            const bool narrow = h->S32split != nullptr;
            const int splits = structured ? oC : pick_splits_waves((int)((sub + 127) / 128), K, 2048, 64);
            const int planes = narrow ? project_planes(sub, K, class_F) : splits;
            ST_TRY(ensure(h, &h->zwork, &h->zwork_bytes, zred * planes));
            float* out = h->zwork;
            cudaError_t e = timed(h, K_PROJECT, 1, st, [&] {
                const float* g = reinterpret_cast<const float*>(p + r0 * row_bytes);
                if (narrow) return launch_tc_project(g, ld, h->S32split, h->pitch, sub, ell, K, class_F, out, (int64_t)sub * ell, h->tc_err, st);
                return launch_tc_gemm_nt_x3(g, ld, S, h->pitch, (int)sub, ell, K, splits, out, ell, (int64_t)sub * ell, 0, h->tc_err, st, class_F);
            });
            if (e == cudaSuccess) {
                done = true;
                h->tc_launches += 1;
                Zparts = out;
                nplanes = planes;
            } else if (e != cudaErrorNotSupported) {
                CU_TRY(e);
            } else {
                count(h, -1);
            }
        }
        if (tc_ok) {
            // row tiles per CTA: as many as TMEM holds (512 columns), fewer when that would leave SMs without work
            const int n_mma = (h->p16_fold ? 2 : 1) * h->p16_npad;
            const int tiles = (int)((sub + 127) / 128);
            int mt = 512 / n_mma >= 4 ? 4 : (512 / n_mma >= 2 ? 2 : 1);
            if (tiles >= 148 && mt > 2) mt = 2;   // measured: pairs of row tiles with two K slices beat single tiles by 25 %
            // rows a page or more apart: the kernel fetches two K tiles per stage (256 bytes per row visit), two row tiles fit
            if (row_bytes >= ((size_t)2 << 20) && mt > 2) mt = 2;
            const int64_t slices_at_least = structured ? oC : (K / 4096 > 0 ? K / 4096 : 1);
            while (mt > 1 && (int64_t)((tiles + mt - 1) / mt) * slices_at_least < 148) mt >>= 1;
            const int splits = structured ? oC : pick_splits_waves((tiles + mt - 1) / mt, K, 4096, 148);
            ST_TRY(ensure(h, &h->zwork, &h->zwork_bytes, zred * splits));
            float* out = h->zwork;
            cudaError_t e = timed(h, K_PROJECT, 1, st, [&] {
                return launch_tc_gemm_nt(p + r0 * row_bytes, SAGE_BF16, ld, h->P16, h->pitch, (int)sub, ell, h->p16_fold, mt, K, splits,
                                         out, ell, (int64_t)sub * ell, h->tc_err, st, class_F);
            });
            if (e == cudaSuccess) {
                done = true;
                h->tc_launches += 1;
                Zparts = out;
                nplanes = splits;
            } else if (e != cudaErrorNotSupported) {
                CU_TRY(e);
            } else {
                count(h, -1);
            }
        }
        if (!done) {
            const int tiles = (int)((sub + 63) / 64) * ((ell + 63) / 64);
            const int splits = structured ? oC : pick_splits(tiles, K, 1024);
            ST_TRY(ensure(h, &h->zwork, &h->zwork_bytes, zred * splits));
            CU_TRY(timed(h, K_PROJECT, 1, st, [&] {
                return launch_gemm_nt(p + r0 * row_bytes, dt, ld, S, h->pitch, (int)sub, ell, K, splits, h->zwork, ell,
                                      (int64_t)sub * ell, st, class_F);
            }));
            Zparts = h->zwork;
            nplanes = splits;
        }
        if (structured) {
            // z = sum_c q_c (T_c + bias column c), classes in ascending order
            ST_TRY(ensure(h, &h->zred, &h->zred_bytes, zred));
            const float* parts = Zparts;
            const int pp = nplanes / oC;
            const char* qsub = static_cast<const char*>(oq) + (size_t)r0 * oldq * elem_size(dt);
            ST_TRY(ensure(h, &h->bias_t, &h->bias_t_bytes, (size_t)oC * ell * sizeof(float)));
            CU_TRY(timed(h, K_PROJECT_REDUCE, 2, st, [&] {
                return launch_outer_combine(qsub, oldq, dt, oC, parts, pp, (int64_t)sub * ell, S + K, h->pitch, h->bias_t, sub, ell, h->zred, st);
            }));
            Zparts = h->zred;
            nplanes = 1;
        }
        // Many K slices (few rows per launch, as in the 512-row chunks of very long rows): summed first by a kernel with a
        // thread per element; the normalise kernel has a warp per row and would walk the slices one after the other.
        if (nplanes > 4) {
            ST_TRY(ensure(h, &h->zred, &h->zred_bytes, zred));
            const float* parts = Zparts;
            const int np = nplanes;
            CU_TRY(timed(h, K_PROJECT_REDUCE, 1, st,
                         [&] { return launch_split_reduce(parts, np, (int64_t)sub * ell, (int)sub, ell, ell, h->zred, ell, st); }));
            Zparts = h->zred;
            nplanes = 1;
        }
        // normalise (summing the K slices of the projection on the way), consensus partials, and in the third pass the scores
        float* zh = store_at >= 0 ? h->zhat + (store_at + r0) * ell : h->zhat;
        float* zn = store_at >= 0 ? h->znorm + (store_at + r0) : h->znorm;
        CU_TRY(timed(h, K_NORMALISE, accumulate ? 2 : 1, st, [&] {
            return launch_normalise(Zparts, nplanes, (int64_t)sub * ell, ell, sub, ell, zh, zn, h->partials, accumulate ? h->zsum : nullptr,
                                    &h->info->flags, st);
        }));
        if (scores_out)
            CU_TRY(timed(h, K_SCORE, 1, st, [&] { return launch_consensus_score(h->zsum, zh, sub, ell, h->u, scores_out + r0, st); }));
    }
    return SAGE_OK;
}


sage_status_t sage_score_chunk(sage_fd_t* h, const void* rows, int64_t n, int64_t ld, int64_t row_offset, void* cuda_stream) {
    ST_TRY(check_handle(h));
    if (h->state != SCORING) {
        set_err("sage_score_chunk: no open scoring pass");
        return SAGE_ERR_BAD_STATE;
    }
    if (n < 0 || (n > 0 && (!rows || ld < h->D)) || row_offset != h->next_row || row_offset + n > h->N_total) {
        set_err("sage_score_chunk: bad argument (n=%lld ld=%lld offset=%lld expected offset=%lld N_total=%lld)", (long long)n,
                (long long)ld, (long long)row_offset, (long long)h->next_row, (long long)h->N_total);
        return SAGE_ERR_INVALID_ARG;
    }
    if (n == 0) return SAGE_OK;
    DeviceGuard g(h->device);
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    ST_TRY(score_rows(h, rows, h->dtype, n, ld, st, h->strict ? -1 : row_offset, true, nullptr));
    h->next_row += n;
    return SAGE_OK;
}

sage_status_t sage_score_chunk_outer(sage_fd_t* h, const void* q, int64_t ldq, const void* feat, int64_t ldf, int64_t n, int32_t C,
                                     int32_t F, int64_t row_offset, void* cuda_stream) {
    ST_TRY(check_handle(h));
    if (h->state != SCORING) {
        set_err("sage_score_chunk_outer: no open scoring pass");
        return SAGE_ERR_BAD_STATE;
    }
    ST_TRY(check_outer(h, "sage_score_chunk_outer", q, ldq, feat, ldf, n, C, F));
    if (row_offset != h->next_row || row_offset + n > h->N_total) {
        set_err("sage_score_chunk_outer: bad argument (n=%lld offset=%lld expected offset=%lld N_total=%lld)", (long long)n,
                (long long)row_offset, (long long)h->next_row, (long long)h->N_total);
        return SAGE_ERR_INVALID_ARG;
    }
    if (n == 0) return SAGE_OK;
    DeviceGuard g(h->device);
    RowSrc src;
    src.q = q;
    src.ldq = ldq;
    src.feat = feat;
    src.ldf = ldf;
    src.C = C;
    src.F = F;
    src.dt = h->dtype;
    ST_TRY(score_rows(h, nullptr, h->dtype, n, 0, static_cast<cudaStream_t>(cuda_stream), h->strict ? -1 : row_offset, true, nullptr, &src));
    h->next_row += n;
    return SAGE_OK;
}

sage_status_t sage_score_end(sage_fd_t* h, float* scores, void* cuda_stream) {
    ST_TRY(check_handle(h));
    if (h->state != SCORING) {
        set_err("sage_score_end: no open scoring pass");
        return SAGE_ERR_BAD_STATE;
    }
    if (h->next_row != h->N_total) {
        set_err("sage_score_end: %lld of %lld rows were given", (long long)h->next_row, (long long)h->N_total);
        return SAGE_ERR_BAD_STATE;
    }
    if (!scores && h->N_total > 0 && !h->strict) {
        set_err("sage_score_end: null scores");
        return SAGE_ERR_INVALID_ARG;
    }
    DeviceGuard g(h->device);
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (h->strict) {     // only the consensus direction is formed here; the scores come from sage_score_apply
        CU_TRY(timed(h, K_SCORE, 1, st, [&] { return launch_consensus_score(h->zsum, h->zhat, 0, h->ell, h->u, nullptr, st); }));
        h->scored_strict = true;
    } else {
        CU_TRY(timed(h, K_SCORE, 1, st, [&] { return launch_consensus_score(h->zsum, h->zhat, h->N_total, h->ell, h->u, scores, st); }));
        h->scored = true;
    }
    h->state = FROZEN;
    return SAGE_OK;
}

sage_status_t sage_score_apply(sage_fd_t* h, const void* rows, int64_t n, int64_t ld, float* scores, void* cuda_stream) {
    ST_TRY(check_handle(h));
    if (h->state != FROZEN || !(h->scored || h->scored_strict)) {
        set_err("sage_score_apply: needs a finished scoring pass (the consensus direction) on this handle");
        return SAGE_ERR_BAD_STATE;
    }
    if (n < 0 || (n > 0 && (!rows || !scores || ld < h->D))) {
        set_err("sage_score_apply: bad argument (n=%lld ld=%lld)", (long long)n, (long long)ld);
        return SAGE_ERR_INVALID_ARG;
    }
    if (n == 0) return SAGE_OK;
    if (h->scored) {     // the N x ell store of the finished pass must survive: this call works in a scratch of its own size class
        set_err("sage_score_apply: the handle keeps the normalised projections of its last pass (option 8 is off); use sage_score");
        return SAGE_ERR_BAD_STATE;
    }
    DeviceGuard g(h->device);
    return score_rows(h, rows, h->dtype, n, ld, static_cast<cudaStream_t>(cuda_stream), -1, false, scores);
}

sage_status_t sage_score(sage_fd_t* h, const void* rows, int64_t n, int64_t ld, float* scores, void* cuda_stream) {
    ST_TRY(sage_score_begin(h, n, cuda_stream));
    sage_status_t s = sage_score_chunk(h, rows, n, ld, 0, cuda_stream);
    if (s != SAGE_OK) {
        h->state = FROZEN;
        return s;
    }
    s = sage_score_end(h, scores, cuda_stream);
    if (s != SAGE_OK) h->state = FROZEN;
    return s;
}

sage_status_t sage_score_outer(sage_fd_t* h, const void* q, int64_t ldq, const void* feat, int64_t ldf, int64_t n, int32_t C, int32_t F,
                               float* scores, void* cuda_stream) {
    ST_TRY(check_handle(h));
    ST_TRY(check_outer(h, "sage_score_outer", q, ldq, feat, ldf, n, C, F));
    ST_TRY(sage_score_begin(h, n, cuda_stream));
    sage_status_t s = sage_score_chunk_outer(h, q, ldq, feat, ldf, n, C, F, 0, cuda_stream);
    if (s != SAGE_OK) {
        h->state = FROZEN;
        return s;
    }
    s = sage_score_end(h, scores, cuda_stream);
    if (s != SAGE_OK) h->state = FROZEN;
    return s;
}

sage_status_t sage_score_intermediates(const sage_fd_t* h, const float** zhat, const float** znorm, const float** u) {
    ST_TRY(check_handle(h));
    if (h->state != FROZEN || !h->zhat || !h->scored) {
        set_err("sage_score_intermediates: no finished scoring pass that kept its projections");
        return SAGE_ERR_BAD_STATE;
    }
    if (zhat) *zhat = h->zhat;
    if (znorm) *znorm = h->znorm;
    if (u) *u = h->u;
    return SAGE_OK;
}

sage_status_t sage_select(const float* scores, int64_t N, double keep_rate, int64_t* idx, int64_t* k_out, void* cuda_stream) {
    if (N < 0 || N >= (1ll << 31) || !(keep_rate == keep_rate) || (N > 0 && !scores)) {
        set_err("sage_select: bad argument (N=%lld keep_rate=%g)", (long long)N, keep_rate);
        return SAGE_ERR_INVALID_ARG;
    }
    const int64_t k = sage_select_count(N, keep_rate);
    if (k > 0 && !idx) {
        set_err("sage_select: null idx");
        return SAGE_ERR_INVALID_ARG;
    }
    if (k > 0) {
        cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
        size_t bytes = 0;
        select_scratch_bytes(N, &bytes);
        void* scratch = nullptr;
        CU_TRY(scratch_alloc(&scratch, bytes, st));
        cudaError_t e = launch_select(scores, N, k, idx, scratch, st);
        cudaError_t e2 = cudaFreeAsync(scratch, st);
        CU_TRY(e);
        CU_TRY(e2);
        count(nullptr, select_launches(N, k));
    }
    if (k_out) *k_out = k;
    return SAGE_OK;
}

sage_status_t sage_score_classes(sage_fd_t* h, const int32_t* labels, int32_t num_classes, float* scores, void* cuda_stream) {
    ST_TRY(check_handle(h));
    if (h->state != FROZEN || !h->scored) {
        set_err("sage_score_classes: needs a finished scoring pass (sage_score or sage_score_end) on this handle");
        return SAGE_ERR_BAD_STATE;
    }
    if (num_classes < 1 || num_classes > 65535 || (h->N_total > 0 && (!labels || !scores))) {
        set_err("sage_score_classes: bad argument (num_classes=%d labels=%p scores=%p)", (int)num_classes, (const void*)labels, (void*)scores);
        return SAGE_ERR_INVALID_ARG;
    }
    DeviceGuard g(h->device);
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    if (num_classes > h->class_cap) {
        CU_TRY(cudaStreamSynchronize(st));
        if (h->class_U) CU_TRY(dev_free(h, h->class_U));
        if (h->class_counts) CU_TRY(dev_free(h, h->class_counts));
        h->class_U = nullptr;
        h->class_counts = nullptr;
        h->class_cap = 0;
        CU_TRY(dev_malloc(h, (void**)&h->class_U, (size_t)num_classes * h->ell * sizeof(float)));
        CU_TRY(dev_malloc(h, (void**)&h->class_counts, (size_t)num_classes * sizeof(int)));
        h->class_cap = num_classes;
    }
    h->class_num = num_classes;
    void* scratch = nullptr;
    const size_t bytes = class_scratch_bytes(h->N_total, h->ell, num_classes);
    if (bytes > 0) CU_TRY(scratch_alloc(&scratch, bytes, st));
    const cudaError_t e = launch_class_scores(h->zhat, labels, h->N_total, h->ell, num_classes, h->class_U, h->class_counts, scores, scratch, st);
    const cudaError_t e2 = scratch ? cudaFreeAsync(scratch, st) : cudaSuccess;
    CU_TRY(e);
    CU_TRY(e2);
    count(h, class_score_launches(h->N_total, h->ell, num_classes));
    return SAGE_OK;
}

sage_status_t sage_score_class_centroids(const sage_fd_t* h, const float** U, const int32_t** counts, int32_t* num_classes) {
    ST_TRY(check_handle(h));
    if (!h->class_U || h->class_num == 0) {
        set_err("sage_score_class_centroids: sage_score_classes has not run on this handle");
        return SAGE_ERR_BAD_STATE;
    }
    if (U) *U = h->class_U;
    if (counts) *counts = h->class_counts;
    if (num_classes) *num_classes = h->class_num;
    return SAGE_OK;
}

sage_status_t sage_select_classes(const float* scores, const int32_t* labels, int64_t N, int32_t num_classes, double keep_rate,
                                  int64_t* idx, int64_t* k_per_class, int64_t* k_out, void* cuda_stream) {
    if (N < 0 || N >= (1ll << 31) || !(keep_rate == keep_rate) || num_classes < 1 || num_classes > 65535 || (N > 0 && (!scores || !labels))) {
        set_err("sage_select_classes: bad argument (N=%lld num_classes=%d keep_rate=%g)", (long long)N, (int)num_classes, keep_rate);
        return SAGE_ERR_INVALID_ARG;
    }
    const int C = num_classes;
    std::vector<long long> kc(C, 0), offs(C, 0);
    long long k = 0;
    if (N > 0) {
        cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
        size_t sel_bytes = 0;
        select_scratch_bytes(N, &sel_bytes);
        const size_t a256 = 255;
        const size_t starts_off = (sel_bytes + a256) & ~a256;
        const size_t counts_off = (starts_off + (size_t)(C + 1) * 4 + a256) & ~a256;
        const size_t kc_off = (counts_off + (size_t)C * 4 + a256) & ~a256;
        const size_t offs_off = (kc_off + (size_t)(C + 1) * 8 + a256) & ~a256;
        const size_t total = offs_off + (size_t)C * 8;
        char* scratch = nullptr;
        CU_TRY(scratch_alloc((void**)&scratch, total, st));
        long long* d_kc = reinterpret_cast<long long*>(scratch + kc_off);
        long long* d_offs = reinterpret_cast<long long*>(scratch + offs_off);
        auto body = [&]() -> sage_status_t {
            if (idx && class_select_in_one(N, C)) {          // sort, quotas and picks in one launch; the quotas come back
                CU_TRY(launch_class_select(scores, labels, N, C, keep_rate, scratch, idx, d_kc, st));
                kc.resize((size_t)C + 1);
                CU_TRY(cudaMemcpyAsync(kc.data(), d_kc, (size_t)(C + 1) * 8, cudaMemcpyDeviceToHost, st));
                CU_TRY(cudaStreamSynchronize(st));
                k = kc[(size_t)C];
                count(nullptr, 1);
                return SAGE_OK;
            }
            unsigned* d_starts = reinterpret_cast<unsigned*>(scratch + starts_off);
            unsigned* d_counts = reinterpret_cast<unsigned*>(scratch + counts_off);
            CU_TRY(launch_class_starts(labels, N, C, d_starts, d_counts, st));
            std::vector<unsigned> counts(C);
            CU_TRY(cudaMemcpyAsync(counts.data(), d_counts, (size_t)C * sizeof(unsigned), cudaMemcpyDeviceToHost, st));
            CU_TRY(cudaStreamSynchronize(st));
            long long n_valid = 0;
            for (int c = 0; c < C; ++c) n_valid += counts[c];
            k = sage_select_count(n_valid, keep_rate);
            // k_c proportional to the class sizes, largest remainder, ties to the smaller class (exact integers)
            std::vector<long long> rem(C, 0);
            long long given = 0;
            if (n_valid > 0)
                for (int c = 0; c < C; ++c) {
                    const long long num = (long long)counts[c] * k;
                    kc[c] = num / n_valid;
                    rem[c] = num - kc[c] * n_valid;
                    given += kc[c];
                }
            std::vector<int> order(C);
            for (int c = 0; c < C; ++c) order[c] = c;
            std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return rem[a] > rem[b]; });
            for (long long t = 0; t < k - given; ++t) kc[order[(size_t)t]] += 1;
            long long run = 0;
            for (int c = 0; c < C; ++c) { offs[c] = run; run += kc[c]; }
            if (k > 0 && !idx) {
                set_err("sage_select_classes: null idx");
                return SAGE_ERR_INVALID_ARG;
            }
            if (k > 0) {
                CU_TRY(cudaMemcpyAsync(d_kc, kc.data(), (size_t)C * 8, cudaMemcpyHostToDevice, st));
                CU_TRY(cudaMemcpyAsync(d_offs, offs.data(), (size_t)C * 8, cudaMemcpyHostToDevice, st));
                CU_TRY(launch_class_pick(scores, labels, N, C, scratch, d_starts, d_kc, d_offs, idx, st));
                CU_TRY(cudaStreamSynchronize(st));        // kc / offs are host vectors of this call
                count(nullptr, class_pick_launches(N, C));
            }
            return SAGE_OK;
        };
        const sage_status_t rc = body();
        cudaFreeAsync(scratch, st);
        if (rc != SAGE_OK) return rc;
    }
    if (k_per_class)
        for (int c = 0; c < C; ++c) k_per_class[c] = kc[c];
    if (k_out) *k_out = k;
    return SAGE_OK;
}

// ---- checkpoint of the sketch state ---------------------------------------------------------------------------
namespace {
struct ExportHeader {
    char magic[8];
    int64_t D;
    int32_t ell, dtype, P, frozen;
    int64_t block, dealt;
    int32_t nsk, delta_rank;
};
struct ExportSketch {
    int32_t rows, pad;
    EigInfo info;
};
// A sketch in the middle of a block: its planes, D values a row, and its small matrices follow.
struct ExportBlock {
    int32_t s_rows, n_raw, n_gram, cycles, np, cycles_of_block;
};
const char kExportMagic[8] = {'S', 'A', 'G', 'E', 'F', 'D', '1', 0}, kExportMagicBlock[8] = {'S', 'A', 'G', 'E', 'F', 'D', '2', 0};

// The device arrays of an open block, one call of f(array, pitch, width, rows), in bytes, for each.
extern "C++" template <typename F>
sage_status_t each_block_array(const sage_fd* h, const sage_fd::Block& k, const ExportBlock& eb, F&& f) {
    const size_t row = (size_t)h->D * 2, pitch = (size_t)k.pitch * 2, ldP = (size_t)k.ldP * 4, ldu = (size_t)k.ldu * 4, ldk = (size_t)h->ldk * 4;
    ST_TRY(f((void*)k.S[k.cur], pitch, row, (size_t)3 * eb.s_rows));
    ST_TRY(f((void*)k.R, pitch, row, (size_t)eb.np * eb.n_raw));
    ST_TRY(f((void*)k.P, ldP, ldP, (size_t)eb.n_gram));
    if (eb.cycles > 0) {
        ST_TRY(f((void*)k.C, ldP, ldP, (size_t)h->ell - 1));
        ST_TRY(f((void*)k.U, ldu, ldu, (size_t)eb.cycles * h->m));
        ST_TRY(f((void*)(k.K + (size_t)(eb.cycles & 1) * h->m * h->ldk), ldk, ldk, (size_t)h->m));
    }
    return SAGE_OK;
}
ExportBlock export_block(const sage_fd* h) {
    const auto& k = h->blk;
    return {k.s_rows, k.n_raw, k.n_gram, k.cycles, k.np, k.L};
}
size_t export_block_bytes(const sage_fd* h, const ExportBlock& eb) {
    size_t total = 0;
    each_block_array(h, block_shape(h), eb, [&](void*, size_t, size_t width, size_t rows) {
        total += width * rows;
        return SAGE_OK;
    });
    return total;
}

int export_rows(const sage_fd* s, bool frozen) { return frozen ? s->ell : s->fill; }
}  // namespace

sage_status_t sage_fd_export_size(const sage_fd_t* h, size_t* bytes) {
    ST_TRY(check_handle(h));
    if (!bytes) {
        set_err("sage_fd_export_size: null bytes");
        return SAGE_ERR_INVALID_ARG;
    }
    if (h->state == SCORING) {
        set_err("sage_fd_export_size: a scoring pass is open");
        return SAGE_ERR_BAD_STATE;
    }
    const bool frozen = h->state == FROZEN;
    size_t total = sizeof(ExportHeader);
    if (!frozen && h->sketching_in_blocks) {
        *bytes = total + sizeof(ExportSketch) + sizeof(ExportBlock) + export_block_bytes(h, export_block(h));
        return SAGE_OK;
    }
    const int nsk = frozen ? 1 : (int)h->kids.size() + 1;
    for (int p = 0; p < nsk; ++p) {
        const sage_fd* s = p == 0 ? h : h->kids[(size_t)p - 1];
        total += sizeof(ExportSketch) + (size_t)export_rows(s, frozen) * h->D * sizeof(float);
    }
    if (frozen) total += (size_t)h->ell * sizeof(float);
    *bytes = total;
    return SAGE_OK;
}

sage_status_t sage_fd_export(sage_fd_t* h, void* dst_host, size_t capacity, size_t* written) {
    size_t need = 0;
    ST_TRY(sage_fd_export_size(h, &need));
    if (!dst_host || capacity < need) {
        set_err("sage_fd_export: destination of %zu bytes is too small (%zu needed)", capacity, need);
        return SAGE_ERR_INVALID_ARG;
    }
    DeviceGuard g(h->device);
    CU_TRY(cudaDeviceSynchronize());           // everything enqueued so far, on the caller's streams and the handle's own
    const bool frozen = h->state == FROZEN;
    char* out = static_cast<char*>(dst_host);
    ExportHeader hd = {};
    std::memcpy(hd.magic, kExportMagic, 8);
    hd.D = h->D;
    hd.ell = h->ell;
    hd.dtype = (int32_t)h->dtype;
    hd.P = h->P;
    hd.frozen = frozen ? 1 : 0;
    hd.block = h->block;
    hd.dealt = h->dealt;
    hd.nsk = frozen ? 1 : (int)h->kids.size() + 1;
    hd.delta_rank = h->delta_rank;
    const bool in_block = !frozen && h->sketching_in_blocks;
    if (in_block) std::memcpy(hd.magic, kExportMagicBlock, 8);
    std::memcpy(out, &hd, sizeof hd);
    out += sizeof hd;
    if (in_block) {
        ExportSketch es = {};
        es.rows = h->fill;
        CU_TRY(cudaMemcpy(&es.info, h->info, sizeof(EigInfo), cudaMemcpyDeviceToHost));
        std::memcpy(out, &es, sizeof es);
        out += sizeof es;
        ST_TRY(block_step(h, h->blk.n_gram, nullptr));         // a step that waits for rows: the same bits now as with them
        CU_TRY(cudaDeviceSynchronize());
        const ExportBlock eb = export_block(h);
        std::memcpy(out, &eb, sizeof eb);
        out += sizeof eb;
        ST_TRY(each_block_array(h, h->blk, eb, [&](void* p, size_t pitch, size_t width, size_t rows) -> sage_status_t {
            if (rows > 0) CU_TRY(cudaMemcpy2D(out, width, p, pitch, width, rows, cudaMemcpyDeviceToHost));
            out += width * rows;
            return SAGE_OK;
        }));
        if (written) *written = (size_t)(out - static_cast<char*>(dst_host));
        return SAGE_OK;
    }
    for (int p = 0; p < hd.nsk; ++p) {
        sage_fd* s = sketch_at(h, p);
        ExportSketch es = {};
        es.rows = export_rows(s, frozen);
        CU_TRY(cudaMemcpy(&es.info, s->info, sizeof(EigInfo), cudaMemcpyDeviceToHost));
        if (frozen)                             // the counters of all sketches, as sage_fd_stats reports them
            for (sage_fd* k : h->kids) {
                EigInfo ki;
                CU_TRY(cudaMemcpy(&ki, k->info, sizeof ki, cudaMemcpyDeviceToHost));
                es.info.shrinks += ki.shrinks;
                es.info.sum_delta += ki.sum_delta;
                es.info.flags |= ki.flags;
                if (ki.max_sweeps > es.info.max_sweeps) es.info.max_sweeps = ki.max_sweeps;
            }
        std::memcpy(out, &es, sizeof es);
        out += sizeof es;
        if (es.rows > 0)
            CU_TRY(cudaMemcpy2D(out, (size_t)h->D * sizeof(float), s->B[s->cur], (size_t)s->pitch * sizeof(float),
                                (size_t)h->D * sizeof(float), (size_t)es.rows, cudaMemcpyDeviceToHost));
        out += (size_t)es.rows * h->D * sizeof(float);
    }
    if (frozen) {
        CU_TRY(cudaMemcpy(out, h->sigma, (size_t)h->ell * sizeof(float), cudaMemcpyDeviceToHost));
        out += (size_t)h->ell * sizeof(float);
    }
    if (written) *written = (size_t)(out - static_cast<char*>(dst_host));
    return SAGE_OK;
}

// A checkpoint from the middle of a block: q, left: what follows its header.
static sage_status_t import_block(sage_fd* h, const ExportHeader& hd, const char* q, size_t left) {
    ExportSketch es;
    ExportBlock eb;
    const sage_fd::Block shape = block_shape(h);
    auto refuse = [] {
        set_err("sage_fd_import: truncated or inconsistent checkpoint");
        return SAGE_ERR_INVALID_ARG;
    };
    if (left < sizeof es + sizeof eb) return refuse();
    std::memcpy(&es, q, sizeof es);
    std::memcpy(&eb, q + sizeof es, sizeof eb);
    q += sizeof es + sizeof eb;
    left -= sizeof es + sizeof eb;
    if (hd.frozen || hd.P != 1 || hd.nsk != 1 || hd.delta_rank != h->ell || h->sketch_only || eb.cycles_of_block != shape.L || eb.s_rows < 0 || eb.s_rows >= h->ell ||
        eb.n_raw < 0 || eb.n_raw >= shape.M - eb.s_rows || eb.n_gram < 0 || eb.n_gram > eb.s_rows + eb.n_raw || eb.cycles < 0 || eb.cycles >= (eb.s_rows < h->ell - 1 ? 1 : shape.L) ||
        eb.np < shape.np || eb.np > (h->dtype == SAGE_F32 ? 3 : 2) || es.rows != eb.s_rows + eb.n_raw - eb.cycles * (h->ell + 1) || es.rows < 0 || es.rows >= h->m ||
        (eb.cycles > 0 && eb.n_gram < h->m + (eb.cycles - 1) * (h->ell + 1)) || left < export_block_bytes(h, eb))
        return refuse();
    DeviceGuard g(h->device);
    ST_TRY(sage_fd_reset(h));
    ST_TRY(sage_fd_set_option(h, 6, 1.0));
    h->block = hd.block;
    h->delta_rank = hd.delta_rank;
    ST_TRY(settle_form(h, IN_BLOCKS));
    if (!h->sketching_in_blocks) {
        set_err("sage_fd_import: no memory for the rows of a block");
        return SAGE_ERR_ALLOC;
    }
    auto& k = h->blk;
    ST_TRY(block_widen(h, eb.np, nullptr));
    CU_TRY(cudaMemcpy(h->info, &es.info, sizeof(EigInfo), cudaMemcpyHostToDevice));
    k.cur = 0;
    ST_TRY(each_block_array(h, k, eb, [&](void* p, size_t pitch, size_t width, size_t rows) -> sage_status_t {
        if (rows > 0) CU_TRY(cudaMemcpy2D(p, pitch, q, width, width, rows, cudaMemcpyHostToDevice));
        q += width * rows;
        return SAGE_OK;
    }));
    k.s_rows = eb.s_rows;
    k.n_raw = eb.n_raw;
    k.n_gram = eb.n_gram;
    k.cycles = eb.cycles;
    h->fill = es.rows;
    h->dealt = hd.dealt;
    h->rows_seen = hd.dealt;
    CU_TRY(cudaDeviceSynchronize());
    return settle_form(h);
}

sage_status_t sage_fd_import(sage_fd_t* h, const void* src_host, size_t bytes, void* cuda_stream) {
    ST_TRY(check_handle(h));
    ExportHeader hd;
    if (!src_host || bytes < sizeof hd) {
        set_err("sage_fd_import: no data");
        return SAGE_ERR_INVALID_ARG;
    }
    std::memcpy(&hd, src_host, sizeof hd);
    const bool in_block = std::memcmp(hd.magic, kExportMagicBlock, 8) == 0;
    if ((!in_block && std::memcmp(hd.magic, kExportMagic, 8) != 0) || hd.D != h->D || hd.ell != h->ell || hd.dtype != (int32_t)h->dtype || hd.P < 1 ||
        hd.P > 64 || hd.nsk < 1 || hd.nsk > hd.P || hd.block < 1 || hd.dealt < 0 || hd.delta_rank < 2 || hd.delta_rank > h->m - 1) {
        set_err("sage_fd_import: not a checkpoint of a sketch with D=%lld ell=%d and this row type", (long long)h->D, h->ell);
        return SAGE_ERR_INVALID_ARG;
    }
    // sizes first: nothing of the handle changes unless the whole checkpoint is consistent
    if (in_block) return import_block(h, hd, static_cast<const char*>(src_host) + sizeof hd, bytes - sizeof hd);
    {
        const char* q = static_cast<const char*>(src_host) + sizeof hd;
        size_t left = bytes - sizeof hd;
        for (int p = 0; p < hd.nsk; ++p) {
            ExportSketch es;
            if (left < sizeof es) { set_err("sage_fd_import: truncated checkpoint"); return SAGE_ERR_INVALID_ARG; }
            std::memcpy(&es, q, sizeof es);
            const size_t rb = (size_t)(es.rows < 0 ? 0 : es.rows) * h->D * sizeof(float);
            if (es.rows < 0 || es.rows >= h->m + (hd.frozen ? 1 : 0) || left < sizeof es + rb) {
                set_err("sage_fd_import: truncated or inconsistent checkpoint");
                return SAGE_ERR_INVALID_ARG;
            }
            q += sizeof es + rb;
            left -= sizeof es + rb;
        }
        if (hd.frozen && left < (size_t)h->ell * sizeof(float)) { set_err("sage_fd_import: truncated checkpoint"); return SAGE_ERR_INVALID_ARG; }
    }
    DeviceGuard g(h->device);
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    ST_TRY(sage_fd_reset(h));
    ST_TRY(sage_fd_set_option(h, 6, (double)hd.P));
    h->block = hd.block;
    if (h->delta_rank != hd.delta_rank) drop_cycles(h);
    h->delta_rank = hd.delta_rank;
    for (sage_fd* k : h->kids) k->delta_rank = hd.delta_rank;
    if (hd.nsk > 1) ST_TRY(ensure_sketches(h));
    ST_TRY(settle_form(h, BY_CYCLES));                  // the rows go to the buffers first
    const char* q = static_cast<const char*>(src_host) + sizeof hd;
    for (int p = 0; p < hd.nsk; ++p) {
        sage_fd* s = sketch_at(h, p);
        s->delta_rank = hd.delta_rank;
        ExportSketch es;
        std::memcpy(&es, q, sizeof es);
        q += sizeof es;
        CU_TRY(cudaMemcpy(s->info, &es.info, sizeof(EigInfo), cudaMemcpyHostToDevice));
        if (es.rows > 0)
            CU_TRY(cudaMemcpy2D(s->B[0], (size_t)s->pitch * sizeof(float), q, (size_t)h->D * sizeof(float), (size_t)h->D * sizeof(float),
                                (size_t)es.rows, cudaMemcpyHostToDevice));
        if (s->pitch > h->D && es.rows > 0)     // columns between D and the pitch are zero in every buffer row
            CU_TRY(cudaMemset2D(s->B[0] + h->D, (size_t)s->pitch * sizeof(float), 0, (size_t)(s->pitch - h->D) * sizeof(float), (size_t)es.rows));
        q += (size_t)es.rows * h->D * sizeof(float);
        s->cur = 0;
        s->fill = hd.frozen ? h->ell : es.rows;
    }
    h->dealt = hd.dealt;
    h->rows_seen = hd.dealt;
    if (!hd.frozen) ST_TRY(settle_form(h));
    if (hd.frozen) {
        CU_TRY(cudaMemcpy(h->sigma, q, (size_t)h->ell * sizeof(float), cudaMemcpyHostToDevice));
        CU_TRY(cudaDeviceSynchronize());
        ST_TRY(enqueue_freeze_aux(h, st));
        h->state = FROZEN;
    } else {
        CU_TRY(cudaDeviceSynchronize());
    }
    return SAGE_OK;
}

sage_status_t sage_fd_stats(sage_fd_t* h, sage_stats_t* out) {
    ST_TRY(check_handle(h));
    if (!out) {
        set_err("sage_fd_stats: null out");
        return SAGE_ERR_INVALID_ARG;
    }
    DeviceGuard g(h->device);
    CU_TRY(cudaDeviceSynchronize());
    EigInfo info;
    CU_TRY(cudaMemcpy(&info, h->info, sizeof info, cudaMemcpyDeviceToHost));
    int tc_err = 0;
    CU_TRY(cudaMemcpy(&tc_err, h->tc_err, sizeof tc_err, cudaMemcpyDeviceToHost));
    int64_t launches = h->launches, tc_launches = h->tc_launches, in_place = h->rows_in_place;
    for (sage_fd* k : h->kids) {             // merged form: counters of all sketches together
        EigInfo ki;
        int kt = 0;
        CU_TRY(cudaMemcpy(&ki, k->info, sizeof ki, cudaMemcpyDeviceToHost));
        CU_TRY(cudaMemcpy(&kt, k->tc_err, sizeof kt, cudaMemcpyDeviceToHost));
        info.shrinks += ki.shrinks;
        info.sum_delta += ki.sum_delta;
        info.flags |= ki.flags;
        if (ki.max_sweeps > info.max_sweeps) info.max_sweeps = ki.max_sweeps;
        tc_err |= kt;
        launches += k->launches;
        tc_launches += k->tc_launches;
        in_place += k->rows_in_place;
    }
    out->rows_seen = h->dealt;
    out->shrinks = info.shrinks;
    out->sum_delta = info.sum_delta;
    out->last_sweeps = info.sweeps;
    out->max_sweeps = info.max_sweeps;
    out->last_rank = info.rank;
    out->device_flags = info.flags | (tc_err ? 4u : 0u);
    out->kernel_launches = launches;
    out->tensor_core_launches = tc_launches;
    out->rows_in_place = in_place;
    return SAGE_OK;
}

sage_status_t sage_fd_profile(sage_fd_t* h, double* ms, int64_t* launches, int32_t capacity) {
    ST_TRY(check_handle(h));
    if (!ms || !launches || capacity < K_NCLASS) {
        set_err("sage_fd_profile: need arrays of at least %d entries", (int)K_NCLASS);
        return SAGE_ERR_INVALID_ARG;
    }
    DeviceGuard g(h->device);
    CU_TRY(cudaDeviceSynchronize());
    for (int c = 0; c < K_NCLASS; ++c) {
        ms[c] = 0.0;
        launches[c] = 0;
    }
    for (int q = 0; q <= (int)h->kids.size(); ++q) {     // merged form: all sketches together (their kernels overlap in time)
        Prof& pr = sketch_at(h, q)->prof;
        for (auto& p : pr.pending) {
            float t = 0.f;
            if (cudaEventElapsedTime(&t, p.a, p.b) == cudaSuccess) {
                pr.ms[p.cls] += t;
                pr.n[p.cls] += 1;
            }
            pr.pool.push_back(p.a);
            pr.pool.push_back(p.b);
        }
        pr.pending.clear();
        for (int c = 0; c < K_NCLASS; ++c) {
            ms[c] += pr.ms[c];
            launches[c] += pr.n[c];
            pr.ms[c] = 0.0;
            pr.n[c] = 0;
        }
    }
    return SAGE_OK;
}

sage_status_t sage_select_from_host(const void* rows_host, int64_t N, int64_t D, int64_t ld, int32_t ell,
                                    sage_dtype_t row_dtype, double keep_rate, int64_t chunk_rows, int device,
                                    float* scores_host, int64_t* idx_host, int64_t* k_out) {
    if (!rows_host || N < 1 || D < 1 || ld < D || !(keep_rate == keep_rate)) {
        set_err("sage_select_from_host: bad argument");
        return SAGE_ERR_INVALID_ARG;
    }
    const int64_t k = sage_select_count(N, keep_rate);
    if (k > 0 && !idx_host) {
        set_err("sage_select_from_host: null idx_host");
        return SAGE_ERR_INVALID_ARG;
    }
    DeviceGuard g(device);
    if (!g.ok) {
        set_err("sage_select_from_host: cannot select CUDA device %d: %s", device, cudaGetErrorString(cudaGetLastError()));
        return SAGE_ERR_CUDA;
    }
    const size_t es = elem_size(row_dtype), row_bytes = (size_t)ld * es;
    constexpr size_t kStage = (size_t)256 << 20;                         // bytes of a staging buffer by default
    // Rows that fit the two staging buffers stay on the device: they cross the bus once, in pieces so that the sketch starts
    // with the first one, and pass 2 takes them as they are. (The caller's chunk_rows sets the memory where it asks for less.)
    const bool resident = chunk_rows >= N || (chunk_rows <= 0 && (size_t)N * row_bytes <= 2 * kStage);
    if (chunk_rows <= 0) {
        chunk_rows = (int64_t)(kStage / row_bytes);
        if (resident) chunk_rows = (N + 7) / 8;
        if (chunk_rows < 2 * ell) chunk_rows = 2 * ell;
    }
    if (chunk_rows > N) chunk_rows = N;
    const int nstage = resident ? 1 : 2;
    const size_t stage_bytes = (size_t)(resident ? N : chunk_rows) * row_bytes;
    sage_fd_t* h = nullptr;
    void* stage[2] = {nullptr, nullptr};
    float* d_scores = nullptr;
    int64_t* d_idx = nullptr;
    cudaStream_t s_copy = nullptr, s_comp = nullptr;
    cudaEvent_t copied[2] = {nullptr, nullptr}, consumed[2] = {nullptr, nullptr}, ready = nullptr;
    sage_status_t rc = SAGE_OK;
    auto body = [&]() -> sage_status_t {
        CU_TRY(cudaStreamCreateWithFlags(&s_copy, cudaStreamNonBlocking));
        CU_TRY(cudaStreamCreateWithFlags(&s_comp, cudaStreamNonBlocking));
        CU_TRY(cudaEventCreateWithFlags(&ready, cudaEventDisableTiming));
        for (int i = 0; i < 2; ++i) {
            if (i < nstage) CU_TRY(scratch_alloc(&stage[i], stage_bytes, s_comp));
            CU_TRY(cudaEventCreateWithFlags(&copied[i], cudaEventDisableTiming));
            CU_TRY(cudaEventCreateWithFlags(&consumed[i], cudaEventDisableTiming));
        }
        CU_TRY(cudaEventRecord(ready, s_comp));                          // the staging memory is this call's from here on
        CU_TRY(cudaStreamWaitEvent(s_copy, ready, 0));
        ST_TRY(create_handle(&h, D, ell, row_dtype, device, false, true, s_comp));
        CU_TRY(scratch_alloc((void**)&d_scores, (size_t)N * sizeof(float), s_comp));
        if (k > 0) CU_TRY(scratch_alloc((void**)&d_idx, (size_t)k * sizeof(int64_t), s_comp));
        const char* src = static_cast<const char*>(rows_host);
        for (int pass = 0; pass < 2; ++pass) {
            if (pass == 1) {
                sage_status_t f = sage_fd_finalize(h, s_comp);
                if (f != SAGE_OK && f != SAGE_ERR_NOT_CONVERGED && f != SAGE_ERR_NONFINITE) return f;
                if (f != SAGE_OK) rc = f;
                ST_TRY(sage_score_begin(h, N, s_comp));
                if (resident) {
                    ST_TRY(sage_score_chunk(h, stage[0], N, ld, 0, s_comp));
                    break;
                }
            }
            int64_t c = 0;
            for (int64_t r0 = 0; r0 < N; r0 += chunk_rows, ++c) {
                const int b = (int)(c & 1);
                const int64_t n = (N - r0 < chunk_rows) ? N - r0 : chunk_rows;
                char* at = static_cast<char*>(resident ? stage[0] : stage[b]) + (resident ? (size_t)r0 * row_bytes : 0);
                if (!resident && (c >= 2 || pass == 1)) CU_TRY(cudaStreamWaitEvent(s_copy, consumed[b], 0));
                CU_TRY(cudaMemcpyAsync(at, src + (size_t)r0 * row_bytes, (size_t)n * row_bytes, cudaMemcpyHostToDevice, s_copy));
                CU_TRY(cudaEventRecord(copied[b], s_copy));
                CU_TRY(cudaStreamWaitEvent(s_comp, copied[b], 0));
                if (pass == 0)
                    ST_TRY(sage_fd_update(h, at, n, ld, s_comp));
                else
                    ST_TRY(sage_score_chunk(h, at, n, ld, r0, s_comp));
                if (!resident) CU_TRY(cudaEventRecord(consumed[b], s_comp));
            }
        }
        ST_TRY(sage_score_end(h, d_scores, s_comp));
        int64_t kk = 0;
        ST_TRY(sage_select(d_scores, N, keep_rate, d_idx, &kk, s_comp));
        if (scores_host) CU_TRY(cudaMemcpyAsync(scores_host, d_scores, (size_t)N * sizeof(float), cudaMemcpyDeviceToHost, s_comp));
        if (k > 0) CU_TRY(cudaMemcpyAsync(idx_host, d_idx, (size_t)k * sizeof(int64_t), cudaMemcpyDeviceToHost, s_comp));
        CU_TRY(cudaStreamSynchronize(s_comp));
        CU_TRY(cudaStreamSynchronize(s_copy));
        // what the device recorded during pass 2 (pass 1 was reported by the freeze)
        int tc_err = 0;
        EigInfo info;
        CU_TRY(cudaMemcpy(&tc_err, h->tc_err, sizeof tc_err, cudaMemcpyDeviceToHost));
        CU_TRY(cudaMemcpy(&info, h->info, sizeof info, cudaMemcpyDeviceToHost));
        if (tc_err || (info.flags & kFlagExchangeTimeout)) {
            set_err("sage_select_from_host: a kernel gave up a bounded wait during the scoring pass (results are not valid)");
            return SAGE_ERR_CUDA;
        }
        if ((info.flags & kFlagNonFinite) && rc == SAGE_OK) {
            set_err("sage_select_from_host: non-finite values were met in the rows (such rows score 0)");
            rc = SAGE_ERR_NONFINITE;
        }
        return SAGE_OK;
    };
    sage_status_t s = body();
    cudaDeviceSynchronize();
    for (int i = 0; i < 2; ++i) {
        if (stage[i]) cudaFreeAsync(stage[i], s_comp);
        if (copied[i]) cudaEventDestroy(copied[i]);
        if (consumed[i]) cudaEventDestroy(consumed[i]);
    }
    if (ready) cudaEventDestroy(ready);
    if (d_scores) cudaFreeAsync(d_scores, s_comp);
    if (d_idx) cudaFreeAsync(d_idx, s_comp);
    sage_fd_destroy(h);
    if (s_copy) cudaStreamDestroy(s_copy);
    if (s_comp) cudaStreamDestroy(s_comp);
    if (s != SAGE_OK) return s;
    if (k_out) *k_out = k;
    return rc;
}

}  // extern "C"
