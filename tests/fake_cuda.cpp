// A CUDA runtime that does nothing but keep books, and launchers that record what they are asked for: csrc/api.cu compiled against it
// runs on the CPU, where a test can let any call fail and look at what the host code did. No arithmetic, no device.
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "sage_internal.h"

namespace {
std::mutex mu;
std::map<std::string, int> calls, fail_at;
struct Append {
    const void *rows, *rows2;
    long long n, n2, row0;
};
std::vector<Append> appends;
int capturing = 0;
thread_local bool no_memory = false;
cudaError_t last = cudaSuccess;

cudaError_t book(const char* name) {
    std::lock_guard<std::mutex> lock(mu);
    const int n = ++calls[name];
    const auto f = fail_at.find(name);
    if (f != fail_at.end() && f->second == n) return last = cudaErrorUnknown;
    return cudaSuccess;
}
template <typename T>
T handle() {
    static long next = 16;
    std::lock_guard<std::mutex> lock(mu);
    return reinterpret_cast<T>(next += 16);
}
void kernel(int) {}
}  // namespace

void* operator new(size_t n) {
    if (no_memory) throw std::bad_alloc();
    if (void* p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }

extern "C" {
int fake_allow_smem_without_memory() {                // what the launchers call before a kernel of much shared memory
    static char kernel;
    no_memory = true;
    const cudaError_t e = sage::allow_smem(&kernel, 1024);
    no_memory = false;
    return (int)e;
}
int fake_allow_smem(int regs) {                       // a kernel that was compiled with 64 registers a thread
    static char kernels[256];
    return (int)sage::allow_smem(&kernels[regs], 1024, regs);
}
int fake_calls(const char* name) { return calls[name]; }
void fake_fail(const char* name, int nth_from_now) { fail_at[name] = calls[name] + nth_from_now; }
void fake_capturing(int on) { capturing = on; }
int fake_appends(long long* out, int capacity) {      // rows, n, rows2, n2, first row, for each append since the last call
    int k = 0;
    for (const Append& a : appends)
        if (k < capacity) {
            const long long v[5] = {(long long)a.rows, a.n, (long long)a.rows2, a.n2, a.row0};
            std::memcpy(out + 5 * k++, v, sizeof v);
        }
    appends.clear();
    return k;
}

#define BOOK if (cudaError_t e = book(__func__)) return e
cudaError_t cudaMalloc(void** p, size_t n) { BOOK; *p = std::calloc(1, n ? n : 1); return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { BOOK; *p = std::calloc(1, n ? n : 1); return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { BOOK; *p = std::calloc(1, n ? n : 1); return cudaSuccess; }
cudaError_t cudaFree(void* p) { BOOK; std::free(p); return cudaSuccess; }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { BOOK; std::free(p); return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { BOOK; *p = handle<cudaMemPool_t>(); return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { BOOK; return cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n) { BOOK; std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemset2D(void*, size_t, int, size_t, size_t) { BOOK; return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { BOOK; std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { BOOK; std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { BOOK; std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpy2D(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind) { BOOK; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaDeviceSynchronize() { BOOK; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* fa, const void*) {
    *fa = cudaFuncAttributes();
    fa->numRegs = 64;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { BOOK; *e = handle<cudaEvent_t>(); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { BOOK; *e = handle<cudaEvent_t>(); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { BOOK; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { BOOK; return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { BOOK; return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) { BOOK; *t = 0.f; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { BOOK; *s = handle<cudaStream_t>(); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { BOOK; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { BOOK; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { BOOK; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
    *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { BOOK; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { BOOK; *g = handle<cudaGraph_t>(); return cudaSuccess; }
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { BOOK; *g = handle<cudaGraph_t>(); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { BOOK; return cudaSuccess; }
cudaError_t cudaGraphAddNode_v2(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t, cudaGraphNodeParams*) {
    BOOK;
    *n = handle<cudaGraphNode_t>();
    return cudaSuccess;
}
cudaError_t cudaGraphKernelNodeSetAttribute(cudaGraphNode_t, cudaLaunchAttributeID, const cudaLaunchAttributeValue*) { BOOK; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) { BOOK; *x = handle<cudaGraphExec_t>(); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { BOOK; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { BOOK; return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { BOOK; return cudaSuccess; }
}  // extern "C"

namespace sage {
#define GO return launch_chained(kernel, dim3(1), dim3(1), 0, st, 0)
cudaError_t launch_append(const void* rows, sage_dtype_t, int64_t n, int64_t, int64_t, float*, int64_t, int row0, cudaStream_t st, const void* rows2, int64_t n2) {
    appends.push_back({rows, rows2, n, n2, row0});
    GO;
}
cudaError_t launch_append_outer(const void* q, int64_t, const void*, int64_t, sage_dtype_t, int64_t n, int, int, float*, int64_t, int row0, cudaStream_t st, const void* q2,
                                const void*, int64_t n2) {
    appends.push_back({q, q2, n, n2, row0});
    GO;
}
cudaError_t launch_outer_combine(const void*, int64_t, sage_dtype_t, int, const float*, int, int64_t, const float*, int64_t, float*, int64_t, int, float*, cudaStream_t st) { GO; }
cudaError_t launch_gemm_nt(const void*, sage_dtype_t, int64_t, const float*, int64_t, int, int, int64_t, int, float*, int64_t, int64_t, cudaStream_t st, int64_t) { GO; }
cudaError_t launch_tc_gemm_nt(const void*, sage_dtype_t, int64_t, const void*, int64_t, int, int, int, int, int64_t, int, float*, int64_t, int64_t, int*, cudaStream_t st, int64_t) { GO; }
cudaError_t launch_tc_gemm_nt_x3(const float*, int64_t, const float*, int64_t, int, int, int64_t, int, float*, int64_t, int64_t, int, int*, cudaStream_t st, int64_t) { GO; }
cudaError_t launch_tc_gram_direct(const float*, int64_t, int, const void*, int64_t, int, int64_t, int, float*, int64_t, int64_t, int*, cudaStream_t st) { GO; }
cudaError_t launch_gram_sym_reduce(const float*, int, int64_t, int, int64_t, float*, int64_t, cudaStream_t st, int) { GO; }
cudaError_t launch_tc_project(const float*, int64_t, const float*, int64_t, int64_t, int, int64_t, int64_t, float*, int64_t, int*, cudaStream_t st) { GO; }
cudaError_t launch_tc_gram_pair(const float*, int64_t, int, int64_t, int, int, float*, int64_t, int64_t, int*, cudaStream_t st) { GO; }
cudaError_t launch_tc_rebuild(const float*, int, int, const float*, float*, int64_t, int64_t, int, int, int*, cudaStream_t st) { GO; }
cudaError_t launch_tc_rebuild_direct(const float*, int, int, const float*, float*, int64_t, int64_t, int, int, const void*, int64_t, int, int*, cudaStream_t st) { GO; }
cudaError_t launch_to_bf16(const float*, int64_t, int, int64_t, __nv_bfloat16*, __nv_bfloat16*, int64_t, cudaStream_t st) { GO; }
cudaError_t launch_split_tf32(const float*, int64_t, int, int64_t, float*, int64_t, cudaStream_t st) { GO; }
cudaError_t launch_split_reduce(const float*, int, int64_t, int, int, int64_t, float*, int64_t, cudaStream_t st) { GO; }
cudaError_t launch_rebuild(const float*, int, const float*, float*, int64_t, int64_t, int, int, int, cudaStream_t st) { GO; }
cudaError_t launch_eig_shrink(const float*, int, int, int, int, int, float*, int, float*, int, float*, int, EigInfo*, float*, int, int, int, cudaStream_t st) { GO; }
cudaError_t launch_normalise(const float*, int, int64_t, int64_t, int64_t, int, float*, float*, float*, double*, unsigned*, cudaStream_t st) { GO; }
cudaError_t launch_consensus_score(const double*, const float*, int64_t, int, float*, float*, cudaStream_t st) { GO; }
cudaError_t launch_class_scores(const float*, const int*, int64_t, int, int, float*, int*, float*, void*, cudaStream_t st) { GO; }
cudaError_t launch_class_starts(const int*, int64_t, int, unsigned*, unsigned*, cudaStream_t st) { GO; }
cudaError_t launch_class_select(const float*, const int*, int64_t, int, double, void*, int64_t*, long long*, cudaStream_t st) { GO; }
cudaError_t launch_class_pick(const float*, const int*, int64_t, int, void*, const unsigned*, const long long*, const long long*, int64_t*, cudaStream_t st) { GO; }
cudaError_t launch_select(const float*, int64_t, int64_t, int64_t*, void*, cudaStream_t st) { GO; }
cudaError_t select_scratch_bytes(int64_t N, size_t* bytes) { *bytes = (size_t)N * 32 + 4096; return cudaSuccess; }
size_t class_scratch_bytes(int64_t, int, int) { return 4096; }
int class_score_launches(int64_t, int, int) { return 1; }
int class_pick_launches(int64_t, int) { return 1; }
size_t eig_work_floats(int n) { return (size_t)n * n; }
int eig_launches(int, int) { return 1; }
int project_planes(int64_t, int64_t, int64_t) { return 1; }
int select_launches(int64_t, int64_t) { return 1; }
bool class_select_in_one(int64_t, int) { return false; }
}  // namespace sage
