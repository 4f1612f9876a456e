// The library's host side (gp_api.cu) without a GPU: the CUDA runtime calls and
// the kernel launchers that it uses are stand-ins that write down what they were
// given.  Device pointers are numbers that nothing reads; memory is a budget.
// Built and driven by test_recorded_launches.py.
#include <cuda_runtime.h>

#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <map>
#include <string>

// what nvcc declares by itself
static inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)((uint64_t)a * b >> 32); }
static inline cudaError_t cudaGetSymbolAddress(void **p, const unsigned int &s) {
    *p = const_cast<unsigned int *>(&s);
    return cudaSuccess;
}

#include "gp_api.cu"

static std::string g_log;
static size_t g_limit = (size_t)1 << 40, g_held = 0;
static uintptr_t g_next = (uintptr_t)1 << 44;
static std::map<void *, size_t> g_sizes;

static void note(const char *fmt, ...) {
    char line[256];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(line, sizeof(line), fmt, ap);
    va_end(ap);
    g_log += line;
    g_log += '\n';
}

extern "C" {
const char *recorded() { return g_log.c_str(); }
void record_anew() { g_log.clear(); }
void memory_limit(size_t bytes) { g_limit = bytes; }

cudaError_t cudaMalloc(void **p, size_t n) {
    const bool ok = g_held + n <= g_limit;
    note("malloc bytes=%zu ok=%d", n, ok);
    if (!ok) return cudaErrorMemoryAllocation;
    *p = (void *)g_next;
    g_next += (n + 511) / 512 * 512;
    g_sizes[*p] = n;
    g_held += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    note("free bytes=%zu", g_sizes[p]);
    g_held -= g_sizes[p];
    g_sizes.erase(p);
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpy(void *, const void *, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *t, cudaEvent_t, cudaEvent_t) { return *t = 1.0f, cudaSuccess; }
}

namespace gpk {
static cudaError_t eval_noted(const char *what, int rows_per_thread, int fmode, const EvalArgs &a) {
    note("%s rows_per_thread=%d fmode=%d cls=%d qcls=%d ld=%lld rows=%lld x_unit=%d vec=%d", what,
         rows_per_thread, fmode, a.cls, a.qcls, (long long)a.ld, (long long)a.n_rows, a.x_unit, a.vec_ok);
    return cudaSuccess;
}
#define INSTANCE(R, F)                                                                                \
    cudaError_t launch_eval_r##R##_f##F(const EvalArgs &a, int, int, cudaStream_t) {                  \
        return eval_noted(a.pred ? "predict" : "eval", R, F, a);                                      \
    }
#define INFO(R, F) int info_eval_r##R##_f##F(int, int, int *, bool) { return 4; }
#define INFO8(F) int info_eval_r8_f##F(int, int, int *, bool, bool) { return 4; }
INSTANCE(4, 2) INSTANCE(4, 0) INSTANCE(8, 2) INSTANCE(8, 0) INSTANCE(16, 2) INSTANCE(16, 0)
INFO(4, 2) INFO(4, 0) INFO(16, 2) INFO(16, 0) INFO8(2) INFO8(0)
cudaError_t launch_predict(const EvalArgs &a, int, int, cudaStream_t) { return eval_noted("predict", 4, 0, a); }
cudaError_t launch_predict_f2(const EvalArgs &a, int, int, cudaStream_t) { return eval_noted("predict", 4, 2, a); }
int info_predict(int, int, int *) { return 4; }
int info_predict_f2(int, int, int *) { return 4; }
cudaError_t launch_grad(const GradArgs &a, int, cudaStream_t, int *) {
    note("grad bucket=%d n_feat=%d ld=%lld", a.bucket, a.n_feat, (long long)a.ld);
    return cudaSuccess;
}

// the workspace of an evaluation: only its size matters here
Layout make_layout(int n_progs, int n_chunks, bool grad, bool moments) {
    Layout L{};
    L.mom = moments;
    L.total = (size_t)n_progs * (grad ? kGradCodeStride : kCodeStride) * 8 + (size_t)n_progs * n_chunks * 64;
    return L;
}
Workspace carve(void *base, const Layout &L, bool) {
    Workspace w{};
    w.counters = static_cast<unsigned long long *>(base);
    w.bytes = L.total;
    return w;
}
void static_scratch_forget() {}
cudaError_t launch_compile(const CompileArgs &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_order(const ProgMeta *, int, int32_t *, int32_t *, cudaStream_t, unsigned long long *, int, int,
                         double *, int64_t) { return cudaSuccess; }
cudaError_t launch_sumw(const float *, int64_t, double *, double *, unsigned long long *, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t launch_ystats(const float *, const float *, int64_t, const double *, double *, double *,
                          unsigned long long *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_finalize(const FinalizeArgs &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_grad_finalize(const GradFinalizeArgs &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_plain(const PlainArgs &, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_adam(const AdamArgs &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_consts(gp_node *, const int32_t *, int, float *, bool, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_tournament(const TournArgs &, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_mutate(const MutArgs &, cudaStream_t) { return cudaSuccess; }
cudaError_t probe_pipes(double *, cudaStream_t) { return cudaSuccess; }

// the rank fitness: about what a batch takes (28 bytes a row and some)
size_t rank_scratch_bytes(int n_seg, int64_t n, bool weighted) {
    return (size_t)n_seg * ((size_t)n * (weighted ? 17 : 24) + 2560);
}
size_t target_part_bytes(int64_t n) { return (size_t)(n / 2048 + 2) * 24; }
cudaError_t target_ranks(const float *, const float *, int64_t, void *, uint32_t *, double *, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t spearman_batch(const float *, int n_seg, int64_t, const uint32_t *, const double *, const float *,
                           void *, float *, double *, cudaStream_t) {
    note("rank segments=%d", n_seg);
    return cudaSuccess;
}
}  // namespace gpk
