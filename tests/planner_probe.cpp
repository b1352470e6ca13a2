// The library's host code (planning, argument checks, batches) on a machine without a GPU: the CUDA
// calls it makes are answered with GB300's limits, and a launch keeps its plan for the test to read.
#include <cuda_runtime.h>
#include <stdlib.h>
#include <string.h>

#include "fim_host.cu"
#include "fim_noalloc.cu"
#include "fim_tune.cu"
#include "fim_batch.cu"

namespace {
Plan g_plan;  // of the last launch
int g_launches = 0;
std::vector<BatchClass> g_classes;  // of the last batch
std::vector<int> g_class_ctas;

constexpr int kSms = 152, kSmemPerSm = 228 * 1024, kSmemOptin = 227 * 1024;

// Resident CTAs per SM at 64 registers per thread; `fixed` bytes of static shared memory.
int resident(int threads, int smem, int fixed) {
    const int by_smem = kSmemPerSm / ((smem + fixed + 1024 + 127) / 128 * 128);
    return std::min(std::min(65536 / (threads * 64), by_smem), std::min(2048 / threads, 32));
}
}  // namespace

namespace fim {
fim_status launch_tile_kernel(Plan& p, cudaStream_t) {
    g_plan = p;
    ++g_launches;
    return resident(p.threads, p.smem_bytes, 128) >= 1 ? FIM_OK : FIM_ERR_UNSUPPORTED;
}
fim_status launch_tile_kernel_fixed(Plan& p, unsigned char*, size_t capacity, cudaStream_t st, bool launch) {
    const long long tiles = (long long)p.tiles_x * p.tiles_y;
    const long long grid = std::min<long long>(tiles, (long long)resident(p.threads, p.smem_bytes, 128) * kSms);
    if (grid < 1 || 256 + (size_t)grid * (size_t)p.scratch_per_cta > capacity) return FIM_ERR_UNSUPPORTED;
    return launch ? launch_tile_kernel(p, st) : FIM_OK;
}
fim_status launch_percentile_ranks(const float*, long long, int, int, int, int*, cudaStream_t) { return FIM_OK; }
fim_status read_and_clear_device_status(cudaStream_t) { return FIM_OK; }
fim_status batch_class_k8(const BatchClass& c, const BatchClassArgs* a, int* occ, cudaStream_t) {
    if (a == nullptr) {
        *occ = resident(c.threads, c.smem, 1024);
        g_classes.push_back(c);
        g_class_ctas.push_back(*occ);
    }
    return FIM_OK;
}
fim_status batch_class_k4(const BatchClass& c, const BatchClassArgs* a, int* occ, cudaStream_t st) {
    return batch_class_k8(c, a, occ, st);
}
}  // namespace fim

extern "C" {
// The plan of a learned launch or of training rows, kept like a launch's.
int probe_bracket(const fim_kernel* k, int dtype, int w, int h) {
    return bracket_plan(k, dtype, w, h, device_smem_limit(), &g_plan);
}

// Resident CTAs per SM of the class of the given jobs and threads in the last batch (0: no such class).
int probe_class(int dtype, int threads, int jobs) {
    int ctas = 0;
    for (size_t i = 0; i < g_classes.size(); ++i)
        if (g_classes[i].dtype == dtype && g_classes[i].threads == threads && g_classes[i].njobs == jobs)
            ctas = g_class_ctas[i];
    return ctas;
}
void probe_forget_classes() {
    g_classes.clear();
    g_class_ctas.clear();
}

// A field of the last launch's plan.
long long probe(const char* f) {
    const Plan& p = g_plan;
    if (!strcmp(f, "launches")) return g_launches;
    if (!strcmp(f, "Tx")) return p.Tx;
    if (!strcmp(f, "Ty")) return p.Ty;
    if (!strcmp(f, "threads")) return p.threads;
    if (!strcmp(f, "N")) return p.N;
    if (!strcmp(f, "spilled")) return p.loc_om < 0;
    if (!strcmp(f, "codes")) return p.codes > 0;
    if (!strcmp(f, "rank_base")) return p.rank_base;
    if (!strcmp(f, "rel_max")) return p.rel_max;
    if (!strcmp(f, "feasible")) return p.N - p.n + p.rank - p.rank_base;  // highest, as stored
    if (!strcmp(f, "wide")) return p.wide;
    if (!strcmp(f, "sort")) return p.sort;
    if (!strcmp(f, "inside")) {  // tiles whose box lies inside the image
        int n = 0;
        for (int t = 0; t < p.tiles_x * p.tiles_y; ++t) {
            const int x = t % p.tiles_x * p.Tx + p.xmin, y = t / p.tiles_x * p.Ty + p.ymin;
            n += x >= 0 && y >= 0 && x + p.S <= p.w && y + p.SH <= p.h;
        }
        return n;
    }
    if (!strcmp(f, "resident")) return resident(p.threads, p.smem_bytes, 128);
    abort();
}

cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? kSms
         : a == cudaDevAttrMaxSharedMemoryPerMultiprocessor ? kSmemPerSm
         : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? kSmemOptin : 0;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) { memset(p, 0, sizeof *p); return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = malloc(n + 1); return cudaSuccess; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) { *t = 1.f; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = const_cast<void*>(s); return cudaSuccess; }
cudaError_t cudaGetDriverEntryPoint(const char*, void**, unsigned long long, cudaDriverEntryPointQueryResult*) { return cudaErrorUnknown; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void**, unsigned, unsigned long long, cudaDriverEntryPointQueryResult*) { return cudaErrorUnknown; }
}
