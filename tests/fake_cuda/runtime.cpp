// A CUDA runtime without a GPU, for tests of the engine's host side: device memory is host memory, kernels
// do not run but are counted by name, graphs replay what was launched while they were captured, and the
// event clock advances by a settable time per kernel launch (resident marches: per launch of the most indices).
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "kernels.h"

namespace {

std::mutex mu;
std::map<const void *, std::string> names;   // registered kernels
std::map<std::string, int64_t> counts;       // launches by kernel name
std::vector<std::pair<std::string, double>> costs;
int64_t queries = 0, captures = 0, host_frees = 0;
double clock_ms = 0;
int fail_resident = 0;                       // resident launches report a wait that ran out
int fail_late = 0;                           // 1: copies back never land, and the stream fails from the first look at one on (2)
bool capturing = false;
std::vector<std::string> captured;
thread_local int device = 0;

struct Event { double at = 0; };
struct Graph { std::vector<std::string> kernels; };

void run(const std::string &k, double part = 1)
{
    if (capturing) {
        captured.push_back(k);
        return;
    }
    ++counts[k];
    for (const auto &c : costs)
        if (k.find(c.first) != std::string::npos) {
            clock_ms += part * c.second;
            break;
        }
}

cudaError_t launch(const void *f, double part = 1)
{
    std::lock_guard<std::mutex> lk(mu);
    auto it = names.find(f);
    if (it == names.end()) return cudaErrorInvalidDeviceFunction;
    run(it->second, part);
    return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- what tests read and set -----------------------------------------------------------
int64_t fake_launches(const char *part)
{
    std::lock_guard<std::mutex> lk(mu);
    int64_t n = 0;
    for (const auto &c : counts)
        if (c.first.find(part) != std::string::npos) n += c.second;
    return n;
}
int64_t fake_queries() { return queries; }
int64_t fake_captures() { return captures; }
void fake_cost(const char *part, double ms) { costs.insert(costs.begin(), {part, ms}); }
int64_t fake_host_frees() { return host_frees; }
void fake_fail_late(int on) { fail_late = on; }
void fake_fail_resident(int on) { fail_resident = on; }
// The first `most` shapes of the resident march and the model's clocks for each, in the order they come.
int fake_res_shapes(int cyl, int fp64, int nx, int ny, int nsims, int most, int *rows_cluster, double *clocks)
{
    cas::ResShapes shapes(cyl, fp64, nx, ny, nsims);
    cas::Res2dShape q;
    int n = 0;
    while (n < most && shapes.next(&q, &clocks[n])) rows_cluster[n++] = 100 * q.rb + q.cluster;
    return n;
}
int fake_device(int set)
{
    if (set >= 0) device = set;
    return device;
}
void fake_reset()
{
    std::lock_guard<std::mutex> lk(mu);
    counts.clear();
    costs.clear();
    queries = captures = host_frees = 0;
    fail_resident = fail_late = 0;
    clock_ms = 0;
}

// ---- kernels ---------------------------------------------------------------------------
void **__cudaRegisterFatBinary(void *) { return (void **)calloc(1, sizeof(void *)); }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *)
{
    std::lock_guard<std::mutex> lk(mu);
    names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *s, void *st)
{
    *g = *b = dim3(1);
    *s = 0;
    *(cudaStream_t *)st = nullptr;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f)
{
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t, cudaStream_t) { return launch((const void *)k); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *f, void **args)
{
    if (fail_resident) *(*(const cas::DevRes *const *)args[0])->status = 1;
    return launch(f, *(const int *)args[2] / (double)cas::RES_LAUNCH_INDICES);
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
// clusters that fit 152 SMs of 228 KB shared memory and 64 K registers (128 a thread), in one pool
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *c)
{
    ++queries;
    const int smem = 228 * 1024 / ((int)c->dynamicSmemBytes + 2048), regs = 65536 / (128 * (int)c->blockDim.x);
    *n = 152 * (smem < regs ? smem : regs) / (int)c->attrs[0].val.clusterDim.x;
    return cudaSuccess;
}

// ---- device, memory --------------------------------------------------------------------
cudaError_t cudaGetDeviceCount(int *n) { *n = 2; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { device = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }   // asked for the SMs alone
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) { *f = *t = (size_t)4 << 30; return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { *p = calloc(1, n); return *p ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void *p)
{
    ++host_frees;
    return cudaFree(p);
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorInvalidValue; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "error of the fake runtime"; }

// ---- streams, events, graphs -----------------------------------------------------------
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return fail_late == 2 ? cudaErrorLaunchFailure : cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t) new Event; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete (Event *)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { ((Event *)e)->at = clock_ms; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t)
{
    if (fail_late) fail_late = 2;
    return fail_late ? cudaErrorNotReady : cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b)
{
    *ms = (float)(((Event *)b)->at - ((Event *)a)->at);
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode)
{
    capturing = true;
    captured.clear();
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g)
{
    capturing = false;
    ++captures;
    *g = (cudaGraph_t) new Graph{captured};
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long)
{
    *x = (cudaGraphExec_t) new Graph(*(Graph *)g);
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete (Graph *)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { delete (Graph *)x; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t)
{
    std::lock_guard<std::mutex> lk(mu);
    for (const auto &k : ((Graph *)x)->kernels) run(k);
    return cudaSuccess;
}

}  // extern "C"
