// A CUDA runtime on host memory, for CPU tests of the library's host code
// (gm_api.cu, linked with this file instead of the CUDA runtime and the kernel
// files).  Copies and memsets happen at once.  A transport launch is pending on
// its stream until the host waits for it; what it does is to leave records in
// its photon out-queue as often as host_cuda_leave() asked.  Calls are counted by
// name, and host_cuda_fail() makes one of them fail.
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "gm_host.h"

namespace {

struct Stream {
    long issued = 0, done = 0;
    struct Graph *capture = nullptr;
};
struct Event {
    Stream *s = nullptr;
    long at = 0;
};
struct Node {
    int kind;  // 0 copy, 1 kernel
    void *dst;
    const void *src;
    size_t n;
    const void *fn;
    unsigned shared;  // bytes of dynamic shared memory
    gm::TransportArgs args;
};
struct Graph {
    std::vector<Node *> nodes;
};
struct Exec {
    std::vector<Node> nodes;
    std::vector<const Node *> of;  // the graph's nodes they were made from
};

std::map<std::string, long> calls;
std::map<std::string, long> fail_at;
int leave = 0;
long misfits = 0;
std::vector<Stream *> streams;
std::vector<const void *> launched;  // compiled kernels, by launch

bool fails(const char *name) {
    const long n = ++calls[name];
    auto it = fail_at.find(name);
    return it != fail_at.end() && it->second == n;
}
#define CALL(name) \
    if (fails(#name)) return cudaErrorUnknown

Stream *of(cudaStream_t s) { return (Stream *)s; }

void kernel(const gm::TransportArgs &a, const void *fn, unsigned shared, Stream *s) {
    ++s->issued;
    if (shared != gm::transport_smem_bytes(a.tab_bytes)) ++misfits;
    launched.push_back(fn);
    if (leave > 0) {
        --leave;
        *a.out[0].cursor = 3;
    }
}

}  // namespace

extern "C" {

// Test interface.
void host_cuda_reset() {
    calls.clear();
    fail_at.clear();
    launched.clear();
    leave = 0;
    misfits = 0;
}
void host_cuda_leave(int launches) { leave = launches; }
void host_cuda_fail(const char *name, int nth_from_now) { fail_at[name] = calls[name] + nth_from_now; }
long host_cuda_calls(const char *name) { return calls[name]; }
long host_cuda_pending() {
    long n = 0;
    for (Stream *s : streams) n += s->issued - s->done;
    return n;
}
// launches whose shared memory is not the size their tables take
long host_cuda_misfits() { return misfits; }
long host_cuda_launched(const void **fn, long max) {
    for (long i = 0; i < max && i < (long)launched.size(); ++i) fn[i] = launched[i];
    return (long)launched.size();
}

// The runtime.
#ifndef __CUDA_ARCH__
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { return *n = 1, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 2, cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) { return *f = *t = 1ull << 30, cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int *l, int *g) { return *l = 0, *g = -1, cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) {
    CALL(cudaMalloc);
    *p = calloc(1, n);
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void *p) { return free(p), cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { return *p = malloc(n), cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMallocHost(p, n); }
cudaError_t cudaFreeHost(void *p) { return free(p), cudaSuccess; }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned, int) {
    streams.push_back(new Stream);
    return *s = (cudaStream_t)streams.back(), cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    for (size_t i = 0; i < streams.size(); ++i)
        if (streams[i] == of(s)) streams.erase(streams.begin() + i);
    return delete of(s), cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    CALL(cudaStreamSynchronize);
    of(s)->done = of(s)->issued;
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) {
    CALL(cudaStreamWaitEvent);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return *e = (cudaEvent_t) new Event, cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return delete (Event *)e, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    CALL(cudaEventRecord);
    *(Event *)e = Event{of(s), of(s)->issued};
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
    CALL(cudaEventSynchronize);
    const Event &v = *(Event *)e;
    if (v.s && v.s->done < v.at) v.s->done = v.at;
    return cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t e) { return cudaEventSynchronize(e); }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.f, cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) {
    CALL(cudaMemsetAsync);
    memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    CALL(cudaMemcpyAsync);
    if (of(st)->capture)
        of(st)->capture->nodes.push_back(new Node{0, d, s, n, nullptr, 0, {}});
    else
        memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus *c) {
    *c = of(s)->capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
    CALL(cudaStreamBeginCapture);
    of(s)->capture = new Graph;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g) {
    *g = (cudaGraph_t)of(s)->capture;
    of(s)->capture = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long) {
    CALL(cudaGraphInstantiate);
    Exec *e = new Exec;
    for (const Node *n : ((Graph *)g)->nodes) e->nodes.push_back(*n), e->of.push_back(n);
    return *x = (cudaGraphExec_t)e, cudaSuccess;
}
cudaError_t cudaGraphGetNodes(cudaGraph_t g, cudaGraphNode_t *nodes, size_t *n) {
    CALL(cudaGraphGetNodes);
    const Graph &G = *(Graph *)g;
    if (nodes)
        for (size_t i = 0; i < *n; ++i) nodes[i] = (cudaGraphNode_t)G.nodes[i];
    *n = G.nodes.size();
    return cudaSuccess;
}
cudaError_t cudaGraphNodeGetType(cudaGraphNode_t n, cudaGraphNodeType *t) {
    *t = ((Node *)n)->kind ? cudaGraphNodeTypeKernel : cudaGraphNodeTypeMemcpy;
    return cudaSuccess;
}
cudaError_t cudaGraphKernelNodeGetParams(cudaGraphNode_t n, cudaKernelNodeParams *p) {
    memset(p, 0, sizeof *p);
    p->func = const_cast<void *>(((Node *)n)->fn);
    p->sharedMemBytes = ((Node *)n)->shared;
    return cudaSuccess;
}
cudaError_t cudaGraphExecKernelNodeSetParams(cudaGraphExec_t x, cudaGraphNode_t n, const cudaKernelNodeParams *p) {
    CALL(cudaGraphExecKernelNodeSetParams);
    Exec &e = *(Exec *)x;
    for (size_t i = 0; i < e.nodes.size(); ++i)
        if (e.of[i] == (const Node *)n) {
            e.nodes[i].fn = p->func;
            e.nodes[i].shared = p->sharedMemBytes;
            e.nodes[i].args = *(const gm::TransportArgs *)p->kernelParams[0];
            return cudaSuccess;
        }
    return cudaErrorInvalidValue;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) {
    CALL(cudaGraphLaunch);
    for (const Node &n : ((Exec *)x)->nodes) {
        if (n.kind)
            kernel(n.args, n.fn, n.shared, of(s));
        else
            memcpy(n.dst, n.src, n.n);
    }
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
    for (Node *n : ((Graph *)g)->nodes) delete n;
    return delete (Graph *)g, cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) {
    CALL(cudaGraphExecDestroy);
    return delete (Exec *)x, cudaSuccess;
}

// no kernels are compiled in: nothing to register
void **__cudaRegisterFatBinary(void *) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
#endif

}  // extern "C"

// The kernel files' host side.
namespace gm {
cudaError_t launch_build_tables(const gpumcd_material *, int, const TableGeom &, double, double, float *,
                                cudaStream_t) { return cudaSuccess; }
cudaError_t launch_grid_energies(const TableGeom &, float *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_pack_phantom(const uint8_t *, const float *, uint64_t, int, uint32_t *, unsigned int *, int *,
                                cudaStream_t) { return cudaSuccess; }
cudaError_t launch_majorants(const float *, const unsigned int *, int, float *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_spectrum(const double *, const double *, int, float *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_fold(const unsigned long long *, const uint32_t *, uint64_t, int, uint64_t, double, double *,
                        double *, unsigned long long *, unsigned long long *, int, cudaStream_t) { return cudaSuccess; }
int sthr_blocks(uint64_t, int) { return 1; }
cudaError_t launch_sthr(const double *, const double *, uint64_t, double, void *, unsigned long long *,
                        const unsigned long long *, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_fold_noalloc(int, const unsigned long long *, const uint32_t *, uint64_t, int, uint64_t, double,
                                double, double *, double *, cudaStream_t, unsigned long long *) { return cudaSuccess; }
cudaError_t launch_philox(const uint32_t *, uint2, uint64_t, int, uint32_t *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_group_order(const PlanDev &, uint32_t, unsigned *, uint16_t *, uint32_t *, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t launch_debug_sample(const float *, const Phys &, int, float, int, const float *, int, uint64_t, uint64_t,
                                float *, cudaStream_t) { return cudaSuccess; }
size_t transport_smem_bytes(uint32_t tab_bytes) { return 16384 + tab_bytes; }
cudaError_t transport_configure() { return cudaSuccess; }
// one compiled kernel for each combination of the two, as far as host code can tell
const void *transport_kernel(const TransportArgs &a, int, int) {
    static const char k[4] = {};
    return &k[(a.n_plans == 1) + 2 * (a.phsp != 0)];
}
cudaError_t launch_transport(const TransportArgs &a, int grid, int block, int bps, cudaStream_t s) {
    if (fails("launch_transport")) return cudaErrorUnknown;
    const void *fn = transport_kernel(a, block, bps);
    const unsigned shared = (unsigned)transport_smem_bytes(a.tab_bytes);
    if (of(s)->capture)
        of(s)->capture->nodes.push_back(new Node{1, nullptr, nullptr, 0, fn, shared, a});
    else
        kernel(a, fn, shared, of(s));
    (void)grid;
    return cudaSuccess;
}
}  // namespace gm
