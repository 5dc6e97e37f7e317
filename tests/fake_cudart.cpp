// A stand-in for the CUDA runtime, linked with the library's own object files in place of
// libcudart: no GPU, kernels do nothing, "device" memory is host memory.  It keeps what the
// host code asked for -- function attributes per device, launches with their stream, shared
// memory and cluster, streams with their priority -- and refuses what a GPU would refuse.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

namespace {

struct Stream {
    int priority, device;
    bool capturing;
};
struct Launch {
    std::string name;
    unsigned grid, block, cluster;
    size_t smem;
    int device, priority;
    bool captured, chained;
};

std::recursive_mutex mu;
std::map<const void*, std::string> names;                       // host stub -> device name
std::map<std::pair<int, const void*>, int> smem_limit;          // (device, function)
std::map<std::string, int> static_smem;                         // by a part of the name
std::vector<Launch> launches;
int devices = 1, clusters_fit = 1000;
thread_local int device = 0;
thread_local cudaError_t last = cudaSuccess;  // of the launches, for cudaGetLastError
thread_local struct { dim3 grid, block; size_t smem; cudaStream_t s; } call;
void (*attr_hook)() = nullptr;  // runs after every change of a function attribute

Stream* stream_of(cudaStream_t s) { return reinterpret_cast<Stream*>(s); }

int static_of(const void* f) {
    for (const auto& e : static_smem)
        if (names[f].find(e.first) != std::string::npos) return e.second;
    return 0;
}

int limit_of(const void* f) {  // of the dynamic shared memory, on the current device
    const auto lim = smem_limit.find({device, f});
    return lim == smem_limit.end() ? 48 * 1024 - static_of(f) : lim->second;
}

cudaError_t launch(const void* f, dim3 g, dim3 b, size_t smem, cudaStream_t s, unsigned cluster,
                   bool chained) {
    std::lock_guard<std::recursive_mutex> l(mu);
    const int most = limit_of(f);
    Stream* st = stream_of(s);
    if (st && st->device != device) return cudaErrorInvalidResourceHandle;
    if ((long long)smem > most) return cudaErrorInvalidValue;
    if (cluster > 8 && clusters_fit == 0) return cudaErrorLaunchOutOfResources;
    launches.push_back({names[f], g.x, b.x, cluster, smem, device, st ? st->priority : 0,
                        st && st->capturing, chained});
    return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- what the tests use ----
void fake_reset(int n_devices) {  // the attributes stay, as a process keeps them
    std::lock_guard<std::recursive_mutex> l(mu);
    static_smem.clear();
    launches.clear();
    devices = n_devices;
    clusters_fit = 1000;
    device = 0;
    attr_hook = nullptr;
}
void fake_set_device(int d) { device = d; }
int fake_device() { return device; }
void fake_static_smem(const char* part, int bytes) { static_smem[part] = bytes; }
void fake_clusters_fit(int n) { clusters_fit = n; }  // clusters of more than eight CTAs
void fake_attr_hook(void (*f)()) { attr_hook = f; }
void fake_capture(void* s, int on) { stream_of((cudaStream_t)s)->capturing = on != 0; }
void* fake_stream(int priority) { return new Stream{priority, device, false}; }
int fake_launches() { return (int)launches.size(); }
// field of launch k: 0 grid, 1 block, 2 cluster, 3 shared memory, 4 device, 5 priority, 6 captured,
// 7 chained
long long fake_launch(int k, int field, char* name, int room) {
    const Launch& x = launches[k];
    std::strncpy(name, x.name.c_str(), room - 1);
    name[room - 1] = 0;
    const long long v[8] = {x.grid, x.block, x.cluster, (long long)x.smem, x.device, x.priority,
                            x.captured, x.chained};
    return v[field];
}

// ---- registration and launches ----
void** __cudaRegisterFatBinary(void*) {
    static void* h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*,
                            dim3*, dim3*, int*) {
    names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, cudaStream_t s) {
    call = {g, b, sm, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* sm, void* s) {
    *g = call.grid;
    *b = call.block;
    *sm = call.smem;
    *(cudaStream_t*)s = call.s;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t sm, cudaStream_t s) {
    return last = launch((const void*)k, g, b, sm, s, 1, false);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
    unsigned cluster = 1;
    bool chained = false;
    for (unsigned k = 0; k < c->numAttrs; ++k)
        if (c->attrs[k].id == cudaLaunchAttributeClusterDimension)
            cluster = c->attrs[k].val.clusterDim.x;
        else if (c->attrs[k].id == cudaLaunchAttributeProgrammaticStreamSerialization)
            chained = c->attrs[k].val.programmaticStreamSerializationAllowed != 0;
    return launch(f, c->gridDim, c->blockDim, c->dynamicSmemBytes, c->stream, cluster, chained);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
        std::lock_guard<std::recursive_mutex> l(mu);
        if (v + static_of(f) > 227 * 1024) return cudaErrorInvalidValue;
        smem_limit[{device, f}] = v;
    }
    if (attr_hook) attr_hook();
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void* f) {
    std::memset(a, 0, sizeof(*a));
    a->sharedSizeBytes = (size_t)static_of(f);
    a->maxDynamicSharedSizeBytes = limit_of(f);
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
    *n = clusters_fit;
    return cudaSuccess;
}

// ---- memory: the host's ----
cudaError_t cudaMalloc(void** p, size_t n) {
    *p = std::calloc(1, n);
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void* p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy2D(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h,
                         cudaMemcpyKind) {
    for (size_t y = 0; y < h; ++y) std::memcpy((char*)d + y * dp, (const char*)s + y * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) {
    std::memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
    std::memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* s) {
    *p = const_cast<void*>(s);
    return cudaSuccess;
}

// ---- devices, streams, events, graphs ----
cudaError_t cudaGetDevice(int* d) {
    *d = device;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
    if (d < 0 || d >= devices) return cudaErrorInvalidDevice;
    device = d;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetStreamPriorityRange(int* least, int* greatest) {
    *least = 0;
    *greatest = -5;
    return cudaSuccess;
}
cudaError_t cudaStreamGetPriority(cudaStream_t s, int* p) {
    *p = s ? stream_of(s)->priority : 0;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int p) {
    p = p > 0 ? 0 : p < -5 ? -5 : p;  // the runtime clamps a priority to the range
    *s = (cudaStream_t)fake_stream(p);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    delete stream_of(s);
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
    if (!s || stream_of(s)->capturing) return cudaErrorStreamCaptureUnsupported;
    stream_of(s)->capturing = true;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
    stream_of(s)->capturing = false;
    *g = (cudaGraph_t) new int(0);
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st) {
    *st = s && stream_of(s)->capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    return s && stream_of(s)->capturing ? cudaErrorStreamCaptureUnsupported : cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = (cudaEvent_t) new int(0);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    delete (int*)e;
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.0f;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
    *x = (cudaGraphExec_t) new int(0);
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
    delete (int*)g;
    return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) {
    delete (int*)x;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}

}  // extern "C"
