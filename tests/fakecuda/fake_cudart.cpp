// A stand-in for the CUDA runtime, linked with the library's host code in place
// of the real one, so that its host side can be tested without a GPU: devices
// that each keep their own function attributes, allocations that are counted,
// launches that are checked against the attributes, recorded, and refused on
// request.  Device memory is host memory; of the kernels only what the host
// reads back is played (the state words, the final basis, the lane's rings).
#include <cuda_runtime_api.h>
#include <unistd.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

// What a kernel leaves for the host to read (fake_kernels.cu).
extern "C" void fake_play(const char* name, void** args);
extern "C" int fake_lane_running();
extern "C" int fake_plan_status, fake_plan_fail, fake_plan_k;   // what the next pivots end with

namespace {
constexpr int kSms = 152, kOptin = 232448, kPerSm = 233472, kReserved = 1024, kStatic = 1024;

std::recursive_mutex mu;
std::map<const void*, std::string>& names() {          // (filled by static constructors)
    static std::map<const void*, std::string> n;
    return n;
}
struct Attr {
    int smem = 0;
    bool wide = false;   // clusters of more than 8 blocks
};
std::map<std::pair<int, const void*>, Attr> attrs;   // of (device, kernel)
std::map<void*, size_t> blocks;                      // device allocations
size_t live = 0, peak = 0;
std::string log_text, refuse;
// A lane's launch: the event recorded behind it is ready once it has ended, and
// batch kernels launched meanwhile wait for that (fake_batch_waits).
cudaEvent_t lane_event = nullptr;
bool lane_launched = false;
int batch_waits = 0;
thread_local bool waits_for_lane = false;
thread_local int device = 0;
thread_local cudaError_t last = cudaSuccess;
struct Call {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
};
thread_local Call call;

cudaError_t fail(cudaError_t e) { return last = e; }
bool is(const std::string& name, const char* what) { return name.find(what) != std::string::npos; }

void* take(size_t bytes) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    void* p = calloc(1, bytes + 256);
    if (!p) return nullptr;
    blocks[p] = bytes;
    live += bytes;
    peak = live > peak ? live : peak;
    return p;
}
void give(void* p) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    auto it = blocks.find(p);
    if (it == blocks.end()) return;
    live -= it->second;
    blocks.erase(it);
    free(p);
}

cudaError_t launch(const void* f, dim3 grid, dim3 block, void** args, size_t smem, unsigned cluster) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    const std::string name = names().count(f) ? names()[f] : "?";
    const Attr at = attrs[{device, f}];
    char line[512];
    snprintf(line, sizeof line, "%d %s %u %u %zu\n", device, name.c_str(), grid.x * grid.y, block.x, smem);
    if (!refuse.empty() && is(name, refuse.c_str())) {
        log_text += std::string("refused ") + line;
        return fail(cudaErrorCooperativeLaunchTooLarge);
    }
    if (smem > (size_t)(at.smem ? at.smem : 48 * 1024) || (cluster > 8 && !at.wide)) {
        log_text += std::string("invalid ") + line;
        return fail(cudaErrorInvalidValue);
    }
    log_text += line;
    if (is(name, "k_team_serve")) lane_launched = true;
    if (is(name, "k_batch_solve") && batch_waits) waits_for_lane = true;
    fake_play(name.c_str(), args);
    return cudaSuccess;
}
}  // namespace

// ------------------------------------------------------------ the test's side
extern "C" {
void fake_reset() {
    std::lock_guard<std::recursive_mutex> lk(mu);
    log_text.clear();
    refuse.clear();
    fake_plan_status = fake_plan_fail = fake_plan_k = 0;
    peak = live;
}
void fake_plan(int status, int failed, int k) {
    fake_plan_status = status;
    fake_plan_fail = failed;
    fake_plan_k = k;
}
void fake_refuse(const char* what) { refuse = what; }
const char* fake_log() { return log_text.c_str(); }
long long fake_live() { return (long long)live; }
long long fake_peak() { return (long long)peak; }
void fake_batch_waits(int on) { batch_waits = on; }
void fake_set_device(int d) { device = d; }

// --------------------------------------------------------------- registration
void** __cudaRegisterFatBinary(void*) { return (void**)malloc(8); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*,
                            int*) {
    names()[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
    call = Call{g, b, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
    *g = call.grid;
    *b = call.block;
    *smem = call.smem;
    *(cudaStream_t*)s = call.stream;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** args, size_t smem, cudaStream_t) {
    return launch((const void*)k, g, b, args, smem, 1);
}
cudaError_t cudaLaunchKernel(const void* f, dim3 g, dim3 b, void** args, size_t smem, cudaStream_t) {
    return launch(f, g, b, args, smem, 1);
}
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3 g, dim3 b, void** args, size_t smem, cudaStream_t) {
    return launch(f, g, b, args, smem, 1);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
    unsigned cluster = 1;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[i].val.clusterDim.x;
    return launch(f, c->gridDim, c->blockDim, args, c->dynamicSmemBytes, cluster);
}

// --------------------------------------------------------------------- devices
cudaError_t cudaGetDevice(int* d) {
    *d = device;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
    device = d;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    switch (a) {
        case cudaDevAttrMultiProcessorCount: *v = kSms; break;
        case cudaDevAttrMaxSharedMemoryPerBlockOptin: *v = kOptin; break;
        case cudaDevAttrMaxSharedMemoryPerMultiprocessor: *v = kPerSm; break;
        case cudaDevAttrReservedSharedMemoryPerBlock: *v = kReserved; break;
        case cudaDevAttrCooperativeLaunch: *v = 1; break;
        default: *v = 0;
    }
    return cudaSuccess;
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "fake error"; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
    memset(a, 0, sizeof *a);
    a->sharedSizeBytes = kStatic;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
        if (v < 0 || v > kOptin - kStatic) return fail(cudaErrorInvalidValue);
        attrs[{device, f}].smem = v;
    } else if (a == cudaFuncAttributeNonPortableClusterSizeAllowed) {
        attrs[{device, f}].wide = v != 0;
    }
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int threads, size_t smem,
                                                                   unsigned) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    const Attr at = attrs[{device, f}];
    *n = 0;
    if (smem > (size_t)(at.smem ? at.smem : 48 * 1024)) return cudaSuccess;
    const int by_threads = is(names()[f], "k_pivot") ? (threads <= 256 ? 256 : threads) / threads : 512 / threads;
    const int by_smem = (int)(kPerSm / (smem + kStatic + kReserved));
    *n = by_threads < by_smem ? by_threads : by_smem;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    const Attr at = attrs[{device, f}];
    *n = 0;
    if (c->dynamicSmemBytes > (size_t)(at.smem ? at.smem : 48 * 1024) || (c->gridDim.x > 8 && !at.wide))
        return fail(cudaErrorInvalidValue);
    *n = 1;
    return cudaSuccess;
}

// ---------------------------------------------------------------------- memory
cudaError_t cudaMalloc(void** p, size_t n) { return (*p = take(n)) ? cudaSuccess : fail(cudaErrorMemoryAllocation); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) {
    *p = (cudaMemPool_t)1;
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaFree(void* p) {
    give(p);
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return (*p = calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFreeHost(void* p) {
    free(p);
    return cudaSuccess;
}
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) {
    *d = h;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t) {
    for (size_t i = 0; i < h; ++i) memcpy((char*)d + i * dp, (const char*)s + i * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) {
    memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
    memset(a, 0, sizeof *a);
    a->type = cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* s) {
    *p = (void*)s;
    return cudaSuccess;
}

// ---------------------------------------------------------- streams and events
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = (cudaStream_t)malloc(8);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    free(s);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
    while (waits_for_lane) {
        {
            std::lock_guard<std::recursive_mutex> lk(mu);
            waits_for_lane = fake_lane_running() != 0;
        }
        usleep(100);
    }
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* st) {
    *st = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return fail(cudaErrorNotSupported); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return fail(cudaErrorNotSupported); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return fail(cudaErrorNotSupported); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return fail(cudaErrorNotSupported); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    *e = (cudaEvent_t)malloc(8);
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    free(e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    if (lane_launched) {
        lane_event = e;
        lane_launched = false;
    }
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t e) {
    std::lock_guard<std::recursive_mutex> lk(mu);
    return e == lane_event && fake_lane_running() ? cudaErrorNotReady : cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.f;
    return cudaSuccess;
}
}
