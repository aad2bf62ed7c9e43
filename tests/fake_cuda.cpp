// A stand-in for the CUDA runtime, linked with the host runtime (st_runtime.cu)
// and stand-ins for the kernel launchers (fake_launch.cu) to run it without a
// GPU.
//
// Streams and events carry the set of operations they are ordered after, so a
// test can ask whether a stream waits for everything another one was given;
// one launch can be made to fail; device memory has a size limit.  Device
// pointers are never dereferenced.
#include <cstdint>
#include <cstdlib>
#include <set>
#include <string>
#include <vector>

#include <cuda_runtime_api.h>

namespace {
typedef std::set<int> Ops;
struct Stream { Ops ops; int own = 0; };
struct Event { Ops ops; };
Stream g_null;
std::vector<Stream*> g_streams;
std::vector<std::string> g_names;  // of the launches so far
int g_op = 0, g_fail = -1;
size_t g_limit = ~size_t(0), g_used = 0;
std::vector<std::pair<char*, size_t>> g_mem;
uintptr_t g_next = uintptr_t(1) << 40;

Stream* str(cudaStream_t s) { return s ? reinterpret_cast<Stream*>(s) : &g_null; }
Event* evt(cudaEvent_t e) { return reinterpret_cast<Event*>(e); }
}  // namespace

cudaError_t fake_launch(const char* name, cudaStream_t s, cudaEvent_t started) {
    const int k = static_cast<int>(g_names.size());
    g_names.push_back(name);
    if (k == g_fail) return cudaErrorLaunchOutOfResources;
    if (started) evt(started)->ops = str(s)->ops;  // (only that the launch has begun)
    str(s)->ops.insert(g_op++);
    str(s)->own++;
    return cudaSuccess;
}

// what the tests ask
extern "C" {
void fake_reset(int fail_launch, int64_t mem_limit) {
    g_names.clear();
    g_fail = fail_launch;
    g_limit = mem_limit < 0 ? ~size_t(0) : size_t(mem_limit);
}
int64_t fake_used() { return static_cast<int64_t>(g_used); }
int fake_launches() { return static_cast<int>(g_names.size()); }
const char* fake_launch_name(int k) { return g_names[k].c_str(); }
void* fake_stream() {
    g_streams.push_back(new Stream());
    return g_streams.back();
}
// operations given to any other stream that `s` is not ordered after
int fake_unjoined(void* s) {
    int n = 0;
    for (Stream* t : g_streams)
        for (int op : t->ops) n += !str(static_cast<cudaStream_t>(s))->ops.count(op);
    return n;
}
// operations given to streams other than `s`
int fake_elsewhere(void* s) {
    int n = 0;
    for (Stream* t : g_streams)
        if (t != s) n += t->own;
    return n;
}

// the CUDA runtime
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 232448;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
    if (n > g_limit || g_used > g_limit - n) return cudaErrorMemoryAllocation;
    *p = reinterpret_cast<void*>(g_next);
    g_next += (n + 511) & ~size_t(511);
    g_mem.push_back({static_cast<char*>(*p), n});
    g_used += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    for (auto& m : g_mem)
        if (m.first == p) {
            g_used -= m.second;
            m = {nullptr, 0};
        }
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return (*p = malloc(n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFreeHost(void* p) {
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t s) {
    str(s)->ops.insert(g_op++);
    str(s)->own++;
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = static_cast<cudaStream_t>(fake_stream());
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    for (size_t k = 0; k < g_streams.size(); ++k)
        if (g_streams[k] == str(s)) {
            delete g_streams[k];
            g_streams.erase(g_streams.begin() + k);
            break;
        }
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* st) {
    *st = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    *e = reinterpret_cast<cudaEvent_t>(new Event());
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    delete evt(e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    evt(e)->ops = str(s)->ops;
    return cudaSuccess;
}
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t s, unsigned) { return cudaEventRecord(e, s); }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    str(s)->ops.insert(evt(e)->ops.begin(), evt(e)->ops.end());
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 0.f;
    return cudaSuccess;
}
}  // extern "C"
