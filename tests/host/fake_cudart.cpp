// fake_cudart.cpp -- a CUDA runtime on the host for tests of the library's host
// side: several devices whose work is done when it is waited for, memory of a
// stated capacity, memory pools, graphs, and calls that fail when told to.
// Kernels do nothing.  It counts two things that must not happen: memory
// given back while work is outstanding on its device, and a graph launch that
// uses memory given back before.
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <mutex>
#include <set>
#include <string>
#include <vector>

namespace {
std::recursive_mutex mu;
typedef std::lock_guard<std::recursive_mutex> Lock;

struct Block {
    size_t bytes;
    int dev;
    bool pooled, live;
};
struct Graph {
    std::vector<const void *> uses;
};
int n_devices = 1;
thread_local int current = 0;
thread_local cudaError_t last = cudaSuccess;
std::map<const char *, Block> blocks;
std::map<std::pair<int, const void *>, bool> busy;  // (device, stream)
std::map<const void *, int> stream_dev;
std::map<const void *, Graph *> capturing;
std::set<const void *> execs;
std::map<int, size_t> used, idle;  // live bytes, unused bytes the pools keep
size_t capacity = (size_t)1 << 40;
size_t keep = 0;  // the pools' release threshold
long violations = 0;
std::map<const void *, int> smem_limit;  // per kernel
struct Fail {
    int after, count;
};
std::map<std::string, Fail> fails;

bool fails_now(const char *fn) {
    auto it = fails.find(fn);
    if (it == fails.end()) return false;
    if (it->second.after-- > 0) return false;
    if (it->second.count-- > 0) return true;
    return false;
}
cudaError_t ret(cudaError_t e) {
    if (e != cudaSuccess) last = e;
    return e;
}
int dev_of(const void *stream) { return stream ? stream_dev[stream] : current; }
void work(const void *stream, const void *use) {
    auto it = capturing.find(stream);
    if (it != capturing.end())
        it->second->uses.push_back(use);
    else
        busy[{dev_of(stream), stream}] = true;
}
bool device_busy(int dev) {
    for (auto &b : busy)
        if (b.first.first == dev && b.second) return true;
    return false;
}
void wait_device(int dev) {
    for (auto &b : busy)
        if (b.first.first == dev) b.second = false;
}
const Block *block_of(const void *p) {
    auto it = blocks.upper_bound((const char *)p);
    if (it == blocks.begin()) return nullptr;
    --it;
    return (const char *)p < it->first + it->second.bytes ? &it->second : nullptr;
}
cudaError_t allocate(void **p, size_t bytes, int dev, bool pooled) {
    size_t &id = idle[dev];
    const size_t from_idle = pooled ? (id < bytes ? id : bytes) : 0;
    if (used[dev] + id - from_idle + bytes > capacity) return ret(cudaErrorMemoryAllocation);
    id -= from_idle;
    used[dev] += bytes;
    *p = calloc(1, bytes ? bytes : 1);  // never reused: addresses of freed blocks stay known
    blocks[(const char *)*p] = Block{bytes, dev, pooled, true};
    return cudaSuccess;
}
cudaError_t release(void *p, bool async) {
    if (!p) return cudaSuccess;
    auto it = blocks.find((const char *)p);
    if (it == blocks.end() || !it->second.live) {
        ++violations;
        return ret(cudaErrorInvalidValue);
    }
    Block &b = it->second;
    if (async && device_busy(b.dev)) ++violations;
    if (!async) wait_device(b.dev);  // cudaFree waits for the block's device
    b.live = false;
    used[b.dev] -= b.bytes;
    if (b.pooled) idle[b.dev] = idle[b.dev] + b.bytes < keep ? idle[b.dev] + b.bytes : keep;
    return cudaSuccess;
}
cudaError_t launch(const void *fn, size_t smem, cudaStream_t s) {
    const auto it = smem_limit.find(fn);
    if (smem > (size_t)(it == smem_limit.end() ? 48 * 1024 : it->second)) return ret(cudaErrorInvalidValue);
    work(s, nullptr);
    return cudaSuccess;
}
}  // namespace

extern "C" {
void fake_reset(int devices) {
    Lock l(mu);
    n_devices = devices, current = 0, last = cudaSuccess, violations = 0;
    capacity = (size_t)1 << 40;
    fails.clear(), busy.clear();
}
void fake_fail(const char *fn, int after, int count) {
    Lock l(mu);
    fails[fn] = Fail{after, count};
}
void fake_fail_none() {
    Lock l(mu);
    fails.clear();
}
int fake_failed(const char *fn) {  // whether a call told to fail has done so
    Lock l(mu);
    return fails.count(fn) && fails[fn].after < 0;
}
void fake_capacity(size_t bytes) { capacity = bytes; }
size_t fake_used(int dev) { return used[dev]; }
size_t fake_idle(int dev) { return idle[dev]; }
long fake_violations() { return violations; }

cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
cudaError_t cudaGetDevice(int *d) {
    *d = current;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
    if (d < 0 || d >= n_devices) return ret(cudaErrorInvalidDevice);
    current = d;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    Lock l(mu);
    if (!capturing.empty()) return ret(cudaErrorStreamCaptureUnsupported);
    wait_device(current);
    return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t bytes) {
    Lock l(mu);
    if (fails_now("alloc")) return ret(cudaErrorMemoryAllocation);
    return allocate(p, bytes, current, false);
}
cudaError_t cudaFree(void *p) {
    Lock l(mu);
    return release(p, false);
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t *pool, const cudaMemPoolProps *props) {
    *pool = (cudaMemPool_t)(size_t)(props->location.id + 1);
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr a, void *v) {
    if (a == cudaMemPoolAttrReleaseThreshold) keep = *(unsigned long long *)v;
    return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t pool, size_t bytes) {
    Lock l(mu);
    size_t &id = idle[(int)(size_t)pool - 1];
    id = id < bytes ? id : bytes;
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void **p, size_t bytes, cudaMemPool_t pool, cudaStream_t) {
    Lock l(mu);
    if (fails_now("alloc")) return ret(cudaErrorMemoryAllocation);
    return allocate(p, bytes, (int)(size_t)pool - 1, true);
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t) {
    Lock l(mu);
    return release(p, true);
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    Lock l(mu);
    if (fails_now("copy")) return ret(cudaErrorUnknown);
    memcpy(d, s, n);
    work(st, d);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t st) {
    Lock l(mu);
    memset(d, v, n);
    work(st, d);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) {
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaHostRegister(void *, size_t, unsigned) { return cudaSuccess; }
cudaError_t cudaHostUnregister(void *) { return cudaSuccess; }

cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    Lock l(mu);
    if (fails_now("stream")) return ret(cudaErrorUnknown);
    *s = (cudaStream_t)malloc(16);
    stream_dev[*s] = current;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    Lock l(mu);
    if (capturing.count(s)) return ret(cudaErrorStreamCaptureUnsupported);
    busy[{dev_of(s), s}] = false;
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
    Lock l(mu);
    capturing[s] = new Graph;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g) {
    Lock l(mu);
    *g = (cudaGraph_t)capturing[s];
    capturing.erase(s);
    if (fails_now("capture")) {
        *g = nullptr;
        return ret(cudaErrorStreamCaptureInvalidated);
    }
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t g, unsigned long long) {
    Lock l(mu);
    if (fails_now("instantiate") || !g) return ret(cudaErrorUnknown);
    *e = (cudaGraphExec_t) new Graph(*(Graph *)g);
    execs.insert(*e);
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t s) {
    Lock l(mu);
    if (!execs.count(e)) return ret(cudaErrorInvalidValue);
    for (const void *p : ((Graph *)e)->uses) {
        const Block *b = p ? block_of(p) : nullptr;
        if (b && !b->live) ++violations;
    }
    work(s, nullptr);
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
    Lock l(mu);
    execs.erase(e);
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) {
    *e = (cudaEvent_t)malloc(16);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.f;
    return cudaSuccess;
}

cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
    Lock l(mu);
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) smem_limit[f] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
    Lock l(mu);
    return launch(f, c->dynamicSmemBytes, c->stream);
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t smem, cudaStream_t s) {
    Lock l(mu);
    return launch(k, smem, s);
}
static thread_local struct {
    dim3 g, b;
    size_t smem;
    void *stream;
} config;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, void *stream) {
    config.g = g, config.b = b, config.smem = smem, config.stream = stream;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *stream) {
    *g = config.g, *b = config.b, *smem = config.smem, *(void **)stream = config.stream;
    return cudaSuccess;
}
void **__cudaRegisterFatBinary(void *) {
    static void *h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
cudaError_t cudaGetSymbolAddress(void **, const void *) { return ret(cudaErrorInvalidSymbol); }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *) {
    return ret(cudaErrorUnknown);
}
}
