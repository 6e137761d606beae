// A CUDA runtime for host tests of the library's host code: "device" memory is
// host memory, kernels do nothing, and the work of a stream runs when the stream
// is waited for, no earlier.  An upload from pageable memory that is still queued
// when its source changes (or is freed: freed memory is filled) is counted, pool
// memory is accounted as the driver does, and a kernel can be made to record an
// error code in its error word.
#include <cuda_runtime_api.h>
#include <malloc.h>

#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <vector>

namespace {

struct Pool {
    size_t used = 0, reserved = 0, most = 0;
};
struct Block {
    size_t bytes;
    Pool* pool;
};
std::recursive_mutex mu;
std::map<cudaStream_t, std::vector<std::function<void()>>> queues;
std::map<void*, Block> blocks;
std::set<void*> pinned;
Pool dflt;
std::map<const void*, std::string> kernels;
std::map<std::string, long long> launches;
std::string fail_name;
int fail_arg = 0, fail_code = 0;
long long stale_uploads = 0, uploads = 0;
const void* last_upload = nullptr;
thread_local struct {
    dim3 g, b;
    size_t s;
    cudaStream_t st;
} cfg;

#define LOCK std::lock_guard<std::recursive_mutex> lk(mu)

void run(cudaStream_t st) {
    std::vector<std::function<void()>> q;
    q.swap(queues[st]);
    for (auto& f : q) f();
}
void run_all() {
    std::vector<cudaStream_t> s;
    for (auto& q : queues) s.push_back(q.first);
    for (auto st : s) run(st);
}

bool is_pinned(const void* p) {
    for (void* b : pinned)
        if (p >= b && p < (char*)b + 65536) return true;
    return false;
}

cudaError_t alloc(void** p, size_t n, Pool& pool) {
    *p = aligned_alloc(512, (n + 511) & ~size_t(511));
    if (!*p) return cudaErrorMemoryAllocation;
    blocks[*p] = Block{n, &pool};
    pool.used += n;
    pool.reserved = std::max(pool.reserved, pool.used);
    pool.most = std::max(pool.most, pool.used);
    return cudaSuccess;
}

cudaError_t copy(void* dst, const void* src, size_t n, cudaMemcpyKind kind, cudaStream_t st) {
    if (kind != cudaMemcpyHostToDevice || is_pinned(src)) {
        queues[st].push_back([=] { memcpy(dst, src, n); });
        return cudaSuccess;
    }
    ++uploads;
    last_upload = dst;
    std::vector<char> now((const char*)src, (const char*)src + n);
    queues[st].push_back([=] {
        if (memcmp(now.data(), src, n) != 0) ++stale_uploads;
        memcpy(dst, now.data(), n);
    });
    return cudaSuccess;
}

cudaError_t launch(const void* f, void** args, cudaStream_t st) {
    const std::string& name = kernels[f];
    ++launches[name];
    if (!fail_name.empty() && name.find(fail_name) != std::string::npos) {
        int* word = *(int**)args[fail_arg];
        const int code = fail_code;
        queues[st].push_back([=] { *word = code; });
    }
    return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- the tests' side ----
// from now on: kernels whose name contains `name` write code to the word that
// their argument `arg` points to ("": none does)
void fake_fail(const char* name, int arg, int code) {
    LOCK;
    fail_name = name;
    fail_arg = arg;
    fail_code = code;
}
// freed memory is filled and stays mapped, so that a late read of it is seen
void fake_fill_freed(int on) {
    mallopt(M_MMAP_THRESHOLD, on ? 1 << 30 : 128 * 1024);
    mallopt(M_TRIM_THRESHOLD, on ? 1 << 30 : 128 * 1024);
    mallopt(M_PERTURB, on ? 0xa5 : 0);
}
long long fake_stale_uploads() { return stale_uploads; }
long long fake_uploads() { return uploads; }
// the start of the block that the last upload went to
const void* fake_last_upload_block() {
    LOCK;
    auto it = blocks.upper_bound(const_cast<void*>(last_upload));
    return it == blocks.begin() ? nullptr : (--it)->first;
}
long long fake_default_pool_most() { return (long long)dflt.most; }
long long fake_launches(const char* name) {
    LOCK;
    long long n = 0;
    for (auto& k : launches)
        if (k.first.find(name) != std::string::npos) n += k.second;
    return n;
}

// ---- launches ----
void** __cudaRegisterFatBinary(void*) {
    static void* h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    LOCK;
    kernels[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, cudaStream_t st) {
    cfg.g = g, cfg.b = b, cfg.s = s, cfg.st = st;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
    *g = cfg.g, *b = cfg.b, *s = cfg.s, *(cudaStream_t*)st = cfg.st;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t, cudaStream_t st) {
    LOCK;
    return launch((const void*)k, args, st);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
    LOCK;
    return launch(f, args, c->stream);
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }

// ---- device ----
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetStreamPriorityRange(int* lo, int* hi) {
    *lo = *hi = 0;
    return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    static void* m = aligned_alloc(512, 32 << 20);
    *p = m;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
    memset(a, 0, sizeof(*a));
    a->type = cudaMemoryTypeDevice;
    return cudaSuccess;
}

// ---- memory ----
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) {
    LOCK;
    return alloc(p, n, dflt);
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t pool, cudaStream_t) {
    LOCK;
    return alloc(p, n, *(Pool*)pool);
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t st) {
    LOCK;
    auto it = blocks.find(p);
    if (it == blocks.end()) return cudaErrorInvalidValue;
    it->second.pool->used -= it->second.bytes;
    blocks.erase(it);
    queues[st].push_back([=] { free(p); });
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
    LOCK;
    *p = calloc(1, std::max<size_t>(n, 65536));
    pinned.insert(*p);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
    LOCK;
    run_all();
    pinned.erase(p);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
    LOCK;
    return copy(d, s, n, k, st);
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    LOCK;
    run_all();
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
    LOCK;
    queues[st].push_back([=] { memset(d, v, n); });
    return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
    LOCK;
    run_all();
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) {
    *p = (cudaMemPool_t) new Pool();
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t p) {
    delete (Pool*)p;
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t p, cudaMemPoolAttr a, void* v) {
    LOCK;
    *(unsigned long long*)v = a == cudaMemPoolAttrReservedMemCurrent ? ((Pool*)p)->reserved : ((Pool*)p)->used;
    return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t keep) {
    LOCK;
    Pool& q = *(Pool*)p;
    q.reserved = std::max(q.used, std::min(q.reserved, keep));
    return cudaSuccess;
}

// ---- streams, events, graphs ----
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = (cudaStream_t)malloc(16);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t st) {
    LOCK;
    run(st);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t st) {
    LOCK;
    run(st);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = (cudaEvent_t)malloc(16);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    free((void*)e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) {
    LOCK;
    run_all();
    return cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaErrorNotReady; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.f;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

// ---- cuFFT: not reached by these tests ----
int cufftDestroy(int) { return 1; }
int cufftExecC2R(int, void*, void*) { return 1; }
int cufftExecR2C(int, void*, void*) { return 1; }
int cufftPlanMany(int*, int, int*, int*, int, int, int*, int, int, int, int) { return 1; }
int cufftSetStream(int, cudaStream_t) { return 1; }

}  // extern "C"
