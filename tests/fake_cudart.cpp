// A stand-in for the CUDA runtime, for tests of the library's host code without
// a GPU: it is linked with the library's objects, kernels are recorded instead
// of run, device pointers are numbers, and memory is a budget.  It keeps the
// rules of the runtime that the host code has to respect: the opt-in to more
// than 48 KB of dynamic shared memory belongs to the device, a launch without
// it fails, nothing is allocated while a stream is captured unless the thread
// asked for it, a graph with allocation nodes is instantiated once, and what a
// graph refers to has to be there when it runs.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <set>
#include <string>
#include <vector>

namespace {

struct Launch {
    std::string name;
    std::vector<uintptr_t> needs;  // allocations a recorded launch refers to
};
struct UserObject {
    void *ptr;
    cudaHostFn_t destroy;
    int refs;
};
struct Graph {
    std::vector<Launch> launches;
    std::vector<UserObject *> objects;
    bool alloc_nodes = false;
    int execs = 0;
};
struct Exec {
    std::vector<Launch> launches;
    std::vector<UserObject *> objects;
    Graph *from;
};
struct Pool {
    size_t used = 0, held = 0;
    uint64_t keep = 0;
};

int device = 0;
cudaError_t last = cudaSuccess;
size_t budget = (size_t)1 << 40, used = 0;
uintptr_t next_ptr = 1ull << 32;
std::map<uintptr_t, size_t> live;                        // cudaMalloc
std::map<uintptr_t, std::pair<Pool *, size_t>> pooled;   // from a pool
std::map<const void *, std::string> names;
std::map<std::pair<int, const void *>, int> smem_limit;
std::map<cudaStream_t, Graph *> capturing;
std::set<Pool *> pools;
int capture_mode = cudaStreamCaptureModeGlobal;
int fill = 0;  // byte that results of 16 bytes or more consist of
long fail_skip = -1, fail_count = 0;
std::string record;
struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
} config;

cudaError_t fail(cudaError_t e) { return last = e; }
void log(const std::string &s) { record += s + "\n"; }

size_t pool_held() {
    size_t n = 0;
    for (Pool *p : pools) n += p->held;
    return n;
}
bool refused(size_t n) {
    if (fail_skip == 0 && fail_count > 0) {
        fail_count--;
        return true;
    }
    if (fail_skip > 0) fail_skip--;
    return used + pool_held() + n > budget;
}
uintptr_t fresh(size_t n) {
    const uintptr_t p = next_ptr;
    next_ptr += (n + 0xffff) & ~(size_t)0xffff;
    return p;
}
bool capture_forbids() { return !capturing.empty() && capture_mode != cudaStreamCaptureModeRelaxed; }

void release(std::vector<UserObject *> &objects) {
    for (UserObject *o : objects)
        if (--o->refs == 0) {
            o->destroy(o->ptr);
            delete o;
        }
    objects.clear();
}

}  // namespace

extern "C" {

// ---- control, for the tests ---------------------------------------------------
void fake_reset() {
    device = 0;
    last = cudaSuccess;
    budget = (size_t)1 << 40;
    fail_skip = -1;
    fail_count = 0;
    fill = 0;
    capture_mode = cudaStreamCaptureModeGlobal;
    record.clear();
}
void fake_budget(size_t bytes) { budget = bytes; }
size_t fake_used() { return used + pool_held(); }
// after `skip` more allocations, `count` of them are refused
void fake_refuse(long skip, long count) {
    fail_skip = skip;
    fail_count = count;
}
void fake_fill(int byte) { fill = byte; }
void fake_device(int d) { device = d; }
const char *fake_log() { return record.c_str(); }
void fake_clear_log() { record.clear(); }

// ---- registration and launches -----------------------------------------------------
void **__cudaRegisterFatBinary(void *) {
    static void *handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *fun, char *, const char *name, int, void *, void *, void *, void *,
                            int *) {
    names[fun] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t stream) {
    config = Config{grid, block, smem, stream};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream) {
    *grid = config.grid;
    *block = config.block;
    *smem = config.smem;
    *(cudaStream_t *)stream = config.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fun) {
    *k = (cudaKernel_t)fun;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t stream) {
    const void *fun = (const void *)k;
    auto lim = smem_limit.find({device, fun});
    if (smem > 48 * 1024 && (lim == smem_limit.end() || (size_t)lim->second < smem)) return fail(cudaErrorInvalidValue);
    Launch l;
    l.name = names[fun];
    // (mode, fields, ...), in fixed point (mode, limbs, info, fields, spinor limbs, ...)
    if (l.name.find("k_dslash") != std::string::npos) l.needs.push_back(*(uintptr_t *)args[1]);
    if (l.name.find("k_dslash_fx") != std::string::npos) l.needs.push_back(*(uintptr_t *)args[4]);
    auto c = capturing.find(stream);
    if (c != capturing.end()) {
        c->second->launches.push_back(l);
        log("captured " + l.name);
        return cudaSuccess;
    }
    if (l.name.find("k_dslash") != std::string::npos && l.name.find("_fx") == std::string::npos) {
        char io[64];  // (mode, fields, in, out, ...)
        snprintf(io, sizeof io, " in %llx out %llx", *(unsigned long long *)args[2], *(unsigned long long *)args[3]);
        l.name += io;
    }
    log("run " + l.name + " " + std::to_string(grid.x) + "x" + std::to_string(grid.y) + " " + std::to_string(block.x));
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *fun, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) smem_limit[{device, fun}] = v;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
    memset(a, 0, sizeof *a);
    a->maxThreadsPerBlock = 1024;
    return cudaSuccess;
}

// ---- errors, devices ----------------------------------------------------------------
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
const char *cudaGetErrorString(cudaError_t e) {
    static char text[32];
    snprintf(text, sizeof text, "error %d", (int)e);
    return text;
}
cudaError_t cudaGetDevice(int *d) {
    *d = device;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
    device = d;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) {
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return capture_forbids() ? fail(cudaErrorStreamCaptureUnsupported) : cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
    *f = nullptr;
    if (q) *q = cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *) {
    *p = (void *)fresh(1);
    return cudaSuccess;
}

// ---- memory ---------------------------------------------------------------------------
cudaError_t cudaMalloc(void **p, size_t n) {
    if (capture_forbids()) return fail(cudaErrorStreamCaptureUnsupported);
    if (refused(n)) return fail(cudaErrorMemoryAllocation);
    const uintptr_t a = fresh(n);
    live[a] = n;
    used += n;
    *p = (void *)a;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    if (!p) return cudaSuccess;
    if (capture_forbids()) return fail(cudaErrorStreamCaptureUnsupported);
    auto it = live.find((uintptr_t)p);
    if (it == live.end()) return fail(cudaErrorInvalidValue);
    used -= it->second;
    live.erase(it);
    return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) {
    const size_t u = used + pool_held();
    *f = budget > u ? budget - u : 0;
    *t = budget;
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
    *p = calloc(1, n);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) {
    free(p);
    return cudaSuccess;
}
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned) {
    *d = h;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *dst, const void *, size_t n, cudaMemcpyKind kind, cudaStream_t) {
    if (kind == cudaMemcpyDeviceToHost) memset(dst, n >= 16 ? fill : 0, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }

cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) {
    Pool *q = new Pool();
    pools.insert(q);
    *p = (cudaMemPool_t)q;
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t p) {
    pools.erase((Pool *)p);
    delete (Pool *)p;
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t p, cudaMemPoolAttr a, void *v) {
    if (a == cudaMemPoolAttrReleaseThreshold) ((Pool *)p)->keep = *(uint64_t *)v;
    return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t n) {
    Pool *q = (Pool *)p;
    const size_t to = q->used > n ? q->used : n;
    if (q->held > to) q->held = to;
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t pool, cudaStream_t s) {
    Pool *q = (Pool *)pool;
    auto c = capturing.find(s);
    if (c != capturing.end()) {  // an allocation node: nothing is taken now
        c->second->alloc_nodes = true;
        const uintptr_t a = fresh(n);
        pooled[a] = {nullptr, 0};
        *p = (void *)a;
        return cudaSuccess;
    }
    const size_t more = q->used + n > q->held ? q->used + n - q->held : 0;
    if (refused(more)) return fail(cudaErrorMemoryAllocation);
    q->used += n;
    q->held += more;
    const uintptr_t a = fresh(n);
    pooled[a] = {q, n};
    *p = (void *)a;
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t) {
    auto it = pooled.find((uintptr_t)p);
    if (it == pooled.end()) return fail(cudaErrorInvalidValue);
    if (it->second.first) it->second.first->used -= it->second.second;
    pooled.erase(it);
    return cudaSuccess;
}

// ---- streams, events ------------------------------------------------------------------
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    *s = (cudaStream_t)fresh(1);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) {
    *e = (cudaEvent_t)fresh(1);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    static int n = 0;
    *ms = 1.f / ++n;  // every candidate of a tuner is faster than the one before
    return cudaSuccess;
}

// ---- capture and graphs ------------------------------------------------------------------
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
    capturing[s] = new Graph();
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g) {
    *g = (cudaGraph_t)capturing[s];
    capturing.erase(s);
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus *st) {
    *st = capturing.count(s) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t s, cudaStreamCaptureStatus *st, unsigned long long *id,
                                     cudaGraph_t *g, const cudaGraphNode_t **, const cudaGraphEdgeData **, size_t *) {
    auto c = capturing.find(s);
    *st = c != capturing.end() ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    if (c != capturing.end()) {
        if (id) *id = (uintptr_t)c->second;
        if (g) *g = (cudaGraph_t)c->second;
    }
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *m) {
    const int old = capture_mode;
    capture_mode = *m;
    *m = (cudaStreamCaptureMode)old;
    return cudaSuccess;
}
cudaError_t cudaUserObjectCreate(cudaUserObject_t *o, void *ptr, cudaHostFn_t destroy, unsigned refs, unsigned) {
    *o = (cudaUserObject_t) new UserObject{ptr, destroy, (int)refs};
    return cudaSuccess;
}
cudaError_t cudaUserObjectRelease(cudaUserObject_t o, unsigned) {
    std::vector<UserObject *> v{(UserObject *)o};
    release(v);
    return cudaSuccess;
}
cudaError_t cudaGraphRetainUserObject(cudaGraph_t g, cudaUserObject_t o, unsigned, unsigned) {
    ((Graph *)g)->objects.push_back((UserObject *)o);  // cudaGraphUserObjectMove
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t g, unsigned long long) {
    Graph *q = (Graph *)g;
    if (q->alloc_nodes && q->execs) return fail(cudaErrorNotSupported);
    q->execs++;
    for (UserObject *o : q->objects) o->refs++;
    *e = (cudaGraphExec_t) new Exec{q->launches, q->objects, q};
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
    for (const Launch &l : ((Exec *)e)->launches) {
        bool ok = true;
        for (uintptr_t a : l.needs) ok = ok && (live.count(a) || (a == 0));
        log((ok ? "replayed " : "STALE ") + l.name);
    }
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
    release(((Graph *)g)->objects);
    ((Graph *)g)->launches.clear();
    return cudaSuccess;  // kept: an executable graph may still point to it
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
    release(((Exec *)e)->objects);
    ((Exec *)e)->from->execs--;
    delete (Exec *)e;
    return cudaSuccess;
}

}  // extern "C"
