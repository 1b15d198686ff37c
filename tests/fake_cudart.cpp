// A CUDA runtime for host-side tests, preloaded under libsdd.so: no GPU, no kernel runs.  Asynchronous copies
// and fills are queued and carried out as late as the host's waits allow; until then their pinned sources are
// write-protected, and a write of the host to one is counted (fake_races).  Launches are recorded (fake_launches).
// FAKE_CLUSTER limits the thread-block clusters that the device takes (0 or unset: any).
#include <cuda_runtime_api.h>

#include <signal.h>
#include <sys/mman.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
struct Op {
    void* dst;
    const void* src;   // null: a fill
    size_t n;
    int value;
};
struct Event { cudaStream_t stream = nullptr; size_t upto = 0; };
struct Stream { std::vector<Op> ops; size_t done = 0; };
std::map<cudaStream_t, Stream> streams;
std::map<const char*, size_t> device, pinned;
std::map<const void*, std::string> names;
std::string launched;
int races = 0, handles = 0;

bool within(const std::map<const char*, size_t>& m, const void* p)
{
    auto it = m.upper_bound((const char*)p);
    return it != m.begin() && (--it, (const char*)p < it->first + it->second);
}
void protect(const void* p, size_t n, bool on)
{
    if (!within(pinned, p)) return;
    const size_t a = (size_t)p / 4096 * 4096, e = ((size_t)p + n + 4095) / 4096 * 4096;
    mprotect((void*)a, e - a, on ? PROT_READ : PROT_READ | PROT_WRITE);
}
void on_write(int, siginfo_t* i, void*)
{
    const char* at = (const char*)i->si_addr;
    if (!within(pinned, at)) abort();
    for (auto& s : streams)
        for (size_t k = s.second.done; k < s.second.ops.size(); ++k) {
            const Op& o = s.second.ops[k];
            if (o.src && at >= (const char*)o.src && at < (const char*)o.src + o.n) ++races;
        }
    protect(at, 1, false);
}
void drain(cudaStream_t s, size_t upto)
{
    Stream& q = streams[s];
    for (; q.done < upto; ++q.done) {
        Op& o = q.ops[q.done];
        if (!o.src) memset(o.dst, o.value, o.n);
        else {
            protect(o.dst, o.n, false);
            memcpy(o.dst, o.src, o.n);
            protect(o.src, o.n, false);
        }
    }
}
void drain(cudaStream_t s) { drain(s, streams[s].ops.size()); }
void* fresh(std::map<const char*, size_t>& m, size_t n)
{
    void* p = calloc(1, n + 256);
    m[(const char*)p] = n;
    return p;
}
void record(const void* fn, dim3 g, dim3 b, size_t smem, unsigned cluster)
{
    launched += names[fn] + " " + std::to_string(g.x) + " " + std::to_string(b.x) + " " + std::to_string(smem) + " " +
                std::to_string(cluster) + "\n";
}
struct { dim3 g, b; size_t smem; cudaStream_t s; } pending;
}  // namespace

extern "C" {
int fake_races() { return races; }
const char* fake_launches() { return launched.c_str(); }

void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* fn, char*, const char* name, int, void*, void*, void*, void*, int*)
{
    names[fn] = name;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fn) { *k = (cudaKernel_t)fn; return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s)
{
    pending = {g, b, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s)
{
    *g = pending.g; *b = pending.b; *smem = pending.smem; *(cudaStream_t*)s = pending.s;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t smem, cudaStream_t)
{
    record((const void*)k, g, b, smem, 1);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void**)
{
    unsigned cluster = 1;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[i].val.clusterDim.x;
    record(fn, c->gridDim, c->blockDim, c->dynamicSmemBytes, cluster);
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* c)
{
    const char* e = getenv("FAKE_CLUSTER");
    unsigned most = e ? (unsigned)atoi(e) : 0, cluster = 1;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[i].val.clusterDim.x;
    *n = most && cluster > most ? 0 : 8;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { *n = 4; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) { memset(a, 0, sizeof *a); return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }

cudaError_t cudaMalloc(void** p, size_t n) { *p = fresh(device, n); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned)
{
    struct sigaction a = {};
    a.sa_sigaction = on_write;
    a.sa_flags = SA_SIGINFO;
    sigaction(SIGSEGV, &a, nullptr);
    *p = mmap(nullptr, n, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    pinned[(const char*)*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) { device.erase((const char*)p); free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p)
{
    munmap(p, pinned[(const char*)p]);
    pinned.erase((const char*)p);
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p)
{
    memset(a, 0, sizeof *a);
    a->type = within(device, p) ? cudaMemoryTypeDevice : within(pinned, p) ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind, cudaStream_t s)
{
    if (!within(device, src) && !within(pinned, src)) drain(s);  // pageable source: taken at once
    streams[s].ops.push_back(Op{dst, src, n, 0});
    protect(src, n, true);
    if ((!within(device, src) && !within(pinned, src)) || (!within(device, dst) && !within(pinned, dst))) drain(s);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* dst, const void* src, size_t n, cudaMemcpyKind)
{
    memcpy(dst, src, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* dst, int v, size_t n, cudaStream_t s)
{
    streams[s].ops.push_back(Op{dst, nullptr, n, v});
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)(size_t)(++handles); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { drain(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { drain(s); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t) new Event; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete (Event*)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    *(Event*)e = Event{s, streams[s].ops.size()};
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) { drain(((Event*)e)->stream, ((Event*)e)->upto); return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t e) { return cudaEventSynchronize(e); }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
}
