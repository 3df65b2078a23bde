// A stand-in for the CUDA runtime on machines without a GPU, for tests of the library's host paths:
// which kernels are launched with which arguments, what is copied, waited for, allocated and given back,
// and what a call does when the runtime refuses one.  Kernels do nothing.  Device memory is host memory;
// an address named by fake_memory is never touched.  Linked with the library's objects in the place of
// the runtime (tests/_fake_cuda.py).
#include <cuda_runtime_api.h>

#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {

struct Mem {
    size_t bytes;
    int type, device;       // cudaMemoryType
    bool real;
};
std::map<const char*, Mem> mems;
std::string logbuf;
int device = 0;
cudaError_t last = cudaSuccess;
std::string fail_name;
int fail_at = 0, fail_err = 0;
struct Config {
    dim3 g, b;
    size_t smem;
    cudaStream_t s;
} pushed;
void (*hook)(const char*, void**) = nullptr;
size_t serial = 0x1000;     // handles of streams, events, graphs, pools

void note(const char* fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    logbuf += buf;
    logbuf += '\n';
}

// by host stub; filled by the other objects' start-up code, which may run before this file's
std::map<const void*, std::string>& kernels()
{
    static std::map<const void*, std::string> k;
    return k;
}

// the error of this call of `name`, if it is the one that fails
cudaError_t err(const char* name)
{
    if (fail_at > 0 && fail_name == name && --fail_at == 0) return last = (cudaError_t)fail_err;
    return cudaSuccess;
}

const Mem* find(const void* p)
{
    auto it = mems.upper_bound(static_cast<const char*>(p));
    if (it == mems.begin()) return nullptr;
    --it;
    return static_cast<const char*>(p) < it->first + it->second.bytes ? &it->second : nullptr;
}
bool touchable(const void* p)
{
    const Mem* m = find(p);
    return !m || m->real;
}

cudaError_t alloc(const char* name, void** p, size_t n)
{
    const cudaError_t e = err(name);
    if (e != cudaSuccess) return e;
    *p = aligned_alloc(256, (n + 511) / 256 * 256);
    mems[static_cast<char*>(*p)] = Mem{n, cudaMemoryTypeDevice, device, true};
    note("%s %p %zu", name, *p, n);
    return cudaSuccess;
}
cudaError_t release(const char* name, void* p)
{
    note("%s %p", name, p);
    if (!p) return cudaSuccess;
    if (!mems.erase(static_cast<char*>(p))) return last = cudaErrorInvalidValue;
    free(p);
    return cudaSuccess;
}

cudaError_t copy(const char* name, void* d, const void* s, size_t n, int kind, cudaStream_t st)
{
    note("%s %p %p %zu %d %p", name, d, s, n, kind, (void*)st);
    const cudaError_t e = err(name);
    if (e == cudaSuccess && touchable(d) && touchable(s)) memmove(d, s, n);
    return e;
}

cudaError_t launch(const void* f, dim3 g, dim3 b, void** args, size_t smem, cudaStream_t s, int pdl)
{
    const std::string& n = kernels()[f];
    note("launch %s %u %u %u %u %zu %p %d", n.c_str(), g.x, g.y, g.z, b.x * b.y * b.z, smem, (void*)s, pdl);
    if (hook) hook(n.c_str(), args);
    return err("launch");
}

template <class T>
cudaError_t make(const char* name, T* h)
{
    const cudaError_t e = err(name);
    if (e != cudaSuccess) return e;
    *h = (T)(serial += 16);
    note("%s %p", name, (void*)*h);
    return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- the tests' side
const char* fake_log() { return logbuf.c_str(); }
void fake_clear() { logbuf.clear(); }
void fake_fail(const char* name, int nth, int e)
{
    fail_name = name;
    fail_at = nth;
    fail_err = e;
    last = cudaSuccess;
}
void fake_memory(void* p, size_t bytes, int type, int dev)
{
    if (bytes) mems[static_cast<char*>(p)] = Mem{bytes, type, dev, false};
    else mems.erase(static_cast<char*>(p));
}
void fake_device(int d) { device = d; }
void fake_hook(void (*f)(const char*, void**)) { hook = f; }
size_t fake_live()
{
    size_t n = 0;
    for (auto& m : mems) n += m.second.real;
    return n;
}

// ---- what nvcc's host code calls
void** __cudaRegisterFatBinary(void*) { return reinterpret_cast<void**>(&serial); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*)
{
    kernels()[f] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s)
{
    pushed = Config{g, b, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s)
{
    *g = pushed.g;
    *b = pushed.b;
    *smem = pushed.smem;
    *static_cast<cudaStream_t*>(s) = pushed.s;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f)
{
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** args, size_t smem, cudaStream_t s)
{
    return launch((const void*)k, g, b, args, smem, s, 0);
}

// ---- the runtime
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args)
{
    int pdl = 0;
    for (unsigned i = 0; i < c->numAttrs; ++i) pdl |= c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization;
    return launch(f, c->gridDim, c->blockDim, args, c->dynamicSmemBytes, c->stream, pdl);
}
cudaError_t cudaGetLastError()
{
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t) { return "an error of the stand-in"; }
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int d)
{
    *v = a == cudaDevAttrMultiProcessorCount ? (d == 0 ? 152 : 76) : 1;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int d)
{
    memset(p, 0, sizeof *p);
    snprintf(p->name, sizeof p->name, "stand-in %d", d);
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned)
{
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p)
{
    memset(a, 0, sizeof *a);
    const Mem* m = find(p);
    a->type = m ? (cudaMemoryType)m->type : cudaMemoryTypeUnregistered;
    a->device = m ? m->device : -2;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { return alloc("cudaMalloc", p, n); }
cudaError_t cudaFree(void* p) { return release("cudaFree", p); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return alloc("cudaMallocAsync", p, n); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return alloc("cudaMallocFromPoolAsync", p, n); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return release("cudaFreeAsync", p); }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { return make("cudaMemPoolCreate", p); }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t keep)
{
    note("cudaMemPoolTrimTo %p %zu", (void*)p, keep);
    return err("cudaMemPoolTrimTo");
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) { return copy("cudaMemcpy", d, s, n, k, nullptr); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st)
{
    return copy("cudaMemcpyAsync", d, s, n, k, st);
}
cudaError_t cudaMemset(void* d, int v, size_t n)
{
    if (touchable(d)) memset(d, v, n);
    return err("cudaMemset");
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = const_cast<void*>(s); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return make("cudaStreamCreateWithFlags", s); }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) { return make("cudaStreamCreateWithPriority", s); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { note("cudaStreamDestroy %p", (void*)s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s)
{
    note("cudaStreamSynchronize %p", (void*)s);
    return err("cudaStreamSynchronize");
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned)
{
    note("cudaStreamWaitEvent %p %p", (void*)s, (void*)e);
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { note("cudaDeviceSynchronize"); return cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int* least, int* greatest) { *least = 0; *greatest = -5; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return make("cudaEventCreate", e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return make("cudaEventCreateWithFlags", e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { note("cudaEventDestroy %p", (void*)e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { note("cudaEventRecord %p %p", (void*)e, (void*)s); return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) { note("cudaStreamBeginCapture %p", (void*)s); return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return make("cudaStreamEndCapture", g); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) { return make("cudaGraphInstantiate", x); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t) { note("cudaGraphLaunch %p", (void*)x); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { note("cudaGraphDestroy %p", (void*)g); return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { note("cudaGraphExecDestroy %p", (void*)x); return cudaSuccess; }

}  // extern "C"
