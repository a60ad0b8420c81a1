"""The library's host code on a stand-in for the CUDA runtime, for tests of what
it plans, allocates, captures and launches where no GPU is needed (or where a
GPU could not be asked to fail).  The objects of the built library are linked
against the calls below instead of the CUDA runtime: device memory is zeroed
host memory, copies copy, kernels are only written down (name, grid, whether a
graph was being captured), events and streams are tokens, and each time taken is
shorter than the last (a tuner keeps its last candidate).  Allocations from a
given size on can be made to fail.  A graph launched after a piece of memory that
existed at its capture was freed counts as stale.
"""
import ctypes as C
import glob
import importlib.util
import os
import shutil
import subprocess

SRC = r"""
#include <cuda_runtime.h>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

namespace {
std::recursive_mutex mu;
typedef std::lock_guard<std::recursive_mutex> Lock;
struct Launch { std::string name; unsigned grid; bool captured; };
struct Graph { std::vector<Launch> nodes; int64_t born; };
struct Block { size_t bytes; int64_t born; };
std::map<const void *, std::string> &names() { static auto *m = new std::map<const void *, std::string>; return *m; }
std::map<void *, Block> &blocks() { static auto *m = new std::map<void *, Block>; return *m; }
std::vector<Launch> &launches() { static auto *v = new std::vector<Launch>; return *v; }
Graph *capture = nullptr;
int64_t tick = 0, last_freed_born = 0, stale = 0, graphs = 0, captures = 0, syncing = 0;
std::vector<std::pair<int64_t, int64_t>> &freed() { static auto *v = new std::vector<std::pair<int64_t, int64_t>>; return *v; }
size_t fail_from = SIZE_MAX, live = 0, peak = 0;
cudaError_t last = cudaSuccess;
cudaError_t err(cudaError_t e) { if (e != cudaSuccess) last = e; return e; }
struct Conf { dim3 g, b; size_t s; void *st; };
thread_local std::vector<Conf> conf;

cudaError_t alloc(void **p, size_t n)
{
    Lock l(mu);
    *p = nullptr;
    if (n >= fail_from) return err(cudaErrorMemoryAllocation);
    void *q = std::calloc(1, n ? n : 1);
    if (!q) return err(cudaErrorMemoryAllocation);
    blocks()[q] = Block{n, ++tick};
    live += n;
    if (live > peak) peak = live;
    *p = q;
    return cudaSuccess;
}
cudaError_t release(void *p)
{
    Lock l(mu);
    if (!p) return cudaSuccess;
    auto it = blocks().find(p);
    if (it == blocks().end()) return err(cudaErrorInvalidValue);
    live -= it->second.bytes;
    freed().emplace_back(it->second.born, ++tick);
    blocks().erase(it);
    std::free(p);
    return cudaSuccess;
}
cudaError_t run(const void *f, unsigned grid)
{
    Lock l(mu);
    auto it = names().find(f);
    Launch k{it == names().end() ? "?" : it->second, grid, capture != nullptr};
    if (capture) capture->nodes.push_back(k);
    launches().push_back(k);
    return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- what the tests read and set
void host_fail_from(size_t n) { Lock l(mu); fail_from = n; }
void host_clear() { Lock l(mu); launches().clear(); graphs = captures = stale = syncing = 0; peak = live; }
int64_t host_launches() { Lock l(mu); return (int64_t)launches().size(); }
const char *host_name(int64_t i) { Lock l(mu); return launches()[i].name.c_str(); }
int64_t host_grid(int64_t i) { Lock l(mu); return launches()[i].grid; }
int64_t host_graphs() { return graphs; }
int64_t host_captures() { return captures; }
int64_t host_stale() { return stale; }
int64_t host_syncing() { return syncing; }   // cudaMalloc and cudaFree calls
size_t host_live() { return live; }
size_t host_peak() { return peak; }

// ---- the runtime
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *)
{ Lock l(mu); names()[host] = name; }
static std::map<const void *, size_t> &vars() { static auto *m = new std::map<const void *, size_t>; return *m; }
void __cudaRegisterVar(void **, char *host, char *, const char *, int, size_t n, int, int) { vars()[host] = n; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, cudaStream_t st) { conf.push_back({g, b, s, st}); return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *s, void *st)
{ Conf c = conf.back(); conf.pop_back(); *g = c.g; *b = c.b; *s = c.s; *(void **)st = c.st; return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3, void **, size_t, cudaStream_t) { return run((const void *)k, g.x); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) { return run(f, c->gridDim.x); }
cudaError_t cudaMalloc(void **p, size_t n) { ++syncing; return alloc(p, n); }
cudaError_t cudaFree(void *p) { if (p) ++syncing; return release(p); }
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return alloc(p, n); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return release(p); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void *d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *v)
{ static std::map<const void *, void *> at; void *&q = at[v]; if (!q) q = std::calloc(1, vars()[v]); *p = q; return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) { *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0; return cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int *a, int *b) { *a = 0; *b = -5; return cudaSuccess; }
cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **p, unsigned, unsigned long long, cudaDriverEntryPointQueryResult *)
{ *p = nullptr; return cudaErrorInvalidValue; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) { std::memset(a, 0, sizeof *a); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) { *n = 3; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *) { *n = 4; return cudaSuccess; }
static void *token() { return std::calloc(1, 16); }
cudaError_t cudaStreamCreate(cudaStream_t *s) { *s = (cudaStream_t)token(); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return cudaStreamCreate(s); }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned, int) { return cudaStreamCreate(s); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { std::free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) { *s = cudaStreamCaptureStatusNone; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)token(); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { static int n; *ms = 1.f / (1.f + 0.01f * ++n); return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode)
{ Lock l(mu); capture = new Graph{{}, ++tick}; ++captures; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { Lock l(mu); *g = (cudaGraph_t)capture; capture = nullptr; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t g, unsigned long long) { *e = (cudaGraphExec_t) new Graph(*(Graph *)g); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete (Graph *)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { delete (Graph *)e; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t)
{
    Lock l(mu);
    Graph *g = (Graph *)e;
    ++graphs;
    for (auto &f : freed())
        if (f.first < g->born && f.second > g->born) { ++stale; break; }
    for (auto &k : g->nodes) launches().push_back(Launch{k.name, k.grid, false});
    return cudaSuccess;
}
}
"""


class Host:
    """The binding over the stand-in (``nbsym``) and what the stand-in saw."""

    def __init__(self, folder):
        from paper_1003_3896_gb300 import build
        build.build()
        pkg = os.path.dirname(build.__file__)
        folder = str(folder)
        src = os.path.join(folder, "hostcuda.cpp")
        with open(src, "w") as f:
            f.write(SRC)
        inc = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
        lib = os.path.join(folder, "libnbsym.so")
        objs = sorted(glob.glob(os.path.join(pkg, "_build", "*.o")))
        subprocess.run([shutil.which("g++"), "-O1", "-std=c++17", "-shared", "-fPIC", "-I", inc, src,
                        *objs, "-Wl,-Bsymbolic", "-Wl,--no-undefined", "-lpthread", "-o", lib],
                       check=True)
        shutil.copy(os.path.join(pkg, "nbsym.py"), folder)
        spec = importlib.util.spec_from_file_location("nbsym_host", os.path.join(folder, "nbsym.py"))
        self.nbsym = importlib.util.module_from_spec(spec)
        import sys
        sys.modules["nbsym_host"] = self.nbsym   # dataclasses look their module up
        spec.loader.exec_module(self.nbsym)
        self.lib = C.CDLL(lib)
        for name in ("launches", "graphs", "captures", "stale", "syncing", "live", "peak"):
            getattr(self.lib, "host_" + name).restype = C.c_int64
        self.lib.host_name.restype = C.c_char_p
        self.lib.host_name.argtypes = self.lib.host_grid.argtypes = [C.c_int64]
        self.lib.host_grid.restype = C.c_int64
        self.lib.host_fail_from.argtypes = [C.c_size_t]

    def fail_from(self, nbytes=None):
        """Allocations of at least nbytes fail (None: all succeed)."""
        self.lib.host_fail_from(2 ** 64 - 1 if nbytes is None else int(nbytes))

    def clear(self):
        self.lib.host_clear()

    def __getattr__(self, name):
        if name in ("graphs", "captures", "stale", "syncing", "live", "peak"):
            return int(getattr(self.lib, "host_" + name)())
        raise AttributeError(name)

    def launches(self):
        """[(demangled-enough kernel name, grid)] since the last clear()."""
        n = int(self.lib.host_launches())
        return [(self.lib.host_name(i).decode(), int(self.lib.host_grid(i))) for i in range(n)]

    def ran(self, what):
        return [k for k in self.launches() if what in k[0]]
