"""The library's host code on a stand-in for the CUDA runtime (no GPU): device memory is host memory,
zero at first, and kernels do nothing, but that sums over rows of several vectors come out as one (norms,
by which the host divides).  A projected matrix stays zero, and a solve ends at its first check.

What it keeps watch on: buffers that are still allocated, allocations failed on request, launches by
kernel name, shared memory asked for beyond a kernel's limit (refused, as the runtime does), limits
lowered once set, and host memory that changes between an asynchronous copy from it and the next
synchronisation (the runtime may read it until then).
"""
import contextlib
import ctypes
import os
import subprocess

from paper_1003_4570_gb300 import build, omen

SOURCE = r"""
#include <cuda_runtime_api.h>
#include <sys/uio.h>
#include <unistd.h>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>
static std::mutex mu;
static thread_local cudaError_t last = cudaSuccess;
static std::map<void*, size_t> live;
static long fail_at = -1, changed = 0, lowered = 0;
static std::map<const void*, std::string> names;
static std::map<const void*, int> limits;
static std::map<std::string, long> launches;
struct Pending { const char* src; std::string was; };
static std::vector<Pending> pending;
struct Config { dim3 g, b; size_t s; cudaStream_t st; };
static thread_local Config config;

static cudaError_t take(void** p, size_t n) {
  std::lock_guard<std::mutex> l(mu);
  if (fail_at >= 0 && fail_at-- == 0) { *p = nullptr; return cudaErrorMemoryAllocation; }
  *p = calloc(1, n ? n : 1);
  live[*p] = n;
  return cudaSuccess;
}
static cudaError_t give(void* p) {
  std::lock_guard<std::mutex> l(mu);
  if (!p) return cudaSuccess;
  if (!live.erase(p)) return cudaErrorInvalidValue;
  free(p);
  return cudaSuccess;
}
static void reached() {
  std::lock_guard<std::mutex> l(mu);
  for (auto& c : pending) {
    std::string now(c.was.size(), 0);
    iovec to{&now[0], now.size()}, from{(void*)c.src, now.size()};
    if (process_vm_readv(getpid(), &to, 1, &from, 1, 0) != (ssize_t)now.size() || now != c.was) ++changed;
  }
  pending.clear();
}
static cudaError_t run(const void* f, size_t shared, void** args) {
  std::lock_guard<std::mutex> l(mu);
  auto it = limits.find(f);
  if (shared > (size_t)(it == limits.end() ? 48 << 10 : it->second)) return last = cudaErrorInvalidValue;
  const std::string& name = names[f];
  ++launches[name];
  if (name.find("reduce_dev_kernel") != std::string::npos) {   // (partials, chunks, na, nb, out, ...)
    double* out = *(double**)args[4];
    for (int i = 0; out && i < *(int*)args[2] * *(int*)args[3]; ++i) out[2 * i] = 1.0, out[2 * i + 1] = 0.0;
  }
  return cudaSuccess;
}
extern "C" {
long fake_live() { return (long)live.size(); }
void fake_fail(long n) { fail_at = n; }
long fake_changed() { reached(); return changed; }
long fake_lowered() { return lowered; }
void fake_reset() { launches.clear(); changed = lowered = 0; fail_at = -1; pending.clear(); }
const char* fake_launches() {
  static std::string s;
  s.clear();
  for (auto& k : launches) s += k.first + " " + std::to_string(k.second) + "\n";
  return s.c_str();
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, void*, void*, void*, void*, int*) { names[f] = name; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, cudaStream_t st) { config = {g, b, s, st}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
  *g = config.g; *b = config.b; *s = config.s; *(cudaStream_t*)st = config.st;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(void** k, const void* f) { *k = (void*)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(void* k, dim3, dim3, void** a, size_t s, cudaStream_t) { return run(k, s, a); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** a) { return run(f, c->dynamicSmemBytes, a); }
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3, dim3, void** a, size_t s, cudaStream_t) { return run(f, s, a); }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
  std::lock_guard<std::mutex> l(mu);
  if (v > 227 << 10) return last = cudaErrorInvalidValue;
  if (limits.count(f) && v < limits[f]) ++lowered;
  limits[f] = v;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { return take(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return take(p, n); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return take(p, n); }
cudaError_t cudaFree(void* p) { reached(); return give(p); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return give(p); }
cudaError_t cudaMallocHost(void** p, size_t n) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind kind, cudaStream_t) {
  memmove(d, s, n);
  if (kind == cudaMemcpyHostToDevice) {
    std::lock_guard<std::mutex> l(mu);
    pending.push_back({(const char*)s, std::string((const char*)s, n)});
  }
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t) {
  for (size_t i = 0; i < h; ++i) memcpy((char*)d + i * dp, (const char*)s + i * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { reached(); return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { reached(); return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "error"; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { *n = 2; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 2; return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { *p = (cudaMemPool_t)8; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)8; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)8; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {   // every time below the one before
  static int n = 0;
  *ms = 1.f / ++n;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)16; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = (cudaGraph_t)8; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { *e = (cudaGraphExec_t)8; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = (void*)s; return cudaSuccess; }
}
"""


class Watch:
    """What the stand-in has seen since the last reset."""

    def __init__(self, path):
        self._l = ctypes.CDLL(path)
        self._l.fake_launches.restype = ctypes.c_char_p
        for f in ("fake_live", "fake_changed", "fake_lowered"):
            getattr(self._l, f).restype = ctypes.c_long
        self._l.fake_fail.argtypes = [ctypes.c_long]
        self.reset = self._l.fake_reset
        self.fail = self._l.fake_fail         # the n-th allocation from now fails (0: the next)
        self.live = self._l.fake_live
        self.changed = self._l.fake_changed
        self.lowered = self._l.fake_lowered

    def launches(self, part):
        """Launches of the kernels whose mangled name contains `part`."""
        return sum(int(ln.rsplit(" ", 1)[1]) for ln in self._l.fake_launches().decode().splitlines() if part in ln)


def link(folder):
    """The library's objects and the stand-in as one shared library in `folder`."""
    build.build()
    src, out = os.path.join(folder, "runtime.cpp"), os.path.join(folder, "libomen_host.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    objs = [os.path.join(build.BUILD, os.path.basename(s) + ".o") for s in build.sources()]
    # -Bsymbolic: the process may hold a real CUDA runtime with the same names
    subprocess.run([build._nvcc(), "-std=c++17", "-shared", "-cudart", "none", "-Xcompiler", "-fPIC,-fopenmp", "-Xlinker", "-Bsymbolic",
                    "-o", out, src] + objs + ["-lgomp"], check=True, capture_output=True)
    return out


@contextlib.contextmanager
def loaded(folder):
    """The binding on the stand-in: yields its Watch."""
    path, lib, at = link(str(folder)), omen._lib, omen.LIB_PATH
    omen._lib, omen.LIB_PATH = None, path
    try:
        yield Watch(path)
    finally:
        omen._lib, omen.LIB_PATH = lib, at
