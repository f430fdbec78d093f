"""libgs.so's own host code linked against a fake CUDA runtime that runs no
kernel: it records launches, clears and shared-memory limits, holds a launch to
its kernel's limit, and refuses the launch it is told to refuse.  For what the
host side does when a launch fails and for state that belongs to a kernel, on a
machine without a GPU."""
import ctypes
import os
import subprocess

from paper_2405_19614_gb300 import _lib, build

SOURCE = r"""
#include <cuda_runtime_api.h>
#include <map>
#include <mutex>
#include <string>
static std::mutex mu;
static std::map<const void *, std::string> names;
static std::map<const void *, size_t> limits;
static std::string events;
static int count, fail_at;
static cudaError_t last;
static cudaLaunchConfig_t pushed;
static cudaError_t fail(cudaError_t e) { return last = e; }
static cudaError_t step(const char *what, const char *name, size_t smem)
{
    events += std::string(what) + " " + name + " " + std::to_string(smem) + "\n";
    return ++count == fail_at ? fail(cudaErrorInvalidValue) : cudaSuccess;
}
static cudaError_t launch(const void *f, size_t smem)
{
    std::lock_guard<std::mutex> l(mu);
    const size_t limit = limits.count(f) ? limits[f] : 48 * 1024;
    const cudaError_t e = step("launch", names[f].c_str(), smem);
    return e != cudaSuccess ? e : smem > limit ? fail(cudaErrorInvalidValue) : cudaSuccess;
}
extern "C" {
void fake_reset(int refuse) { events.clear(); count = 0; fail_at = refuse; last = cudaSuccess; }
int fake_count() { return count; }
const char *fake_events() { return events.c_str(); }
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *f, char *, const char *name, int, void *, void *, void *, void *, int *)
{
    names[f] = name;
}
cudaError_t __cudaGetKernel(void **k, const void *f) { *k = const_cast<void *>(f); return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, void *s)
{
    pushed.gridDim = g; pushed.blockDim = b; pushed.dynamicSmemBytes = smem; pushed.stream = (cudaStream_t)s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s)
{
    *g = pushed.gridDim; *b = pushed.blockDim; *smem = pushed.dynamicSmemBytes; *(cudaStream_t *)s = pushed.stream;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(void *k, dim3, dim3, void **, size_t smem, cudaStream_t) { return launch(k, smem); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **)
{
    return launch(f, c->dynamicSmemBytes);
}
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t)
{
    std::lock_guard<std::mutex> l(mu);
    return step("clear", "-", 0);
}
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return fail(cudaErrorInvalidSymbol); }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *)
{
    *p = nullptr;
    return cudaErrorNotSupported;
}
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned)
{
    *n = 4;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute, int v)
{
    std::lock_guard<std::mutex> l(mu);
    limits[f] = (size_t)v;
    events += "limit " + names[f] + " " + std::to_string(v) + "\n";
    return cudaSuccess;
}
}
"""


class FakeLib:
    """The library's entry points (call them with plain numbers as pointers:
    nothing is read through them) and what they asked of the runtime."""

    def __init__(self, folder):
        objs = [os.path.join(build.BUILD_DIR, s.replace(".cu", ".o")) for s in build.SOURCES]
        build.build(force=not all(os.path.exists(o) for o in objs))
        src, so = os.path.join(folder, "fake.cpp"), os.path.join(folder, "libgs_fake.so")
        with open(src, "w") as f:
            f.write(SOURCE)
        subprocess.check_call([build.nvcc(), "-shared", "-cudart", "none", "-Xcompiler", "-fPIC", "-std=c++17",
                               "-Xcompiler", "-fvisibility=default", "-Xlinker", "-Bsymbolic", "-o", so, src, *objs])
        self.lib = ctypes.CDLL(so)
        for name, (args, res) in _lib.SIGNATURES.items():
            f = getattr(self.lib, name)
            f.argtypes, f.restype = args, res
        self.lib.fake_events.restype = ctypes.c_char_p

    def run(self, call, refuse=0):
        """(status of call(entry points), launches and clears asked for, events);
        the refuse-th launch or clear is refused."""
        self.lib.fake_reset(refuse)
        status = call(self.lib)
        events = [tuple(e.split()) for e in self.lib.fake_events().decode().splitlines()]
        return status, self.lib.fake_count(), events
