"""A build of the library whose calls to a few CUDA runtime functions can be made to fail or wait, on the host.

The sources are compiled as they are, with a header in front that renames those functions.  An allocation
fails by asking the runtime for more than any address space holds, so that it leaves the runtime's error as a real one
does; no memory runs out and nothing faults on the GPU.  Tests set the plan's fields
through Faults; at rest every call passes through."""
import contextlib
import ctypes
import os
import subprocess
from concurrent.futures import ThreadPoolExecutor

HEADER = r"""
#pragma once
#include <cuda_runtime.h>
#include <cub/cub.cuh>
#include <chrono>
#include <cstring>
#include <thread>
struct GpopFaults {
    long long fail_alloc;   // the allocation that fails (0: the next one; -1: none), and its repetitions at once
    long long allocs;       // allocations so far
    int until_trim;         // ... but not once a memory pool has been trimmed
    int failing;            // an allocation of last_bytes has failed, and none has succeeded since
    unsigned long long last_bytes;
    int launch_error;       // what a cooperative launch returns (0: it is made)
    int memset_delay_ms;    // the legacy stream waits this long before a cudaMemset
    int copy_delay_ms;      // ... before a cudaMemcpy to the device, which returns once it has taken its source
};
extern "C" __attribute__((visibility("default"))) GpopFaults gpop_faults;
inline bool gpop_fails(size_t n) {
    GpopFaults &f = gpop_faults;
    if (f.failing && f.last_bytes == n) return true;
    f.failing = 0;
    if (f.fail_alloc < 0 || f.allocs++ != f.fail_alloc) return false;
    f.failing = 1;
    f.last_bytes = n;
    return true;
}
inline cudaError_t gpop_no_memory() {
    void *p = nullptr;
    return cudaMalloc(&p, (size_t)1 << 60);
}
template <typename T> inline cudaError_t gpop_malloc(T **p, size_t n) {
    return gpop_fails(n) ? gpop_no_memory() : cudaMalloc((void **)p, n);
}
template <typename T> inline cudaError_t gpop_malloc_pool(T **p, size_t n, cudaMemPool_t pool, cudaStream_t s) {
    return gpop_fails(n) ? gpop_no_memory() : cudaMallocFromPoolAsync((void **)p, n, pool, s);
}
inline cudaError_t gpop_trim(cudaMemPool_t pool, size_t keep) {
    if (gpop_faults.until_trim) gpop_faults.failing = 0;
    return cudaMemPoolTrimTo(pool, keep);
}
inline cudaError_t gpop_coop(const void *f, dim3 g, dim3 b, void **a, size_t m, cudaStream_t s) {
    return gpop_faults.launch_error ? (cudaError_t)gpop_faults.launch_error : cudaLaunchCooperativeKernel(f, g, b, a, m, s);
}
inline void gpop_sleep(void *ms) { std::this_thread::sleep_for(std::chrono::milliseconds((size_t)ms)); }
inline cudaError_t gpop_memset(void *p, int v, size_t n) {
    if (gpop_faults.memset_delay_ms) cudaLaunchHostFunc(0, gpop_sleep, (void *)(size_t)gpop_faults.memset_delay_ms);
    return cudaMemset(p, v, n);
}
inline cudaError_t gpop_memcpy(void *d, const void *s, size_t n, cudaMemcpyKind kind) {
    if (!gpop_faults.copy_delay_ms || kind != cudaMemcpyHostToDevice) return cudaMemcpy(d, s, n, kind);
    void *staged = nullptr;  // stays with the process, which ends soon after
    cudaError_t e = cudaMallocHost(&staged, n);
    if (e != cudaSuccess) return e;
    memcpy(staged, s, n);
    cudaLaunchHostFunc(0, gpop_sleep, (void *)(size_t)gpop_faults.copy_delay_ms);
    return cudaMemcpyAsync(d, staged, n, kind, 0);
}
#define cudaMalloc gpop_malloc
#define cudaMallocFromPoolAsync gpop_malloc_pool
#define cudaMemPoolTrimTo gpop_trim
#define cudaLaunchCooperativeKernel gpop_coop
#define cudaMemset gpop_memset
#define cudaMemcpy gpop_memcpy
"""

COOPERATIVE_LAUNCH_TOO_LARGE = 720  # cudaErrorCooperativeLaunchTooLarge


class Faults(ctypes.Structure):
    _fields_ = [("fail_alloc", ctypes.c_longlong), ("allocs", ctypes.c_longlong), ("until_trim", ctypes.c_int),
                ("failing", ctypes.c_int), ("last_bytes", ctypes.c_ulonglong), ("launch_error", ctypes.c_int),
                ("memset_delay_ms", ctypes.c_int), ("copy_delay_ms", ctypes.c_int)]

    @contextlib.contextmanager
    def plan(self, **kw):
        """The fields of kw for the calls within; at rest again afterwards."""
        self.rest()
        for k, v in kw.items():
            setattr(self, k, v)
        try:
            yield self
        finally:
            self.rest()

    def rest(self):
        self.fail_alloc, self.allocs, self.until_trim, self.failing = -1, 0, 0, 0
        self.last_bytes = self.launch_error = self.memset_delay_ms = self.copy_delay_ms = 0


def build(out_dir):
    """Compiles the variant into out_dir; returns its path."""
    from paper_1806_08092_gb300 import _build as b
    head, plan = os.path.join(out_dir, "faults.h"), os.path.join(out_dir, "faults.cu")
    with open(head, "w") as f:
        f.write(HEADER)
    with open(plan, "w") as f:
        f.write('extern "C" { GpopFaults gpop_faults = {-1, 0, 0, 0, 0, 0, 0, 0}; }\n')
    sources = [os.path.join(b.CSRC, s) for s in b.SOURCES] + [plan]

    def compile_one(src):
        obj = os.path.join(out_dir, os.path.basename(src).replace(".cu", ".o"))
        subprocess.run([b.nvcc(), *b.ARCH, *b.FLAGS, "-include", head, "-c", src, "-o", obj], check=True, capture_output=True)
        return obj

    with ThreadPoolExecutor(len(sources)) as ex:
        objs = list(ex.map(compile_one, sources))
    lib = os.path.join(out_dir, "libgpop_faults.so")
    subprocess.run([b.nvcc(), *b.ARCH, "-shared", "-o", lib, *objs], check=True, capture_output=True)
    return lib


@contextlib.contextmanager
def use(lib):
    """The package on the variant; yields its Faults.  Graphs made within are closed within."""
    from paper_1806_08092_gb300 import _lib
    before, _lib._lib = _lib._lib, None
    try:
        yield Faults.in_dll(_lib.load(lib), "gpop_faults")
    finally:
        _lib._lib = before
