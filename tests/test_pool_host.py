"""The library's memory pool (csrc/pool.cu) against a fake of the CUDA runtime and of the driver's
context functions, on the CPU: which context and pool an allocation uses, and that the caller's
own context and device stay current.  (A second context is not made on a GPU here.)"""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2502_12878_gb300", "csrc")

FAKE = r"""
#pragma once
#include <stddef.h>
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaErrorMemoryAllocation = 2 };
typedef struct stream_* cudaStream_t;
typedef struct pool_* cudaMemPool_t;
#define cudaStreamPerThread ((cudaStream_t)2)
enum { cudaMemAllocationTypePinned = 1, cudaMemHandleTypeNone = 0, cudaMemLocationTypeDevice = 1,
       cudaMemPoolAttrReleaseThreshold = 4, cudaEnableDefault = 0 };
enum cudaDriverEntryPointQueryResult { cudaDriverEntryPointSuccess = 0 };
struct cudaMemPoolProps { int allocType, handleTypes; struct { int type, id; } location; };
struct cudaPointerAttributes { int device; };
cudaError_t cudaGetDevice(int*);
cudaError_t cudaSetDevice(int);
cudaError_t cudaDeviceSynchronize();
cudaError_t cudaGetLastError();
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes*, const void*);
cudaError_t cudaMemPoolCreate(cudaMemPool_t*, const cudaMemPoolProps*);
cudaError_t cudaMemPoolDestroy(cudaMemPool_t);
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, int, void*);
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t);
cudaError_t cudaMallocAsync(void**, size_t, cudaStream_t);
cudaError_t cudaMallocFromPoolAsync(void**, size_t, cudaMemPool_t, cudaStream_t);
cudaError_t cudaFreeAsync(void*, cudaStream_t);
cudaError_t cudaStreamSynchronize(cudaStream_t);
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void**, unsigned, int,
                                             cudaDriverEntryPointQueryResult*);
"""

# contexts: 100 * device + generation is a device's primary one, 7777 the caller's own
DRIVER = r"""
#include <stdio.h>
#include <string.h>
#include <string>
#include "pool.cuh"
static std::string trace;
static int dev = 0, cur = 0, gen = 1, pools = 0, fail = 0;
static bool inited = false;
static bool up[2] = {false, false};
static void log(const char* f, long a = -1) {
    char b[64];
    snprintf(b, sizeof b, a < 0 ? "%s " : "%s%ld ", f, a);
    trace += b;
}
static int primary(int d) { return 100 * d + gen; }
#define OK cudaSuccess
cudaError_t cudaGetDevice(int* d) { *d = dev; return OK; }
cudaError_t cudaSetDevice(int d) {
    log("set", d);
    inited = up[d] = true; dev = d; cur = primary(d);
    return OK;
}
cudaError_t cudaDeviceSynchronize() { log("devsync", dev); return OK; }
cudaError_t cudaGetLastError() { return OK; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    a->device = (int)((size_t)p / 1000);
    return OK;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps* q) {
    *p = (cudaMemPool_t)(size_t)++pools;
    log("create", q->location.id);
    return OK;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return OK; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, int, void*) { return OK; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t) { log("trim", (long)(size_t)p); return OK; }
cudaError_t cudaMallocAsync(void** p, size_t, cudaStream_t) { log("default"); *p = 0; return OK; }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t, cudaMemPool_t q, cudaStream_t) {
    log("pool", (long)(size_t)q);
    *p = 0;
    return fail-- > 0 ? cudaErrorMemoryAllocation : OK;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { log("free", (long)(size_t)p); return OK; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { log("sync", dev); return OK; }
static int ctx_id(void* c, unsigned long long* id) {
    *id = c ? (size_t)c : cur;
    return *id ? 0 : 201;
}
static int ctx_current(void** c) { *c = (void*)(size_t)cur; return inited ? 0 : 3; }
static int device_get(int* d, int n) { *d = n; return 0; }
static int state(int d, unsigned* f, int* a) { *f = 0; *a = up[d]; return 0; }
static int retain(void** c, int d) { *c = (void*)(size_t)primary(d); return 0; }
static int release(int) { return 0; }
cudaError_t cudaGetDriverEntryPointByVersion(const char* n, void** p, unsigned, int,
                                             cudaDriverEntryPointQueryResult* r) {
    *r = cudaDriverEntryPointSuccess;
    std::string s = n;
    *p = s == "cuCtxGetId" ? (void*)ctx_id : s == "cuCtxGetCurrent" ? (void*)ctx_current
       : s == "cuDeviceGet" ? (void*)device_get
       : s == "cuDevicePrimaryCtxGetState" ? (void*)state
       : s == "cuDevicePrimaryCtxRetain" ? (void*)retain
       : s == "cuDevicePrimaryCtxRelease" ? (void*)release : nullptr;
    return *p ? OK : cudaErrorInvalidValue;
}
static void alloc(const char* what) {
    void* p;
    const cudaError_t e = rbffd::pool_alloc(&p, 1000, 0);
    printf("%s: %s-> %d, device %d, context %d\n", what, trace.c_str(), (int)e, dev, cur);
    trace.clear();
}
int main() {
    alloc("no context");
    alloc("again");
    cur = 7777;
    alloc("own context");
    cur = primary(0);
    alloc("back");
    dev = 1; cur = 7777;                       // device 1's primary context is not there
    alloc("own context on 1");
    cur = 0;
    alloc("no context on 1");
    dev = 0; cur = 0;
    alloc("other thread");
    gen = 2; cur = primary(0);                 // after a reset
    alloc("reset");
    fail = 1;
    alloc("full once");
    fail = 2;
    alloc("full");
    return 0;
}
"""


def _run(tmp_path, driver):
    (tmp_path / "cuda_runtime_api.h").write_text(FAKE)
    (tmp_path / "driver.cpp").write_text(driver)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-I", str(tmp_path), "-I", CSRC, "-x", "c++",
                    os.path.join(CSRC, "pool.cu"), str(tmp_path / "driver.cpp"), "-o", exe],
                   check=True)
    return subprocess.run([exe], check=True, capture_output=True,
                          text=True).stdout.strip().split("\n")


def test_contexts_and_pools(tmp_path):
    assert _run(tmp_path, DRIVER) == [
        "no context: set0 create0 pool1 -> 0, device 0, context 1",
        "again: pool1 -> 0, device 0, context 1",
        "own context: default -> 0, device 0, context 7777",
        "back: pool1 -> 0, device 0, context 1",
        "own context on 1: default -> 0, device 1, context 7777",
        "no context on 1: set1 create1 pool2 -> 0, device 1, context 101",
        "other thread: set0 pool1 -> 0, device 0, context 1",
        "reset: create0 pool3 -> 0, device 0, context 2",
        "full once: pool3 sync0 trim3 pool3 -> 0, device 0, context 2",
        "full: pool3 sync0 trim3 pool3 -> 2, device 0, context 2",
    ]


FREES = r"""
int main() {
    void* a[3] = {0, (void*)(size_t)40, (void*)(size_t)50};       // of device 0
    void* b[2] = {(void*)(size_t)1040, 0};                        // of device 1
    cudaSetDevice(0);
    trace.clear();
    rbffd::pool_free(a, 3);
    printf("%s| device %d\n", trace.c_str(), dev);
    trace.clear();
    rbffd::pool_free(b, 2);
    printf("%s| device %d\n", trace.c_str(), dev);
    trace.clear();
    rbffd::pool_free(b + 1, 1);
    printf("%s| device %d\n", trace.c_str(), dev);
    return 0;
}
"""


def test_frees_wait_for_the_arrays_own_device(tmp_path):
    """... and give the memory back at once; the current device stays."""
    assert _run(tmp_path, DRIVER.split("int main()")[0] + FREES) == [
        "devsync0 free40 free50 sync0 | device 0",
        "set1 devsync1 free1040 sync1 set0 | device 0",
        "| device 0",
    ]
