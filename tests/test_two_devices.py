"""Radix sorts and packing orders of a process that uses two devices, on a stand-in for the CUDA runtime.

A kernel's attributes (dynamic shared memory above 48 KB, clusters of more than 8 CTAs) belong to the
device that was current when they were set.  The host side of radix_sort.cu is linked with a runtime that
keeps them so and refuses what has not been set; no GPU is used.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))),
                    "include")

pytestmark = pytest.mark.skipif(not os.path.exists(os.path.join(CUDA, "cuda_runtime_api.h")) or shutil.which("g++") is None,
                                reason="CUDA toolkit or g++ not available")

FAKE = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include <utility>
#include <cuda_runtime_api.h>
#include "rtree.h"

static int g_dev = 0, g_most[2], g_bad = 0, g_clusters = 0, g_plain = 0;
static cudaError_t g_last = cudaSuccess;
static std::map<std::pair<int, const void *>, std::map<int, int>> g_attr;  // device, kernel: attributes

static cudaError_t check(const void *f, size_t smem, int cluster)
{
    std::map<int, int> &a = g_attr[{g_dev, f}];
    const bool ok = (smem <= 48 * 1024 || a[cudaFuncAttributeMaxDynamicSharedMemorySize] >= (int)smem) &&
                    (cluster <= 8 || a[cudaFuncAttributeNonPortableClusterSizeAllowed]) && cluster <= g_most[g_dev];
    return ok ? cudaSuccess : cudaErrorInvalidValue;
}
static cudaError_t launch(const void *f, size_t smem, int cluster)
{
    (cluster ? g_clusters : g_plain)++;
    const cudaError_t e = check(f, smem, cluster);
    if (e != cudaSuccess) {
        g_last = e;
        ++g_bad;
    }
    return e;
}
static int cluster_of(const cudaLaunchConfig_t *c)
{
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension)
            return (int)c->attrs[i].val.clusterDim.x;
    return 0;
}

extern "C" {
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
static size_t g_smem;
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t smem, void *) { g_smem = smem; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *smem, void *) { *smem = g_smem; return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t smem, cudaStream_t) { return launch((const void *)k, smem, 0); }
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3, void **, size_t smem, cudaStream_t) { return launch(f, smem, 0); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) { return launch(f, c->dynamicSmemBytes, cluster_of(c)); }
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) { g_attr[{g_dev, f}][a] = v; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int, size_t smem, unsigned)
{
    *n = check(f, smem, 0) == cudaSuccess ? 4 : 0;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *c)
{
    *n = check(f, c->dynamicSmemBytes, cluster_of(c)) == cudaSuccess ? 4 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t) { return "refused"; }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
}

namespace rt {
enum Block { EXACT, SCRATCH, RESULT };
struct KernelTimer {
    KernelTimer(const char *, cudaStream_t);
    ~KernelTimer();
};
KernelTimer::KernelTimer(const char *, cudaStream_t) {}
KernelTimer::~KernelTimer() {}
rtree_status fail(rtree_status st, const char *, ...) { return st; }
rtree_status dmalloc(void **p, size_t, cudaStream_t, const char *, Block) { *p = (void *)0x1000; return RTREE_OK; }
void dfree(void *, cudaStream_t) {}
int sm_count() { return 152; }
rtree_status radix_sort_pairs(const uint32_t *, const uint32_t *, uint32_t *, uint32_t *, int64_t, int, int, cudaStream_t);
rtree_status str_order(const float4 *, int64_t, int64_t, uint32_t *, cudaStream_t);
}

int main(int, char **v)
{
    g_most[0] = atoi(v[1]);
    g_most[1] = atoi(v[2]);
    uint32_t *p = (uint32_t *)0x1000;
    for (int step = 0; step < 3; ++step) {
        g_dev = step & 1;
        g_clusters = g_plain = 0;
        int err = 0;
        for (int64_t n : {(int64_t)3000, (int64_t)1 << 20})
            for (int bits : {8, 9, 18, 32})
                err |= rt::radix_sort_pairs(p, p, p, p, n, 0, bits, nullptr);
        for (int64_t n : {(int64_t)3000, (int64_t)1 << 20})
            err |= rt::str_order((const float4 *)p, n, 256, p, nullptr);
        // the small sorts are clusters where the device has them
        if (err || g_bad || (g_clusters > 0) != (g_most[g_dev] > 0) || g_plain == 0) {
            printf("device %d (clusters of %d): status %d, %d launches refused, %d clusters, %d plain\n", g_dev,
                   g_most[g_dev], err, g_bad, g_clusters, g_plain);
            return 1;
        }
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    from paper_2309_16913_gb300 import build as b
    d = tmp_path_factory.mktemp("devices")
    obj = d / "radix_sort.o"
    subprocess.run([b.nvcc(), *b.NVCC_FLAGS, "-c", os.path.join(b.CSRC, "radix_sort.cu"), "-o", str(obj)], check=True)
    (d / "fake.cpp").write_text(FAKE)
    subprocess.run(["g++", "-std=c++17", "-I", CUDA, "-I", b.INCLUDE, str(d / "fake.cpp"), str(obj), "-o", str(d / "run"),
                    "-lpthread"], check=True)
    return str(d / "run")


@pytest.mark.parametrize("first,second", [(16, 16), (16, 8), (8, 16), (16, 0), (0, 16)])
def test_each_device_gets_its_attributes(exe, first, second):
    r = subprocess.run([exe, str(first), str(second)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
