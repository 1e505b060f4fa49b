"""The cluster launches of the doubling's start on several devices: seed.cu linked with
a fake CUDA runtime that keeps function attributes by device and checks every
launch against them, as the real one does (no GPU needed)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_30379_gb300", "csrc")

FAKE = r"""
#include <cuda_runtime.h>
#include <stddef.h>
#include <map>
static int dev, max_clusters[4];
static std::map<int, int> attrs_[4][2];  // by device and kernel: attribute -> value
static const void *kernels[2];
static std::map<int, int> &attr_of(const void *f)
{
    const int k = kernels[0] == nullptr || kernels[0] == f ? 0 : 1;
    kernels[k] = f;
    return attrs_[dev][k];
}
unsigned last_grid, last_cluster;
size_t last_smem;
extern "C" {
void fake_device(int d, int clusters) { dev = d; max_clusters[d] = clusters; }
cudaError_t cudaGetDevice(int *d) { *d = dev; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v)
{
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize && v > 227 * 1024) return cudaErrorInvalidValue;
    attr_of(f)[a] = v;
    return cudaSuccess;
}
static cudaError_t check(const cudaLaunchConfig_t *c, const void *f)
{
    std::map<int, int> &attr = attr_of(f);
    unsigned cl = 1;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cl = c->attrs[i].val.clusterDim.x;
    const size_t room = attr.count(cudaFuncAttributeMaxDynamicSharedMemorySize)
                            ? attr[cudaFuncAttributeMaxDynamicSharedMemorySize] : 48 * 1024;
    if (cl > 8 && !attr[cudaFuncAttributeNonPortableClusterSizeAllowed]) return cudaErrorInvalidClusterSize;
    if (c->dynamicSmemBytes > room || c->gridDim.x % cl) return cudaErrorInvalidValue;
    last_grid = c->gridDim.x, last_cluster = cl, last_smem = c->dynamicSmemBytes;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *c)
{
    const cudaError_t e = check(c, f);
    *n = e == cudaSuccess ? max_clusters[dev] : 0;
    return e;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) { return check(c, f); }
cudaError_t cudaLaunchKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t) { return cudaErrorUnknown; }
cudaError_t __cudaLaunchKernel(void *, dim3, dim3, void **, size_t, cudaStream_t) { return cudaErrorUnknown; }
cudaError_t __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return cudaSuccess; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaErrorUnknown; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void *) { return 1; }
void **__cudaRegisterFatBinary(void *) { static void *p; return &p; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
char __cudaInitModule(void **) { return 1; }
}
"""

MAIN = r"""
#include <stdio.h>
#include <stdlib.h>
#include "mrc_internal.h"
extern "C" void fake_device(int d, int clusters);
extern unsigned last_grid, last_cluster;
extern size_t last_smem;
void mrc_prof_pre(int, cudaStream_t) {}
void mrc_prof_post(int, cudaStream_t, double, double) {}
// argv: device clusters init d m0 ...
int main(int argc, char **argv)
{
    static SegParams<SeedArgs> P;
    for (int i = 1; i + 4 < argc; i += 5) {
        fake_device(atoi(argv[i]), atoi(argv[i + 1]));
        const int init = atoi(argv[i + 2]) ? (int)mrc_seed_init() : 0;
        P.nseg = 1;
        P.a[0] = SeedArgs{nullptr, nullptr, atoi(argv[i + 3]), atoi(argv[i + 4]), nullptr};
        const int e = (int)mrc_seed(P, 0);
        printf("%d %d %u %u %zu\n", init, e, last_cluster, last_grid, last_smem);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def seed(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("needs nvcc")
    d = tmp_path_factory.mktemp("seed")
    (d / "fake.cpp").write_text(FAKE)
    (d / "main.cu").write_text(MAIN)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-cudart", "none", "-I", CSRC,
                    "--expt-relaxed-constexpr", "-o", str(d / "seed"), str(d / "main.cu"), str(d / "fake.cpp"),
                    os.path.join(CSRC, "seed.cu")], check=True, capture_output=True, text=True)

    def run(*steps):
        out = subprocess.run([str(d / "seed")] + [str(x) for s in steps for x in s], check=True, capture_output=True, text=True)
        return [tuple(int(x) for x in line.split()) for line in out.stdout.splitlines()]

    return run


@pytest.mark.parametrize("init", [1, 0])
@pytest.mark.parametrize("d", [3, 64])
def test_every_device_gets_its_own_attributes(seed, d, init):
    """Device 0 places clusters of 16 CTAs, device 1 too, device 2 none (8 are used there)."""
    got = seed((0, 1, 1, d, 2), (1, 1, init, d, 2), (2, 0, init, d, 2), (0, 1, 0, d, 2), (1, 1, 0, d, 2))
    assert [(g[0], g[1]) for g in got] == [(0, 0)] * 5
    assert [g[2] for g in got] == [16, 16, 8, 16, 16]
    assert all(g[3] == g[2] for g in got)


@pytest.mark.parametrize("clusters", [0, 1])
@pytest.mark.parametrize("d", [1, 32, 33, 460, 461, 512])
def test_every_dimension_fits_either_cluster(seed, d, clusters):
    """d <= 512 starts on clusters of 8 CTAs (a device that places no larger one) as
    on 16, within the shared memory of a CTA."""
    (init, err, cluster, grid, smem), = seed((0, clusters, 1, d, 2))
    assert (init, err, cluster, grid) == (0, 0, 16 if clusters else 8, 16 if clusters else 8)
    assert smem <= 216 * 1024
