"""Which form the distance of a small tensor takes: its host code against a fake of the CUDA runtime (nothing is launched)."""
import os
import subprocess

import pytest

from paper_2510_02822_b200 import build

FAKE = r"""
#include <cuda_runtime_api.h>
#include <stdio.h>
#include <stdlib.h>
#include "flexiq.h"
static int clusters, occupancy_error, launch_error;
static cudaError_t last = cudaSuccess;
static cudaError_t said(const char *what, int error) { printf("%s%s ", what, error ? "!" : ""); if (error) last = (cudaError_t)error; return (cudaError_t)error; }
namespace flexiq {
int device_sm_count(int) { return 148; }
int check_device_sm100() { return 0; }
int set_error(int code, const char *, ...) { return code; }
}
extern "C" {
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *) { *n = clusters; return said("ask", occupancy_error); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **) { return said("cluster", launch_error); }
cudaError_t cudaLaunchKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t) { return said("grid", 0); }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return said("clear", 0); }
}
int main(int, char **v)
{
    clusters = atoi(v[1]); occupancy_error = atoi(v[2]); launch_error = atoi(v[3]);
    const long long n = atoll(v[4]);
    for (int i = 0; i < 2; ++i) printf("%d%s", flexiq_sq_distance_i8((const int8_t *)16, (const int8_t *)32, n, (int64_t *)64, nullptr), i ? "" : " | ");
    printf(" %d", (int)last);
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("distance")
    (d / "fake.cpp").write_text(FAKE)
    nvcc, obj = build._nvcc(), str(d / "evolution.o")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))
    subprocess.run([nvcc, *build.NVCC_FLAGS, "-c", os.path.join(build.CSRC, "flexiq_evolution.cu"), "-o", obj], check=True)
    subprocess.run(["g++", "-std=c++17", f"-I{cuda}/include", f"-I{os.path.dirname(build._DIR)}/include", str(d / "fake.cpp"), obj, "-o", str(d / "host")], check=True)
    return lambda *args: subprocess.run([str(d / "host"), *map(str, args)], check=True, capture_output=True, text=True).stdout


@pytest.mark.parametrize("clusters, occupancy_error, launch_error, n, does", [
    (1, 0, 0, 1 << 20, "ask cluster 0 | cluster 0 0"),                                    # room for a cluster: asked once
    (0, 0, 0, 1 << 20, "ask clear grid 0 | clear grid 0 0"),                              # none: the grid
    (1, 98, 0, 1 << 20, "ask! clear grid 0 | clear grid 0 0"),                            # no answer: the grid, and no error is left behind
    (1, 0, 98, 1 << 20, "ask cluster! clear grid 0 | cluster! clear grid 0 0"),           # refused all the same
    (1, 0, 0, (2 << 20) + 16, "clear grid 0 | clear grid 0 0"), (0, 0, 0, 0, "clear 0 | clear 0 0")])
def test_form_of_the_distance(host, clusters, occupancy_error, launch_error, n, does):
    assert host(clusters, occupancy_error, launch_error, n) == does
