"""``iq_sigma_bound`` where a launch fails, without a GPU: the file is compiled with fakes of the runtime's calls, of which one launch
reports an error.  Only a refusal for want of room sends the call to the radix select; any other error is the caller's to see."""
import os
import subprocess

import pytest

from paper_2006_11735_b200 import build
from paper_2006_11735_b200.binding import ERR_CUDA, OK

PROGRAM = r"""
#include <cuda.h>
#include <cuda_runtime.h>
#include <cmath>
#include <cstdarg>
#include <cstddef>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
static int launches, fail_at;
static cudaError_t error_of_launch;
template <typename... P, typename... A> static cudaError_t fake_launch(const cudaLaunchConfig_t *, void (*)(P...), A...) { return launches++ == fail_at ? error_of_launch : cudaSuccess; }
static cudaError_t fake_alloc(void **p, size_t n, unsigned = 0) { *p = calloc(1, n); return cudaSuccess; }
static cudaError_t fake_free(void *p) { free(p); return cudaSuccess; }
static cudaError_t fake_address(void **d, void *h, unsigned) { *d = h; return cudaSuccess; }
static cudaError_t fake_set(void *p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
static cudaError_t fake_wait(cudaStream_t) { return cudaSuccess; }
static cudaError_t fake_last() { return cudaSuccess; }
static cudaError_t fake_capturing(cudaStream_t, cudaStreamCaptureStatus *s) { *s = cudaStreamCaptureStatusNone; return cudaSuccess; }
#define cudaLaunchKernelEx fake_launch
#define cudaMalloc fake_alloc
#define cudaHostAlloc fake_alloc
#define cudaFree fake_free
#define cudaFreeHost fake_free
#define cudaHostGetDevicePointer fake_address
#define cudaMemset fake_set
#define cudaStreamSynchronize fake_wait
#define cudaGetLastError fake_last
#define cudaStreamIsCapturing fake_capturing
#include "kernel_calib.cu"
namespace iconv {
void set_error(const char *, ...) {}
int cuda_fail(cudaError_t, const char *) { return ICONV_ERR_CUDA; }
int current_device_slot() { return 0; }
}
int main(int argc, char **argv)
{
    error_of_launch = (cudaError_t)atoi(argv[1]);
    fail_at = atoi(argv[2]);
    static int32_t y[100000];
    int32_t bound = 0;
    printf("%d\n", iq_sigma_bound(y, 100000, 0.0015, &bound, nullptr));
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("calib")
    (d / "errors.cu").write_text(PROGRAM)
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, "-o", str(d / "errors"),
                    str(d / "errors.cu")], check=True)
    return str(d / "errors")


@pytest.mark.parametrize("launch", [0, 1, 2])
@pytest.mark.parametrize("error, status", [(0, OK), (9, OK), (701, OK), (912, OK), (2, ERR_CUDA), (98, ERR_CUDA), (400, ERR_CUDA), (719, ERR_CUDA), (905, ERR_CUDA)])
def test_a_failed_launch_is_reported_unless_it_means_that_a_cluster_has_no_room(program, error, status, launch):
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="")              # (its arrays are host memory: the radix select's launches go nowhere)
    out = subprocess.run([program, str(error), str(launch)], check=True, capture_output=True, text=True, env=env, timeout=120).stdout
    assert int(out) == status
