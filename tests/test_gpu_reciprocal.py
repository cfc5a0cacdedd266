"""The reciprocal of the FP64 small-grid step and of the stress and heat-flux
read-out (one cubic step from the hardware's estimate) against CUDA's."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(scope="module")
def lbm():
    return need_gpu()


CU = r"""
#include "k_step_cellwarp64.cuh"
__global__ void k(const double *x, double *mine, double *cuda, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) mine[i] = lbm::rcp_cubic(x[i]), cuda[i] = __drcp_rn(x[i]);
}
extern "C" int both(const double *x, double *mine, double *cuda, int n) {
    double *d;
    if (cudaMalloc(&d, 3 * sizeof(double) * n)) return 1;
    cudaMemcpy(d, x, sizeof(double) * n, cudaMemcpyHostToDevice);
    k<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * n, n);
    cudaMemcpy(mine, d + n, sizeof(double) * n, cudaMemcpyDeviceToHost);
    cudaMemcpy(cuda, d + 2 * n, sizeof(double) * n, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)cudaGetLastError();
}
"""


def test_reciprocal_against_cuda(lbm, tmp_path):
    from paper_1209_5201_gb300 import build
    src, so = tmp_path / "rcp.cu", str(tmp_path / "rcp.so")
    src.write_text(CU)
    subprocess.run([os.path.join(build._cuda_home(), "bin", "nvcc"), *build.ARCH, "-std=c++17", "-shared",
                    "-Xcompiler", "-fPIC", "-I", build.CSRC, "-I", build.INCLUDE, "-o", so, str(src)], check=True)
    both = C.CDLL(so).both
    rng, ptr = np.random.default_rng(4), lambda a: a.ctypes.data_as(C.POINTER(C.c_double))
    # densities, K + rho / 2 and 1 + h over the Knudsen numbers in use, all mantissas
    for lo, hi in ((0.99, 1.01), (0.5, 2.0), (0.5, 1e4), (1.0, 2.0), (1e-30, 1e30)):
        x = lo * (hi / lo) ** rng.random(1 << 18)
        mine, cuda = np.empty_like(x), np.empty_like(x)
        assert both(ptr(x), ptr(mine), ptr(cuda), C.c_int(len(x))) == 0
        ulp = np.spacing(cuda)
        assert np.all(np.abs(mine - cuda) <= ulp)
        # the last step's rounding and the cubic term dropped before it: 2^-60
        # of the value for an estimate of 20 bits, 2^-7 ulp at most
        err = np.abs((1 - x.astype(LD) * mine) / x) / ulp
        assert float(np.max(err)) <= 0.5 + 2.0 ** -6 and np.mean(mine != cuda) < 0.01
