"""GPU: the fp64 reciprocal and reciprocal square root of the factorisations (csrc/device_helpers.cuh) against extended precision.

Reciprocal: the last Newton step's residual is exact to 2^-90 and its result is rounded once, so the relative error is at most
2^-53 (and the square of the step before, far below).  Reciprocal square root: the residual 1 - (x y) y carries the rounding of
x y, up to 2^-53, half of which reaches the result, and that is rounded once: 1.5 x 2^-53."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2503_24358_b200 import build as sq_build

pytestmark = pytest.mark.gpu

SOURCE = r'''
#include "device_helpers.cuh"
__global__ void apply(const double *x, double *rcp, double *rsqrt, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) { rcp[i] = rcp_nr(x[i]); rsqrt[i] = rsqrt_nr(x[i]); }
}
extern "C" int run(const double *x, double *rcp, double *rsqrt, int n)
{
    apply<<<(n + 255) / 256, 256>>>(x, rcp, rsqrt, n);
    return (int)cudaDeviceSynchronize();
}
'''


def test_relative_errors(tmp_path):
    src, lib = tmp_path / "r.cu", tmp_path / "r.so"
    src.write_text(SOURCE)
    subprocess.run([sq_build._nvcc(), *sq_build.NVCC_FLAGS, "-I", sq_build.CSRC, "-shared", str(src), "-o", str(lib)], check=True)
    run = ctypes.CDLL(os.fspath(lib)).run
    run.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]
    rng = np.random.default_rng(2)
    powers = np.ldexp(1.0, np.arange(-960, 961, 8))
    x = np.concatenate([rng.uniform(1.0, 4.0, 200000), np.exp(rng.uniform(np.log(1e-290), np.log(1e290), 200000)),
                        powers, np.nextafter(powers, 0), np.nextafter(powers, np.inf)])
    d = torch.from_numpy(x).cuda()
    a, b = torch.empty_like(d), torch.empty_like(d)
    assert run(d.data_ptr(), a.data_ptr(), b.data_ptr(), len(x)) == 0
    t = x.astype(np.longdouble)
    rcp = np.abs(a.cpu().numpy() * t - 1).max()
    rsqrt = np.abs(b.cpu().numpy() * np.sqrt(t) - 1).max()
    print(f"rcp {float(rcp) * 2 ** 53:.4f}, rsqrt {float(rsqrt) * 2 ** 53:.4f} x 2^-53")
    assert rcp <= 1.001 * 2.0 ** -53 and rsqrt <= 1.501 * 2.0 ** -53
