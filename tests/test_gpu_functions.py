"""The kernels' own elementary functions, on the device, against extended precision
(numpy's longdouble) over the ranges they are used on and at the edges of their tables.

The functions are compiled from the kernels' sources into a small library.  u = 2^-53;
every bound is the sum of the roundings of the function's last operations (given at
each test) and of the truncation its comment states.
"""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1605_08423_gb300 import build as gbuild

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
LD = np.longdouble
PROGRAM = r"""
#include "k_measure.cu"
#include "k_setup.cu"
#include "k_toy.cu"
namespace qmc {
enum { F_ERF_SERIES };
template <int F>
__global__ void apply(int n, const double* __restrict__ in, double* __restrict__ o0, double* __restrict__ o1) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = in[i];
    if constexpr (F == F_ERF_SERIES) o0[i] = erf_over_r_series(x, o1[i]);
}
}  // namespace qmc
using namespace qmc;
extern "C" int run(int f, int n, const double* in, double* o0, double* o1) {
    const int grid = (n + 127) / 128;
    switch (f) {
    case F_ERF_SERIES: apply<F_ERF_SERIES><<<grid, 128>>>(n, in, o0, o1); break;
    default: return 1;
    }
    return cudaDeviceSynchronize() != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    """run(name, x) -> (first output, second output) of the function on the device."""
    import torch
    d = tmp_path_factory.mktemp("functions")
    src, so = d / "functions.cu", d / "libfunctions.so"
    src.write_text(PROGRAM)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, *gbuild.ARCH, *gbuild.FLAGS, "-shared", "-I", gbuild.CSRC, str(src), "-o", str(so)], check=True)
    lib = C.CDLL(os.fspath(so))
    names = PROGRAM[PROGRAM.index("enum {") + 6:PROGRAM.index("}", PROGRAM.index("enum {"))].replace(" ", "").split(",")

    def call(name, x):
        x = torch.tensor(np.ascontiguousarray(x), device="cuda")
        n = len(x)
        out = torch.zeros(2, n, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        ptr = lambda t: C.c_void_p(t.data_ptr())
        assert lib.run(names.index(name), n, ptr(x), ptr(out[0]), ptr(out[1])) == 0
        return out[0].cpu().numpy(), out[1].cpu().numpy()
    return call


# sum_n (-x)^n / (n! (2n + 1)) and its derivative in x: Horner in FP64 on [0, 2/3], where the
# value is 0.81 to 1 and the derivative -0.23 to -1/3; the last operation's rounding (half a
# unit of 1), the one before scaled by x, and the coefficients' own, below 2 u in all
def test_close_pair_erf_series(run):
    x = np.linspace(0.0, 2.0 / 3.0, 100001)
    v, d = run("F_ERF_SERIES", x)
    xl, term = x.astype(LD), np.ones(len(x), LD)
    ref, dref = np.zeros(len(x), LD), np.zeros(len(x), LD)
    for n in range(40):                      # term = (-x)^n / n!
        ref += term / (2 * n + 1)
        dref -= term / (2 * n + 3)
        term = term * -xl / (n + 1)
    assert np.max(np.abs(v - ref)) <= 2 * U
    assert np.max(np.abs(d - dref)) <= 2 * U
