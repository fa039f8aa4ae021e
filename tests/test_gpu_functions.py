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
enum { F_ERF_SERIES, F_EXP, F_RCP, F_RSQRT, F_SQRT_PAIR, F_SINCOS_HALF, F_EWALD_ERF, F_EWALD_ERFC, F_NORMALS };
template <int F>
__global__ void apply(int n, const double* __restrict__ in, double* __restrict__ o0, double* __restrict__ o1, EwTable ew) {
    __shared__ ToyTables toy;
    if constexpr (F == F_NORMALS) fill_tables(toy);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if constexpr (F == F_NORMALS) {        // in: [n][4] 32-bit words
        toy_normals(((const uint4*)in)[i], toy, o0[i], o1[i]);
        return;
    }
    const double x = in[i];
    if constexpr (F == F_ERF_SERIES) o0[i] = erf_over_r_series(x, o1[i]);
    if constexpr (F == F_EXP) o0[i] = qexp(x);
    if constexpr (F == F_RCP) o0[i] = qrcp(x);
    if constexpr (F == F_RSQRT) o0[i] = qrsqrt(x);
    if constexpr (F == F_SQRT_PAIR) o0[i] = qsqrt_pair(x);
    if constexpr (F == F_SINCOS_HALF) sincos_half(x, o0[i], o1[i]);
    if constexpr (F == F_EWALD_ERF || F == F_EWALD_ERFC) o0[i] = ew_eval<true>(ew, F == F_EWALD_ERFC, x, o1 + i);
}
}  // namespace qmc
using namespace qmc;
// kl = kappa L with L = 1 (the Ewald table)
extern "C" int run(int f, int n, const double* in, double* o0, double* o1, double kl) {
    const int grid = (n + 127) / 128;
    EwTable ew{};
    double* t = nullptr;
    if (f == F_EWALD_ERF || f == F_EWALD_ERFC) {
        const double h = 0.75 / (kEwNodes - 1);
        if (cudaMalloc(&t, sizeof(double) * 2 * kEwNodes * kEwTerms) != cudaSuccess) return 1;
        launch_ewald_table(kl, h, t, nullptr);
        ew = EwTable{t, h, 1.0 / h, 1.0, 1.0, 1.0};
    }
#define CASE(F) case F: apply<F><<<grid, 128>>>(n, in, o0, o1, ew); break;
    switch (f) {
        CASE(F_ERF_SERIES) CASE(F_EXP) CASE(F_RCP) CASE(F_RSQRT) CASE(F_SQRT_PAIR) CASE(F_SINCOS_HALF)
        CASE(F_EWALD_ERF) CASE(F_EWALD_ERFC) CASE(F_NORMALS)
    }
    const bool ok = cudaDeviceSynchronize() == cudaSuccess;
    if (t) cudaFree(t);
    return !ok;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    """run(name, x, kappa L) -> (first output, second output) of the function on the device."""
    import torch
    d = tmp_path_factory.mktemp("functions")
    src, so = d / "functions.cu", d / "libfunctions.so"
    src.write_text(PROGRAM)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, *gbuild.ARCH, *gbuild.FLAGS, "-shared", "-I", gbuild.CSRC, str(src), "-o", str(so)], check=True)
    lib = C.CDLL(os.fspath(so))
    names = PROGRAM[PROGRAM.index("enum {") + 6:PROGRAM.index("}", PROGRAM.index("enum {"))].replace(" ", "").split(",")

    def call(name, x, kl=0.0):
        n = len(x)
        x = torch.tensor(np.ascontiguousarray(x).view(np.float64), device="cuda")
        out = torch.zeros(2, n, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        ptr = lambda t: C.c_void_p(t.data_ptr())
        assert lib.run(names.index(name), n, ptr(x), ptr(out[0]), ptr(out[1]), C.c_double(kl)) == 0
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


def _ulps(got, ref):
    """|got - ref| in units of the last place of ref (an extended-precision value)."""
    return np.max(np.abs((got - ref) / np.spacing(np.abs(ref.astype(np.float64)))))


# 2^(j/64) and the final multiply-add, half a unit each; the polynomial's last rounding and that of
# the reduced argument 2^-8 of one each (|p| <= 2^-7.5), the truncation (1.1e-18) 2^-6
def test_table_exponential(run):
    rng = np.random.default_rng(0)
    k = np.arange(-63700, 64500)                                        # interval ends, (k + 1/2) ln 2 / 64
    ends = ((k + 0.5) * (np.log(LD(2)) / 64)).astype(np.float64)
    x = np.concatenate([rng.uniform(-690, 690, 400000), rng.uniform(-1, 1, 100000), rng.uniform(-1e-6, 1e-6, 1000),
                        ends, np.nextafter(ends, 1e9), np.nextafter(ends, -1e9), k * np.log(2.0) / 64,
                        [0.0, -0.0, np.nextafter(690.0, 0), np.nextafter(-690.0, 0)]])
    x = x[np.abs(x) < 690]
    assert _ulps(run("F_EXP", x)[0], np.exp(x.astype(LD))) <= 1.02
    # from 690 on the library's function (one unit in the last place), denormals and limits included
    x = np.concatenate([rng.uniform(-746, -690, 20000), rng.uniform(690, 709.7, 20000), [-690.0, 690.0, -745.2, -746.0]])
    assert _ulps(run("F_EXP", x)[0], np.exp(x.astype(LD))) <= 1.0 + 2.0 ** -10
    with np.errstate(over="ignore"):
        lim = np.array([-747.0, -1e4, -np.inf, 710.0, np.inf])
        assert np.array_equal(run("F_EXP", lim)[0], np.exp(lim))
    assert np.isnan(run("F_EXP", np.array([np.nan]))[0][0])
