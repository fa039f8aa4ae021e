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


def _positive(rng, n, lo, hi):
    """Both halves of a binade and its ends, exponents from lo to hi."""
    m = np.concatenate([rng.uniform(1, 2, n), [1.0, np.nextafter(1.0, 2), np.nextafter(2.0, 1)]])
    return np.ldexp(m, rng.integers(lo, hi, len(m)))


# the last multiply-add's rounding, and of the correction's own 2^-20 of one; the truncation 2^-4 at most
def test_reciprocal(run):
    x = _positive(np.random.default_rng(1), 1000000, -1000, 1000)
    assert _ulps(run("F_RCP", x)[0], 1 / x.astype(LD)) <= 0.57


# rsqrt: the last rounding and that of x y (u/2 of the result: at most half a unit); sqrt: times x,
# whose rounding is another half a unit, on a value at most a unit and a half of the result's off
def test_reciprocal_square_root(run):
    x = _positive(np.random.default_rng(2), 1000000, -1000, 1000)
    assert _ulps(run("F_RSQRT", x)[0], 1 / np.sqrt(x.astype(LD))) <= 1.07
    assert _ulps(run("F_SQRT_PAIR", x)[0], np.sqrt(x.astype(LD))) <= 2.1
    assert np.array_equal(run("F_SQRT_PAIR", np.array([0.0, -0.0]))[0], [0.0, 0.0])


# the last multiply-add's rounding and those before, scaled by x^2 / 6 and x^2 / 2 <= 1/8
def test_sine_and_cosine_of_close_pairs(run):
    x = np.concatenate([np.linspace(-0.5, 0.5, 200001), np.geomspace(1e-12, 0.5, 2000)])
    sn, cs = run("F_SINCOS_HALF", x)
    keep = x != 0.0
    assert _ulps(sn[keep], np.sin(x[keep].astype(LD))) <= 0.75 and np.all(sn[~keep] == 0.0)
    assert _ulps(cs, np.cos(x.astype(LD))) <= 0.75


def _boys(n, x):
    """F_n(x) = int_0^1 s^2n exp(-x s^2) ds by its series of positive terms."""
    term, total = np.ones_like(x) / (2 * n + 1), np.zeros_like(x)
    for j in range(1, 300):
        total += term
        term = term * 2 * x / (2 * n + 1 + 2 * j)
    return np.exp(-x) * total


# Real-space Ewald table, L = 1: erf(kappa r)/r on r^2 <= 3/4 and erfc(kappa r)/r on [1/4, 1), and
# their derivatives in r^2, at nodes, midpoints and between.  erf: exp's unit (2 u), the series and
# the recurrence's few operations on positive terms, Horner's last step: 8 u.  erfc: the
# library's five units (10 u), a square root, two divisions, three products: 16 u.  The
# truncations are the 1e-18 kappa and 2e-16 kappa^3 of common.cuh.
@pytest.mark.parametrize("kl", [0.01, 1.0, 3.0, 5.0, 6.0])
def test_ewald_table(run, kl):
    rng = np.random.default_rng(4)
    h = 0.75 / 511
    k, c = LD(kl), 2 / np.sqrt(LD(np.pi) + LD(1.2246467991473531772e-16))
    for name, lo, hi in (("F_EWALD_ERF", 0.0, 0.75), ("F_EWALD_ERFC", 0.25, 1.0)):
        i = np.arange(0, 682) * h
        r2 = np.concatenate([rng.uniform(lo, hi, 20000), i, i + 0.5 * h, i + 0.4999 * h])
        r2 = r2[(r2 >= lo) & (r2 < hi) | (r2 == lo)]
        v, d = run(name, r2, kl)
        x = k * k * r2.astype(LD)
        f0, f1 = _boys(0, x), _boys(1, x)
        if name == "F_EWALD_ERFC":           # G_n = int_0^inf - F_n
            x = np.maximum(x, LD(1e-30))
            f0 = np.sqrt(1 / (c * c)) / np.sqrt(x) - f0
            f1 = np.sqrt(1 / (c * c)) / (2 * x * np.sqrt(x)) - f1
        roundings = (16 if name == "F_EWALD_ERFC" else 8) * U
        ref, dref = c * k * f0, -c * k ** 3 * f1
        assert np.max(np.abs(v - ref) - roundings * (np.abs(ref) + kl)) <= 1e-18 * kl
        assert np.max(np.abs(d - dref) - roundings * (np.abs(dref) + kl ** 3)) <= 2e-16 * kl ** 3


# Box-Muller normals by tables: log u is good to 3 u relative (its last sum, the table and the
# exponent's product), its square root to 1.5 u + 1.5 units more, sine and cosine to 4 u absolute
# (table, series, and two products): 10 u rho in all.  Words at the log's ends (u next to 0 and
# to 1, the seams at 1 and 0.6875) and at the angles' table points and midpoints.
def test_toy_normals(run):
    rng = np.random.default_rng(6)
    w = rng.integers(0, 2 ** 32, (400000, 4), dtype=np.uint64)

    def words(v):                            # the two words of 53 bits v
        v = np.asarray(v, dtype=np.uint64)
        return np.stack([(v >> np.uint64(26)) << np.uint64(5), (v & np.uint64(2 ** 26 - 1)) << np.uint64(6)], -1)
    ends = np.concatenate([np.arange(64), 2 ** 53 - 1 - np.arange(4096),
                           (0.6875 * 2.0 ** (53 - np.arange(20)[:, None]) + np.arange(-3, 4)).ravel(),
                           (2.0 ** (53 - np.arange(1, 20)[:, None]) + np.arange(-3, 4)).ravel()]).astype(np.uint64)
    angle = (np.arange(512)[:, None] * 2 ** 44 + np.arange(-3, 4)).ravel() % 2 ** 53
    edge = np.concatenate([np.concatenate([words(ends), rng.integers(0, 2 ** 32, (len(ends), 2), dtype=np.uint64)], -1),
                           np.concatenate([rng.integers(0, 2 ** 32, (len(angle), 2), dtype=np.uint64), words(angle)], -1)])
    w = np.concatenate([w, edge]).astype(np.uint32)
    g0, g1 = run("F_NORMALS", w)
    bits = lambda a, b: (a >> 5).astype(LD) * 2 ** 26 + (b >> 6).astype(LD) + LD(0.5)

    def u53(a, b):                           # the kernel's uniform: 53 bits and a half, rounded once to FP64
        return bits(a, b).astype(np.float64).astype(LD) / LD(2) ** 53
    u1, u2 = u53(w[:, 0], w[:, 1]), u53(w[:, 2], w[:, 3])
    rho, th = np.sqrt(-2 * np.log(u1)), 2 * (LD(np.pi) + LD(1.2246467991473531772e-16)) * u2
    for g, ref in ((g0, rho * np.cos(th)), (g1, rho * np.sin(th))):
        assert np.max(np.abs(g - ref) - 10 * U * rho) <= 0.0
