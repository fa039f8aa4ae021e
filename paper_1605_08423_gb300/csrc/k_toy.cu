// k_toy.cu -- the rotating-spring toy model of the SI ("A simple toy model") on
// which the SI compares its integrators: many independent trajectories, one
// thread each, FP64 throughout, state in registers for the whole run.
//
//   U(R) = k/2 (|R| - a)^2 in the plane, f = -grad U = -k (r - a) R / r.
//   Both acceleration matrices of the SI have the radial form
//     S = s_r P_r + s_t P_t,   P_r = R R^T / r^2,  P_t = I - P_r,
//   G_lambda (as printed): s_r = 1/lambda, s_t = 1;
//   H + mu G_lambda:       s_r = k + mu/lambda, s_t = k (1 - a/r) + mu  (H = k P_r + k (1 - a/r) P_t).
//   Then S^{-1} = P_r/s_r + P_t/s_t and the cumbersome term of Eq. standard is
//     Gamma_j = sum_i d_i (S^{-1})_{ji} = R_j [ (1/s_r)'/r + (1/s_r - 1/s_t)/r^2 ],
//   with (1/s_r)' = 0 for both choices (two dimensions: sum_i d_i (R_j R_i / r^2) = R_j / r^2).
//
// Schemes (z = L^{-T} xi, S(R) = L L^T, xi two Box-Muller normals from Philox
// counter (trajectory, step, 0, kToy)):
//   plain     R' = R + D f + sqrt(2 T D) xi                             (S = I)
//   standard  R' = R + D S^{-1} f + T D Gamma + sqrt(2 T D) z          (Eq. standard, gamma = 0)
//   first     y = R + sqrt(2 T D) z,
//             R' = y + D S^{-1} f - 1/2 S^{-1} [S(y) - S(R)] (y - R)   (Eq. smartMarkov)
//   fast      R' = R + D S^{-1} f + sqrt(2 T D) z
//                  - 1/2 S^{-1} [S(R_prev) - S(R)] (R_prev - R)        (Eq. finaldyn)
//   adopted   R' = R + Dt S^{-1} [f - (S(R_prev) - S(R))(R_prev - R)/(2 Db)]
//                  + sqrt(2 T Db) z                                      (Eq. finaldyn_new)
//   norogna   R' = R + D S^{-1} f + sqrt(2 T D) z                      (Eq. norogna)
// R_prev = R on the first step.  Per trajectory the kernel writes
// [x, y, sum U, sum U^2, sum |R|, polar angle travelled, status] with the sums
// over the positions after steps n_burn..n_steps-1; status = s + 1 when S(R) was
// not positive definite at step s (the trajectory stops there), else 0.
#include "common.cuh"
#include "kernels.cuh"

#include "qmcmd.h"

#include <cmath>

namespace qmc {

namespace {

constexpr uint32_t kToy = 8;   // Philox purpose word of the toy-model noise

// Tables of one block (shared memory, filled at its start by the library's log and
// sincospi): 1/c and log c of 128 centres c over [0.6875, 1.375), and sin, cos of
// 2 pi j / 256.
struct ToyTables {
    double2 lg[128], cs[256];
};
constexpr long long kLogOff = 0x3fe6000000000000LL;   // bits of 0.6875

__device__ __forceinline__ void fill_tables(ToyTables& T) {
    for (int i = threadIdx.x; i < 128; i += blockDim.x) {
        const double lo = __longlong_as_double(kLogOff + ((long long)i << 45));
        const double hi = __longlong_as_double(kLogOff + ((long long)(i + 1) << 45));
        // the two intervals that meet at 1 keep c = 1, so that log u -> 0 keeps its relative accuracy
        const double c = (hi == 1.0 || lo == 1.0) ? 1.0 : 1.0 / (0.5 * (lo + hi));
        T.lg[i] = make_double2(c, -log(c));
    }
    for (int j = threadIdx.x; j < 256; j += blockDim.x) {
        double sn, cs;
        sincospi(j / 128.0, &sn, &cs);
        T.cs[j] = make_double2(sn, cs);
    }
    __syncthreads();
}

// 2^53 u of the 53-bit uniform u53(a, b) (the same rounding: one addition of 1/2).
__device__ __forceinline__ double u53_scaled(uint32_t a, uint32_t b) {
    const double hi = __hiloint2double(0x43300000, (int)(a >> 5)) - 4503599627370496.0;      // 2^52 + k - 2^52
    const double lo = __hiloint2double(0x43300000, (int)(b >> 6)) - 4503599627370495.5;      // + 1/2
    return fma(hi, 67108864.0, lo);
}

// The step's two normals from its Philox block, Box-Muller: -2 log u by table and
// series (P. T. P. Tang, ACM Trans. Math. Softw. 16, 1990; r <= 2^-7, to r^7), the
// angle by table and series (|x| <= pi / 256).  36 FP64 operations where the
// library's log, sqrt and sincospi take some 85.
__device__ __forceinline__ void toy_normals(uint4 w, const ToyTables& T, double& xi0, double& xi1) {
    const double v1 = u53_scaled(w.x, w.y), v2 = u53_scaled(w.z, w.w);
    const long long ix = __double_as_longlong(v1), tmp = ix - kLogOff;
    const int e = (int)(tmp >> 52) - 53;                                       // u = 2^e z
    const double z = __longlong_as_double(ix - (tmp & (long long)0xfff0000000000000ULL));
    const double2 lc = T.lg[(int)(tmp >> 45) & 127];
    const double r = fma(z, lc.x, -1.0);
    double q = fma(r, 1.0 / 7.0, -1.0 / 6.0);
    q = fma(q, r, 0.2);
    q = fma(q, r, -0.25);
    q = fma(q, r, 1.0 / 3.0);
    q = fma(q, r, -0.5);
    const double ed = __hiloint2double(0x43300000, e + 0x40000000) - (4503599627370496.0 + 1073741824.0);
    const double lg = fma(ed, 0.69314718055994530942, lc.y) + fma(q, r * r, r);
    const double rho = qsqrt_pair(-2.0 * lg);
    const double magic = 6755399441055744.0;                                   // 1.5 * 2^52
    const double jm = fma(v2, 256.0 / 9007199254740992.0, magic);
    const double x = 6.2831853071795864769 / 9007199254740992.0 * fma(-(9007199254740992.0 / 256.0), jm - magic, v2);
    const double y = x * x;
    const double sn = fma(fma(y, 1.0 / 120.0, -1.0 / 6.0) * y, x, x);
    const double cs = fma(fma(fma(y, -1.0 / 720.0, 1.0 / 24.0), y, -0.5), y, 1.0);
    const double2 t = T.cs[__double2loint(jm) & 255];
    xi0 = rho * (t.y * cs - t.x * sn);
    xi1 = rho * (t.x * cs + t.y * sn);
}

// The same from the library's log and sincospi, without the tables.
__device__ __forceinline__ void toy_normals_library(uint4 w, double& xi0, double& xi1) {
    const double rho = sqrt(-2.0 * log(u53(w.x, w.y)));
    double sn, cs;
    sincospi(2.0 * u53(w.z, w.w), &sn, &cs);
    xi0 = rho * cs;
    xi1 = rho * sn;
}

// x > 0 for a finite or infinite x, false for NaN, on the integer pipe
__device__ __forceinline__ bool positive(double x) {
    const int h = __double2hiint(x);
    return h > 0 && h <= 0x7ff00000;
}

// One thread per trajectory.  The FP64 pipe bounds it, so the step is written for
// few FP64 operations: S = st I + d R R^T with d = (s_r - s_t) / r^2, so that
//   S^{-1} v = p_t v + (p_r - p_t)/r^2 (R.v) R,   p = 1/s,
//   (S(Q) - S(R)) e = (st_Q - st) e + d_Q (Q.e) Q - d (R.e) R,
// take dot products instead of triangular solves, the factor L is only formed for
// the noise z = L^{-T} xi, and with S = G_lambda its second diagonal entry follows
// from det S = 1/lambda.  100003 trajectories of 500 adopted steps: 15.7 ms with the
// Cholesky solves and the library's log, sqrt, sincospi and rsqrt, 10.9 ms now.
// The polar angle travelled: the sum of the per-step increments (each below pi in
// magnitude) equals phi_end - phi_0 + 2 pi (net turns across the negative x axis),
// so only the crossings are counted per step -- sign tests on the y coordinates and
// on the cross product R x R' -- and phi comes from atan2 at the two ends.
// TAB: normals by the tables, which every block fills first; without them (launch_scheme)
// the library's functions.
template <int SCHEME, bool HG, bool TAB>
__global__ void __launch_bounds__(128) toy_kernel(ToyDev p, int n_traj, const double* __restrict__ xy0,
                                                  double* __restrict__ out) {
    __shared__ ToyTables T;
    if constexpr (TAB) fill_tables(T);
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_traj) return;
    const double x0 = xy0[2 * t], y0 = xy0[2 * t + 1];
    double x = x0, y = y0, xp = x, yp = y;
    double r2 = x * x + y * y, ir = qrsqrt(r2), r = r2 * ir;
    double su = 0.0, su2 = 0.0, sr = 0.0, status = 0.0;
    int turns = 0;
    const double D = p.delta, ka = p.k * p.a, pr = 1.0 / p.sr_const;
    auto s_t = [&](double ir_) { return HG ? fma(-ka, ir_, p.k) + p.mu : 1.0; };
    double stp = s_t(ir), dp = (p.sr_const - stp) * (ir * ir);      // S(R_prev), carried from step to step
    const double c22 = HG ? 0.0 : rsqrt(p.sr_const);                // 1 / sqrt(det S) of G_lambda
    for (int s = 0; s < p.n_steps; ++s) {
        double xi0, xi1;
        const uint4 w = philox((uint32_t)t, (uint32_t)s, 0u, kToy, p.key);
        if constexpr (TAB) toy_normals(w, T, xi0, xi1);
        else toy_normals_library(w, xi0, xi1);
        const double fr = fma(ka, ir, -p.k);                        // f = fr R
        // terms added in the order of the schemes above
        double xn, yn, st = 1.0, d = 0.0;
        if constexpr (SCHEME == QMC_TOY_PLAIN) {
            xn = fma(p.amp, xi0, fma(D, fr * x, x));
            yn = fma(p.amp, xi1, fma(D, fr * y, y));
        } else {
            const double ir2 = ir * ir;
            st = s_t(ir);
            d = (p.sr_const - st) * ir2;
            const double dx = d * x, s11 = fma(dx, x, st), s12 = dx * y;
            if (!positive(s11)) { status = s + 1; break; }
            const double i11 = qrsqrt(s11), l21 = s12 * i11;
            double i22;
            if constexpr (HG) {
                const double q = fma(-l21, l21, fma(d * y, y, st));
                if (!positive(q)) { status = s + 1; break; }
                i22 = qrsqrt(q);
            } else {
                i22 = s11 * i11 * c22;
            }
            const double z1 = xi1 * i22, z0 = fma(-l21, z1, xi0) * i11;
            const double pt = HG ? qrcp(st) : 1.0;
            const double gs = (pr - pt) * ir2;
            // S^{-1} v
            auto solve = [&](double vx, double vy, double& wx, double& wy) {
                const double c = gs * fma(x, vx, y * vy);
                wx = HG ? fma(c, x, pt * vx) : fma(c, x, vx);
                wy = HG ? fma(c, y, pt * vy) : fma(c, y, vy);
            };
            // (S(Q) - S(R)) e
            auto diff = [&](double stq, double dq, double qx, double qy, double ex, double ey, double& vx, double& vy) {
                const double a = dq * fma(qx, ex, qy * ey), b = d * fma(x, ex, y * ey);
                vx = fma(a, qx, -(b * x));
                vy = fma(a, qy, -(b * y));
                if constexpr (HG) { vx = fma(stq - st, ex, vx); vy = fma(stq - st, ey, vy); }
            };
            const double prf = pr * fr;                              // S^{-1} f = prf R
            if constexpr (SCHEME == QMC_TOY_STANDARD) {
                const double g = p.T * D * gs;                       // Gamma = gs R
                xn = fma(p.amp, z0, fma(g, x, fma(D, prf * x, x)));
                yn = fma(p.amp, z1, fma(g, y, fma(D, prf * y, y)));
            } else if constexpr (SCHEME == QMC_TOY_FIRST) {
                const double ex = p.amp * z0, ey = p.amp * z1;       // y - R
                const double qx = x + ex, qy = y + ey;
                const double iq = qrsqrt(fma(qx, qx, qy * qy));
                const double stq = s_t(iq);
                double vx, vy, wx, wy;
                diff(stq, (p.sr_const - stq) * (iq * iq), qx, qy, ex, ey, vx, vy);
                solve(vx, vy, wx, wy);
                const double g = D * prf;
                xn = fma(-0.5, wx, fma(g, x, qx));
                yn = fma(-0.5, wy, fma(g, y, qy));
            } else if constexpr (SCHEME == QMC_TOY_FAST || SCHEME == QMC_TOY_ADOPTED) {
                constexpr bool kAdopted = SCHEME == QMC_TOY_ADOPTED;
                double vx, vy, wx, wy;
                diff(stp, dp, xp, yp, xp - x, yp - y, vx, vy);
                solve(vx, vy, wx, wy);
                if constexpr (kAdopted) {
                    xn = fma(p.ampb, z0, fma(p.dt, fma(-p.half_idb, wx, prf * x), x));
                    yn = fma(p.ampb, z1, fma(p.dt, fma(-p.half_idb, wy, prf * y), y));
                } else {
                    xn = fma(-0.5, wx, fma(p.amp, z0, fma(D, prf * x, x)));
                    yn = fma(-0.5, wy, fma(p.amp, z1, fma(D, prf * y, y)));
                }
            } else {   // QMC_TOY_NOROGNA
                xn = fma(p.amp, z0, fma(D, prf * x, x));
                yn = fma(p.amp, z1, fma(D, prf * y, y));
            }
        }
        {
            const bool up = __double_as_longlong(y) >= 0, upn = __double_as_longlong(yn) >= 0;
            if (up != upn) {
                const long long cr = __double_as_longlong(x * yn - y * xn);
                if (up && cr > 0) ++turns;            // counter-clockwise across the negative x axis
                else if (!up && cr < 0) --turns;      // clockwise across it
            }
        }
        xp = x; yp = y; stp = st; dp = d;
        x = xn; y = yn;
        r2 = x * x + y * y;
        ir = qrsqrt(r2);
        r = r2 * ir;
        if (s >= p.n_burn) {
            const double dr = r - p.a;
            const double u = 0.5 * p.k * dr * dr;
            su += u; su2 += u * u; sr += r;
        }
    }
    const double theta = atan2(y, x) - atan2(y0, x0) + 2.0 * kPi * turns;
    double* o = out + 7 * (size_t)t;
    o[0] = x; o[1] = y; o[2] = su; o[3] = su2; o[4] = sr; o[5] = theta; o[6] = status;
}

template <int SCHEME>
void launch_scheme(const ToyDev& p, int n_traj, const double* xy0, double* out, cudaStream_t st) {
    // one warp per block while every warp can have an SM's FP64 issue ports nearly to itself
    const int tpb = n_traj <= 32 * 2 * 152 ? 32 : 128, grid = (n_traj + tpb - 1) / tpb;
    // a block's tables (128 logarithms, 256 sincospi) cost more than one or two steps save:
    // the adopted scheme's 10^6 trajectories take 562 / 749 / 937 / 1124 us for 1 / 2 / 3 / 4
    // steps with them, 440 / 682 / 925 / 1165 with the library's functions (10^3: 23 / 27 /
    // 31 / 33 and 12 / 17 / 21 / 25); the other schemes cross between 2 and 4 too.
    const bool hg = p.s_mode == QMC_TOY_S_HG;
    const auto kernel = p.n_steps <= 2 ? (hg ? toy_kernel<SCHEME, true, false> : toy_kernel<SCHEME, false, false>)
                                       : (hg ? toy_kernel<SCHEME, true, true> : toy_kernel<SCHEME, false, true>);
    kernel<<<grid, tpb, 0, st>>>(p, n_traj, xy0, out);
}

}  // namespace

void launch_toy(const ToyDev& p, int n_traj, const double* xy0, double* out, cudaStream_t st) {
    if (n_traj <= 0) return;
    switch (p.scheme) {
    case QMC_TOY_PLAIN: launch_scheme<QMC_TOY_PLAIN>(p, n_traj, xy0, out, st); break;
    case QMC_TOY_STANDARD: launch_scheme<QMC_TOY_STANDARD>(p, n_traj, xy0, out, st); break;
    case QMC_TOY_FIRST: launch_scheme<QMC_TOY_FIRST>(p, n_traj, xy0, out, st); break;
    case QMC_TOY_FAST: launch_scheme<QMC_TOY_FAST>(p, n_traj, xy0, out, st); break;
    case QMC_TOY_ADOPTED: launch_scheme<QMC_TOY_ADOPTED>(p, n_traj, xy0, out, st); break;
    default: launch_scheme<QMC_TOY_NOROGNA>(p, n_traj, xy0, out, st); break;
    }
}

}  // namespace qmc

// ---------------------------------------------------------------------------
// C ABI (include/qmcmd.h)
// ---------------------------------------------------------------------------
namespace {

int toy_check(const qmc_toy_params* p, int n_traj) {
    if (!p || n_traj < 0) return QMC_ERR_INVALID;
    if (p->scheme < QMC_TOY_PLAIN || p->scheme > QMC_TOY_NOROGNA) return QMC_ERR_INVALID;
    if (p->s_mode != QMC_TOY_S_G && p->s_mode != QMC_TOY_S_HG) return QMC_ERR_INVALID;
    if (!(p->delta > 0) || !(p->lambda > 0) || p->T < 0 || p->alpha < 0 || !(p->k >= 0)) return QMC_ERR_INVALID;
    if (p->n_steps < 0 || p->n_burn < 0 || p->n_burn > p->n_steps) return QMC_ERR_INVALID;
    return QMC_OK;
}

qmc::ToyDev toy_dev(const qmc_toy_params* p) {
    qmc::ToyDev d;
    d.k = p->k; d.a = p->a; d.mu = p->mu;
    d.sr_const = p->s_mode == QMC_TOY_S_HG ? p->k + p->mu / p->lambda : 1.0 / p->lambda;
    d.T = p->T; d.delta = p->delta;
    d.dt = p->delta; d.db = p->delta;
    if (p->scheme == QMC_TOY_ADOPTED && p->alpha > 0) {
        d.dt = (1.0 - std::exp(-p->alpha * p->delta)) / p->alpha;
        d.db = (1.0 - std::exp(-2.0 * p->alpha * p->delta)) / (2.0 * p->alpha);
    }
    d.half_idb = 1.0 / (2.0 * d.db);
    d.amp = std::sqrt(2.0 * p->T * p->delta);
    d.ampb = std::sqrt(2.0 * p->T * d.db);
    d.scheme = p->scheme; d.s_mode = p->s_mode; d.n_steps = p->n_steps; d.n_burn = p->n_burn;
    d.key = qmc::make_key(p->seed);
    return d;
}

}  // namespace

extern "C" int qmc_toy_langevin_device(const qmc_toy_params* p, int n_traj, const double* xy0_dev, double* out_dev,
                                       void* stream) {
    const int rc = toy_check(p, n_traj);
    if (rc != QMC_OK) return rc;
    if (n_traj > 0 && (!xy0_dev || !out_dev)) return QMC_ERR_INVALID;
    qmc::launch_toy(toy_dev(p), n_traj, xy0_dev, out_dev, (cudaStream_t)stream);
    return cudaGetLastError() == cudaSuccess ? QMC_OK : QMC_ERR_CUDA;
}

extern "C" int qmc_toy_langevin(const qmc_toy_params* p, int n_traj, const double* xy0, double* out) {
    const int rc = toy_check(p, n_traj);
    if (rc != QMC_OK) return rc;
    if (n_traj == 0) return QMC_OK;
    if (!xy0 || !out) return QMC_ERR_INVALID;
    double *d_xy = nullptr, *d_out = nullptr;
    const size_t bxy = sizeof(double) * 2 * (size_t)n_traj, bout = sizeof(double) * QMC_TOY_NOUT * (size_t)n_traj;
    if (cudaMalloc(&d_xy, bxy) != cudaSuccess) return QMC_ERR_OOM;
    if (cudaMalloc(&d_out, bout) != cudaSuccess) { cudaFree(d_xy); return QMC_ERR_OOM; }
    int res = QMC_OK;
    if (cudaMemcpy(d_xy, xy0, bxy, cudaMemcpyHostToDevice) != cudaSuccess) res = QMC_ERR_CUDA;
    if (res == QMC_OK) {
        qmc::launch_toy(toy_dev(p), n_traj, d_xy, d_out, nullptr);
        if (cudaGetLastError() != cudaSuccess || cudaMemcpy(out, d_out, bout, cudaMemcpyDeviceToHost) != cudaSuccess)
            res = QMC_ERR_CUDA;
    }
    cudaFree(d_xy);
    cudaFree(d_out);
    if (res != QMC_OK) return res;
    for (int t = 0; t < n_traj; ++t)
        if (out[QMC_TOY_NOUT * (size_t)t + 6] != 0.0) return QMC_ERR_NOT_PD;
    return QMC_OK;
}
