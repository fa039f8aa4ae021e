// bloch.cuh -- Bloch-summed Gaussians of the twisted boundary conditions, shared by
// the orbital kernel (k_twist.cu) and the FP64 measure kernel (k_measure64.cu).
//
//   chi_{a,g}(r) = sum_n exp(i theta.n) exp(-zeta_g |r - R_a - nL|^2) = exp(i theta.k) s_x s_y s_z,
//   s_mu = sum_m exp(i theta_mu m) exp(-zeta (d_mu - m L)^2),  d = r - R_a - kL, k the nearest image.
// Complex values are double2 (x = real, y = imaginary part).
#pragma once
#include "common.cuh"

namespace qmc {

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cinv(double2 a) {
    const double q = a.x * a.x + a.y * a.y;
    return make_double2(a.x / q, -a.y / q);
}
__device__ __forceinline__ double2 czero() { return make_double2(0.0, 0.0); }
__device__ __forceinline__ double cre(double2 a, double2 b) { return a.x * b.x - a.y * b.y; }   // Re(a b)
__device__ __forceinline__ double2 caxpy(double s, double2 a, double t, double2 b) {             // s a + t b
    return make_double2(fma(s, a.x, t * b.x), fma(s, a.y, t * b.y));
}

// Minimum-image vector d0 of r - R_a and the Bloch phase exp(i sg theta.k) of the
// nearest image k: from the phase table ph [3][2M+1] where k lies in it (positions
// within a box side of each other), else by sincos.
__device__ __forceinline__ double2 bloch_min_image(const double* x, const double* __restrict__ Ra, double L, double iL,
                                                   int M, const double2* __restrict__ ph, const double* __restrict__ th,
                                                   double sg, double d0[3]) {
    const double magic = 6755399441055744.0;   // 1.5 * 2^52
    int k[3];
    double kd[3];
    bool in = true;
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
        const double d = x[mu] - Ra[mu], q = fma(d, iL, magic);
        k[mu] = __double2loint(q);
        kd[mu] = q - magic;
        d0[mu] = fma(-kd[mu], L, d);
        in = in && k[mu] >= -M && k[mu] <= M;
    }
    if (in) {
        const int S = 2 * M + 1;
        double2 p = cmul(cmul(ph[k[0] + M], ph[S + k[1] + M]), ph[2 * S + k[2] + M]);
        p.y *= sg;
        return p;
    }
    double sn, cs;
    sincos(sg * (th[0] * kd[0] + th[1] * kd[1] + th[2] * kd[2]), &sn, &cs);
    return make_double2(cs, sn);
}

// Images beyond the nearest one that a Gaussian of exponent z needs per axis, out of
// the M the handle sums on either side: with |d0| <= L/2 the m-th image on the near
// side (towards which d0 points) has exp(-z u^2) at least exp(-z m (m-1) L^2) below
// the nearest image's, the m-th on the far side exp(-z m^2 L^2); those under exp(-40)
// = 4e-18 are left out.  For M = 1 a diffuse Gaussian keeps all three images, one with
// z L^2 > 40 two.
__device__ __forceinline__ int bloch_near(double z, double L, int M) {
    int m = 1;
    while (m < M && z * L * L * (double)(m * (m + 1)) < 40.0) ++m;
    return m;
}
__device__ __forceinline__ int bloch_far(double z, double L, int M) {
    int m = 0;
    while (m < M && z * L * L * (double)((m + 1) * (m + 1)) < 40.0) ++m;
    return m;
}

// One axis of a Bloch-summed Gaussian at the minimum-image coordinate d0:
// s[q] = d^q s / dx^q for q = 0..ND, with the phases ph[m + M] = exp(i theta_mu m)
// (conjugated when sg < 0, the spin-down twist).  With w = -2 zeta u,
//   g = e^{-zeta u^2}: dg = w g, d2g = (w^2 - 2 zeta) g, d3g = w (w^2 - 6 zeta) g.
template <int ND>
__device__ __forceinline__ void bloch_axis(double d0, double z, double L, int near, int far, int M,
                                           const double2* __restrict__ ph, double sg, double2 s[ND + 1]) {
    {
        const double e = qexp(-z * d0 * d0), w = -2.0 * z * d0;
        s[0] = make_double2(e, 0.0);
        if (ND >= 1) s[1] = make_double2(e * w, 0.0);
        if (ND >= 2) s[2] = make_double2(e * fma(w, w, -2.0 * z), 0.0);
        if (ND >= 3) s[3] = make_double2(e * (w * fma(w, w, -6.0 * z)), 0.0);
    }
    const bool pos = d0 >= 0.0;
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
        const bool up = (side == 0) == pos;            // images m > 0
        const int cnt = side == 0 ? near : far;
        double u = d0;
#pragma unroll 1
        for (int k = 1; k <= cnt; ++k) {
            u += up ? -L : L;
            const double2 p = ph[(up ? k : -k) + M];
            const double e = qexp(-z * u * u), w = -2.0 * z * u;
            const double a = e * p.x, b = e * (p.y * sg);
            s[0].x += a; s[0].y += b;
            if (ND >= 1) { s[1].x = fma(a, w, s[1].x); s[1].y = fma(b, w, s[1].y); }
            if (ND >= 2) {
                const double c = fma(w, w, -2.0 * z);
                s[2].x = fma(a, c, s[2].x); s[2].y = fma(b, c, s[2].y);
            }
            if (ND >= 3) {
                const double c = w * fma(w, w, -6.0 * z);
                s[3].x = fma(a, c, s[3].x); s[3].y = fma(b, c, s[3].y);
            }
        }
    }
}

}  // namespace qmc
