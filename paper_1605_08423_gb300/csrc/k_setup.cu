// k_setup.cu -- per-configuration tables of the nuclei (once per R).
//
//  * (sin, cos)(pi R_a / L) for the periodised displacements,
//  * exp(i k.R_a) and the proton structure factor rho_p(k) = sum_a Z exp(i k.R_a),
//  * the proton-proton real-space Ewald energy and its gradient, plus the
//    constant self-interaction term -kappa/sqrt(pi) sum_q q^2 over all 2N charges.
// Everything here is FP64.
#include "common.cuh"
#include "kernels.cuh"

namespace qmc {

// The tables that need only R and the cell, in one launch: blocks of 128
// threads take, in order,
//   bKw   blocks: reciprocal weights (4 pi / L^3) exp(-k^2 / 4 kappa^2) / k^2,
//   bPt   blocks: (sin, cos)(pi R / L) and the FP32 copy of R,
//   bEik  blocks: exp(i k.R_a),
//   N     blocks: nucleus a's proton-proton real-space pairs, one thread per
//         partner (its gradient, and its energy into vpp[a]).
// The pair sums are what bounds it (an FP64 erfc, exp and two divisions per
// image): one block per nucleus spreads them over the chip, where one block
// for all of them took 3.9 ms at N = 128 (26 us in this form).
__global__ void __launch_bounds__(128) setup_r_kernel(int N, int nk, int bKw, int bPt, int bEik, double L, double kappa,
                                                      const int4* __restrict__ kvec, const double* __restrict__ R,
                                                      double* kw, float* kw32, double* ptrig64, float* ptrig32,
                                                      float* R32, double2* eikR, float2* eikR32, double* vpp,
                                                      double* dvpp) {
    __shared__ double red[4][32];
    int blk = blockIdx.x;
    if (blk < bKw) {
        const int k = blk * 128 + threadIdx.x;
        if (k >= nk) return;
        const int4 m = kvec[k];
        const double tp = 2.0 * kPi / L;
        const double k2 = tp * tp * (double)(m.x * m.x + m.y * m.y + m.z * m.z);
        const double v = 4.0 * kPi / (L * L * L) * exp(-k2 / (4.0 * kappa * kappa)) / k2;
        kw[k] = v;
        kw32[k] = (float)v;
        return;
    }
    blk -= bKw;
    if (blk < bPt) {
        const int t = blk * 128 + threadIdx.x;
        if (t >= 3 * N) return;
        R32[t] = (float)R[t];
        const int a = t / 3, mu = t % 3;
        double sn, cs;
        sincospi(R[t] / L, &sn, &cs);
        ptrig64[6 * a + mu] = sn; ptrig64[6 * a + 3 + mu] = cs;
        ptrig32[6 * a + mu] = (float)sn; ptrig32[6 * a + 3 + mu] = (float)cs;
        return;
    }
    blk -= bPt;
    if (blk < bEik) {
        const int t = blk * 128 + threadIdx.x;
        if (t >= N * nk) return;
        const int a = t / nk, k = t - a * nk;
        const int4 m = kvec[k];
        const double ph = 2.0 * (m.x * R[3 * a] + m.y * R[3 * a + 1] + m.z * R[3 * a + 2]) / L;
        double sn, cs;
        sincospi(ph, &sn, &cs);
        eikR[t] = make_double2(cs, sn);
        eikR32[t] = make_float2((float)cs, (float)sn);
        return;
    }
    const int a = blk - bEik;
    double v[4] = {0, 0, 0, 0};
    for (int b = threadIdx.x; b < N; b += 128) {
        if (b == a) continue;
        double gr[3];
        v[0] += ewald_real<double>(R[3 * a] - R[3 * b], R[3 * a + 1] - R[3 * b + 1], R[3 * a + 2] - R[3 * b + 2], L,
                                   kappa, gr);
        v[1] += gr[0]; v[2] += gr[1]; v[3] += gr[2];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = block_sum(v[q], red[q]);
    if (threadIdx.x == 0) {
        vpp[a] = 0.5 * v[0];
        dvpp[3 * a] = v[1]; dvpp[3 * a + 1] = v[2]; dvpp[3 * a + 2] = v[3];
    }
}

// What needs the first launch's tables: block 0 sums the proton-proton energy
// (with the self-interaction constant), the others rho_p(k) and, where the
// split measure path runs, the reciprocal-force matrix (below).
// Reciprocal-space force on the nuclei as a matrix acting on the electron
// structure factor of a sample: with rho(k) = rho_p(k) - rho_e(k) = (rr, ri),
//   F_{a,mu} = sum_k 2 Z w_k (2 pi m_mu / L) [ri cos(k.R_a) - rr sin(k.R_a)],
// T is [3N][2 nk] column-major (column 2k multiplies rr(k), 2k + 1 ri(k)).
__global__ void __launch_bounds__(128) setup_sum_kernel(int N, int nk, int bRho, double L, double kappa,
                                                        const int4* __restrict__ kvec, const double* __restrict__ kw,
                                                        const double2* __restrict__ eikR, const double* __restrict__ vpp,
                                                        double2* rho_p, double* vconst, float* T) {
    __shared__ double red[32];
    int blk = blockIdx.x;
    if (blk == 0) {
        double e = 0.0;
        for (int a = threadIdx.x; a < N; a += 128) e += vpp[a];
        e = block_sum(e, red);
        if (threadIdx.x == 0) vconst[0] = e - kappa / sqrt(kPi) * (2.0 * N);
        return;
    }
    blk -= 1;
    if (blk < bRho) {
        const int k = blk * 128 + threadIdx.x;
        if (k >= nk) return;
        double re = 0, im = 0;
#pragma unroll 8
        for (int a = 0; a < N; ++a) {
            const double2 e = eikR[(size_t)a * nk + k];
            re += e.x; im += e.y;
        }
        rho_p[k] = make_double2(re, im);
        return;
    }
    const int t = (blk - bRho) * 128 + threadIdx.x;
    if (t >= 3 * N * nk) return;
    const int k = t / (3 * N), c = t - k * 3 * N, a = c / 3, mu = c - 3 * a;
    const int4 m = kvec[k];
    const double mm = mu == 0 ? m.x : (mu == 1 ? m.y : m.z);
    const double f = 2.0 * kw[k] * (2.0 * kPi / L) * mm;   // proton charge 1
    const double2 e = eikR[(size_t)a * nk + k];
    T[(size_t)(2 * k) * 3 * N + c] = (float)(-f * e.y);
    T[(size_t)(2 * k + 1) * 3 * N + c] = (float)(f * e.x);
}

void launch_setup(int N, double L, double kappa, int nk, const int4* kvec, const double* R, double* kw,
                  double* ptrig64, float* ptrig32, double2* eikR, double2* rho_p, double* vconst, double* dvpp,
                  double* vpp, float* R32, float2* eikR32, float* kw32, float* Trec, cudaStream_t st) {
    const int bKw = (nk + 127) / 128, bPt = (3 * N + 127) / 128, bEik = (N * nk + 127) / 128;
    setup_r_kernel<<<bKw + bPt + bEik + N, 128, 0, st>>>(N, nk, bKw, bPt, bEik, L, kappa, kvec, R, kw, kw32, ptrig64,
                                                         ptrig32, R32, eikR, eikR32, vpp, dvpp);
    const int bRho = (nk + 127) / 128, bRec = Trec ? (3 * N * nk + 127) / 128 : 0;
    setup_sum_kernel<<<1 + bRho + bRec, 128, 0, st>>>(N, nk, bRho, L, kappa, kvec, kw, eikR, vpp, rho_p, vconst, Trec);
}

// Taylor coefficients of the real-space Ewald table (EwTable in common.cuh),
// once per handle: one thread per node.  F_7 from its (all-positive) series
//   F_n(x) = exp(-x) sum_i (2x)^i / ((2n+1)(2n+3)...(2n+2i+1)),
// F_6..F_0 by F_{n-1} = (2x F_n + exp(-x)) / (2n-1); G_0 from erfc and
// G_n = (exp(-x) + (2n-1) G_{n-1}) / 2x: every term positive, no cancellation.
__global__ void ewald_table_kernel(double kappa, double h, double* __restrict__ t) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= 2 * kEwNodes) return;
    const int which = k / kEwNodes, i = k - which * kEwNodes + (which ? kEwFirstB : 0);
    const double x = kappa * kappa * (h * i), ex = exp(-x);
    double f[kEwTerms];
    if (which == 0) {
        double term = 1.0 / (2 * kEwTerms - 1), sum = 0.0;
        for (int j = 1; j < 400 && term > 1e-18 * sum; ++j) {
            sum += term;
            term *= 2.0 * x / (2 * kEwTerms - 1 + 2 * j);
        }
        f[kEwTerms - 1] = ex * sum;
        for (int n = kEwTerms - 1; n > 0; --n) f[n - 1] = (2.0 * x * f[n] + ex) / (2 * n - 1);
    } else {
        const double r = sqrt(x);
        f[0] = 0.88622692545275801365 * erfc(r) / r;   // sqrt(pi) / 2
        for (int n = 1; n < kEwTerms; ++n) f[n] = (ex + (2 * n - 1) * f[n - 1]) / (2.0 * x);
    }
    double c = 1.1283791670955125739 * kappa;          // 2 / sqrt(pi)
    for (int n = 0; n < kEwTerms; ++n) {
        t[(size_t)k * kEwTerms + n] = c * f[n];
        c *= -kappa * kappa / (n + 1);
    }
}

void launch_ewald_table(double kappa, double h, double* t, cudaStream_t st) {
    ewald_table_kernel<<<(2 * kEwNodes + 63) / 64, 64, 0, st>>>(kappa, h, t);
}

}  // namespace qmc
