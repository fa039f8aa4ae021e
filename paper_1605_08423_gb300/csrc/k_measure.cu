// k_measure.cu -- local energy and nuclear-force sample of every walker, mixed
// form (FP32 with FP64 where it is needed; the FP64 form's kernel is in
// k_measure64.cu).
//
// One CTA per walker.  From the orbital derivative rows (D = grad phi, Lp =
// lap phi at the current electrons), the inverse G of each spin block and
// the positions it computes
//   E_L = -1/2 sum_i [ l_i - |g_i|^2 + lap_i U + |g_i + grad_i U|^2 ] + V_Ewald
//     g_i = sum_j D_ij G_ji,  l_i = sum_j Lp_ij G_ji
// and, by a hand-written reverse-mode pass (recomputing the basis instead of
// storing it), the derivatives with respect to every nucleus R_a:
//   d ln psi / dR_a = - sum_i sum_{b in a} Z_bi grad chi_b(r_i) - sum_i grad_i u_en(i,a)
//   dE_L / dR_a     =   sum_i sum_{b in a} [ P_bi grad chi_b + Z_bi (H_b grad_i U + 1/2 grad lap chi_b) ]
//                     + sum_i [ (g_i + grad_i U) . H(u_en) + 1/2 grad lap u_en ] + dV/dR_a
//   Z = C G,  P = C (G Y G),  Y_ij = -1/2 Lp_ij - grad_i U . D_ij
// (Hellmann-Feynman term dV/dR plus the Pulay terms through the basis centres
// and the e-n Jastrow).  The force sample f = -dE_L/dR - 2(E_L - E) d ln psi/dR
// is assembled later from the per-walker sums accumulated here:
//   [count, sum E_L, sum E_L^2, sum dlnpsi (3N), sum E_L dlnpsi (3N), sum dE_L (3N)].
// Every reduction is a fixed-order warp or block tree (bitwise reproducible).
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"

namespace qmc {

namespace {

using T = float;   // working precision of this kernel

// Basis rows per tile of the orbital force products where n <= 32 (64 above): with
// 4 x 4 outputs a thread 128 rows occupy all 256 threads, 64 rows only half.
constexpr int kPulayRows = 128;

struct MLayout {
    size_t xs, xt, et, gU, lU, Ui, gi, vv, li, facc, gacc, rhot, red, stage, cmask, uni, total;
    // split: the B x n orbital contractions run in the adjoint kernel, so the
    // spin-block work space only holds Y^T / M1 and G (and no epilogue stage)
    __host__ __device__ MLayout(int N, int n, int nk, int mmax, bool split = false) {
        size_t o = 0;
        auto take = [&](size_t bytes) { size_t r = o; o = (o + bytes + 15) & ~size_t(15); return r; };
        xs = take(sizeof(double) * 3 * N);
        xt = take(sizeof(T) * 3 * N);
        et = take(sizeof(T) * 6 * N);
        gU = take(sizeof(T) * 3 * N);
        lU = take(sizeof(T) * N);
        Ui = take(sizeof(T) * N);
        gi = take(sizeof(T) * 3 * N);
        vv = take(sizeof(T) * 3 * N);
        li = take(sizeof(T) * N);
        facc = take(sizeof(double) * 9 * N);
        gacc = take(sizeof(T) * 9 * N);
        rhot = take(sizeof(V2<T>) * nk);
        red = take(sizeof(double) * 64);
        stage = take(split ? 0 : sizeof(double) * kPulayRows * 6);
        cmask = take(sizeof(unsigned) * (size_t)N * ((N + 31) / 32));
        // phase table e^{i m theta}, m = 0..mmax (negative m by conjugation)
        const size_t etab = sizeof(V2<T>) * (size_t)N * 3 * (mmax + 1);
        int np = 4;
        while (np < n) np *= 2;
        const size_t spin = split ? sizeof(T) * 2 * (size_t)np * (np + 4) : sizeof(T) * (size_t)np * (3 * (np + 4) + (np <= 32 ? kPulayRows : 64) + 4);
        // P1 partials: nparts * N <= 256 rows of 5, and (mixed form, N a
        // multiple of 32) the e-e tiles' rows of 5 per electron and partner block
        const size_t jpart = sizeof(T) * 5 * (256 + (size_t)(N / 32) * N);
        // e-e-n-n Jastrow work space: c [N], S [N][3], 8 warps x 5N per electron in hand
        const size_t j34 = sizeof(T) * (split ? 44 : 84) * (size_t)N;
        size_t u = etab > spin ? etab : spin;
        u = u > j34 ? u : j34;
        uni = take(u > jpart ? u : jpart);
        total = o;
    }
};

// FP32 radial factors of the Pade pair functions in t = rho^2, from one
// reciprocal square root and one reciprocal (FP64: pade_factors):
// f1 = u'/(2 rho),  f2 = (u''/rho^2 - u'/rho^3)/4,
// f3 = (u'''/rho^3 - 3 u''/rho^4 + 3 u'/rho^5)/8.
__device__ __forceinline__ void jas_ee_f32(float t, float b, float& u, float& f1, float& f2) {
    const float ir = rsqrtf(t), r = t * ir, ir2 = ir * ir;
    const float iq = __fdividef(1.0f, 1.0f + b * r), iq2 = iq * iq;
    u = 0.5f * r * iq;
    const float u1 = 0.5f * iq2, u2 = -b * iq2 * iq;
    f1 = 0.5f * u1 * ir;
    f2 = 0.25f * (u2 - u1 * ir) * ir2;
}
__device__ __forceinline__ void jas_ep_f32(float t, float b, float Zj, float& u, float& f1, float& f2, float& f3) {
    const float ir = rsqrtf(t), r = t * ir, ir2 = ir * ir;
    const float iq = __fdividef(1.0f, 1.0f + b * r), iq2 = iq * iq;
    u = -Zj * r * iq;
    const float u1 = -Zj * iq2, u2 = 2.0f * Zj * b * iq2 * iq, u3 = -6.0f * Zj * b * b * iq2 * iq2;
    f1 = 0.5f * u1 * ir;
    f2 = 0.25f * (u2 - u1 * ir) * ir2;
    f3 = 0.125f * (u3 - 3.0f * (u2 - u1 * ir) * ir) * ir2 * ir;
}

// FP32 e-n pair terms of d ln psi / dR and dE_L / dR: g = 2 f1 p, H v = 4 f2 p (p.v) + 2 f1 q o v,
// grad lap u = p o (8 f3 |p|^2 + 8 f2 q + 4 f2 sum q - 2 k^2 f1).
__device__ __forceinline__ void ep_jastrow_f32(const float sd[3], const float cd[3], float ell, float k2, float bep,
                                               float Zj, const float vv[3], float dl[3], float de[3]) {
    float p[3], q[3], s2 = 0.f;
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
        p[mu] = ell * sd[mu] * cd[mu];
        q[mu] = cd[mu] * cd[mu] - sd[mu] * sd[mu];
        s2 += sd[mu] * sd[mu];
    }
    float u, f1, f2, f3;
    jas_ep_f32(ell * ell * s2, bep, Zj, u, f1, f2, f3);
    const float pp = p[0] * p[0] + p[1] * p[1] + p[2] * p[2];
    const float sq = q[0] + q[1] + q[2];
    const float pv = p[0] * vv[0] + p[1] * vv[1] + p[2] * vv[2];
    const float c2 = 2.f * f1, c4 = 4.f * f2;
    const float common = 8.f * f3 * pp + c4 * sq - 2.f * k2 * f1;
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
        dl[mu] = -c2 * p[mu];
        de[mu] = c4 * p[mu] * pv + c2 * q[mu] * vv[mu] + 0.5f * p[mu] * (common + 8.f * f2 * q[mu]);
    }
}

// sin and cos of |x| <= 1/2 in FP64 by their Taylor series (terms to x^15, x^16:
// remainder below 1e-19).
__device__ __forceinline__ void sincos_half(double x, double& sn, double& cs) {
    const double y = x * x;
    double p = fma(y, -7.6471637318198164759e-13, 1.6059043836821614599e-10);   // -1/15!, 1/13!
    p = fma(p, y, -2.5052108385441718775e-08);
    p = fma(p, y, 2.7557319223985890653e-06);
    p = fma(p, y, -1.9841269841269841270e-04);
    p = fma(p, y, 8.3333333333333333333e-03);
    p = fma(p, y, -1.6666666666666666667e-01);
    sn = fma(p * y, x, x);
    double q = fma(y, 4.7794773323873852974e-14, -1.1470745597729724714e-11);   // 1/16!, -1/14!
    q = fma(q, y, 2.0876756987868098979e-09);
    q = fma(q, y, -2.7557319223985890653e-07);
    q = fma(q, y, 2.4801587301587301587e-05);
    q = fma(q, y, -1.3888888888888888889e-03);
    q = fma(q, y, 4.1666666666666666667e-02);
    q = fma(q, y, -0.5);
    cs = fma(q, y, 1.0);
}

// erf(kappa r)/r = kappa 2/sqrt(pi) sum_n (-x)^n / (n! (2n + 1)), x = (kappa r)^2 <= 2/3,
// to n = 15 (remainder below 3e-18), with its derivative in x (below 6e-17), both over
// kappa 2/sqrt(pi).
__device__ __forceinline__ double erf_over_r_series(double x, double& d) {
    constexpr double c[16] = {1.0, -1.0 / 3.0, 1.0 / 10.0, -1.0 / 42.0, 1.0 / 216.0, -1.0 / 1320.0, 1.0 / 9360.0,
                              -1.0 / 75600.0, 1.0 / 685440.0, -1.0 / 6894720.0, 1.0 / 76204800.0, -1.0 / 918086400.0,
                              1.0 / 11975040000.0, -1.0 / 168129561600.0, 1.0 / 2528170444800.0,
                              -1.0 / 40537905408000.0};
    double v = c[15];
    d = 0.0;
#pragma unroll
    for (int n = 14; n >= 0; --n) {
        d = fma(d, x, v);
        v = fma(v, x, c[n]);
    }
    return v;
}

// Close electron-proton pair (mixed form, FP64): the e-n Jastrow terms dl (to
// d ln psi/dR_a) and de (to dE_L/dR_a, given vv = g_i + grad_i U), and the nearest
// image's phi(r) = erfc(kappa r)/r with its gradient, for d = r_i - R_a.  The pairs
// are closer than 0.3 bohr, so short series give the trig and the smooth part
// erf(kappa r)/r: some 180 FP64 operations a pair (450 with the library's sincospi,
// erfc, exp and divisions).  Cells and splittings outside the series' range
// (L < 2.1, kappa > 2.5) take the library calls.
__device__ __forceinline__ void close_pair(const double d[3], double L, double iL, double ell, double kappa, double k2,
                                           double bep, double Zj, const double vv[3], double& v, double g[3],
                                           double dl[3], double de[3]) {
    double m[3], p[3], q[3], s2 = 0, r2 = 0;
    const bool small = ell > 0.66;      // |pi m / L| <= asin(0.3 / ell) < 1/2
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
        m[mu] = d[mu] - L * rint(d[mu] * iL);
        double sn, cs;
        if (small) sincos_half(m[mu] * (kPi * iL), sn, cs);
        else sincospi(m[mu] * iL, &sn, &cs);
        const double ss = sn * sn;
        p[mu] = ell * sn * cs;
        q[mu] = fma(-2.0, ss, 1.0);
        s2 += ss;
        r2 += m[mu] * m[mu];
    }
    double c2, c4, c8;
    pade_factors3(ell * ell * s2, bep, -Zj, c2, c4, c8);
    const double pp = p[0] * p[0] + p[1] * p[1] + p[2] * p[2];
    const double pv = p[0] * vv[0] + p[1] * vv[1] + p[2] * vv[2];
    const double c0 = fma(c4, pv, 0.5 * fma(c8, pp, fma(c4, q[0] + q[1] + q[2], -k2 * c2)));
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
        dl[mu] = -c2 * p[mu];
        de[mu] = fma(p[mu], fma(c4, q[mu], c0), c2 * (q[mu] * vv[mu]));
    }
    const double ir = qrsqrt(r2), x = kappa * kappa * r2;
    double sg;
    if (kappa <= 2.5 && small) {
        const double ck = 1.1283791670955126 * kappa;
        double dx;
        const double e = ck * erf_over_r_series(x, dx);
        v = ir - e;
        sg = -(ir * ir * ir) - 2.0 * ck * kappa * kappa * dx;
    } else {
        const double ec = erfc(kappa * (r2 * ir));
        v = ec * ir;
        sg = -(ec * ir + 1.1283791670955126 * kappa * exp(-x)) * ir * ir;
    }
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) g[mu] = sg * m[mu];
}

// e-e-n-n Jastrow orbital chi_a(r_i) = exp(-zeta |d|^2) of electron trig ei and
// nucleus trig pa with its gradient, Hessian, Laplacian and gradient of the
// Laplacian in the electron coordinate (radial chain of f(t) = exp(-zeta t)).
__device__ __forceinline__ T jas34_orbital(const T* ei, const T* pa, T ell, T zeta, T k2, RadialDerivs<T>& rd) {
    T sd[3], cd[3], t;
    disp_trig(ei, pa, ell, sd, cd, t);
    T p[3], q[3];
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
        p[mu] = ell * sd[mu] * cd[mu];
        q[mu] = cd[mu] * cd[mu] - sd[mu] * sd[mu];
    }
    const T e = qexp(-zeta * t);
    radial_chain(p, q, -zeta * e, zeta * zeta * e, -zeta * zeta * zeta * e, k2, rd);
    return e;
}

// Running sum of FP32 terms to FP64-like accuracy without the FP64 pipe: hi + lo,
// each addition's rounding error kept exactly by Knuth's TwoSum (a conversion and
// an FP64 addition take 32 clocks of an SM per warp, these seven FP32 ones two):
// on 276 configurations of N = 16 to 54 the force terms are FP64 sums' to 1.3e-16, and a
// sample of 1501 walkers, N = 54, takes 0.76 ms where FP64 sums take 0.83.
struct Sum2 {
    float h = 0.f, l = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float t = __fadd_rn(h, x), z = __fsub_rn(t, h);
        l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(t, z)), __fsub_rn(x, z)));
        h = t;
    }
    __device__ __forceinline__ double value() const { return (double)h + (double)l; }
};

// kSplit: the B x n orbital contractions and their basis-derivative epilogue
// are left to the tensor-core adjoint kernel; this kernel then writes what
// that kernel needs: K^T per spin block (kt_out), the electrons' (sin, cos)
// and grad U (eg_out, 9 per electron) and E_L of the sample (elw); the
// reciprocal-space force, a fixed [3N][2 nk] matrix times rho(k), is left to a
// GEMM over all walkers, so the structure factor goes out too (rk_out).
// Three CTAs an SM (80 registers): the phases are latency-bound between barriers.
// Without the bound the unsplit instance took 143 registers, one CTA an SM:
// 3.14 ms for 4096 walkers of N = 64, now 1.53 ms.
template <bool kSplit>
__global__ void __launch_bounds__(256, 3) measure_kernel(SysView<T> s, int mmax, int ntask,
                                                      const int4* __restrict__ ktask, const T* __restrict__ kint,
                                                      const double* __restrict__ X,
                                                      const T* __restrict__ D, T* LpY,
                                                      const T* __restrict__ Gt, const double* __restrict__ logdet,
                                                      double* __restrict__ acc, double* __restrict__ out_el,
                                                      double* __restrict__ out_lnpsi, double* __restrict__ out_dl,
                                                      double* __restrict__ out_de, float* __restrict__ kt_out,
                                                      float* __restrict__ eg_out, double* __restrict__ elw,
                                                      float* __restrict__ rk_out) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int N = s.N, n = s.n, G = s.G, nk = s.nk;
    const MLayout lay(N, n, nk, mmax, kSplit);
    double* xs = (double*)(sm + lay.xs);
    T* xt = (T*)(sm + lay.xt);
    T* et = (T*)(sm + lay.et);
    T* gU = (T*)(sm + lay.gU);
    T* lU = (T*)(sm + lay.lU);
    T* Ui = (T*)(sm + lay.Ui);
    T* gi = (T*)(sm + lay.gi);
    T* vvs = (T*)(sm + lay.vv);
    T* li = (T*)(sm + lay.li);
    double* f_dl = (double*)(sm + lay.facc);
    double* f_de = f_dl + 3 * N;
    double* f_dv = f_de + 3 * N;
    // FP32-phase partials per nucleus component (one writer each; FP64 sums
    // above hold the FP64 close-pair terms and the SIMT Pulay epilogue)
    T* g_dl = (T*)(sm + lay.gacc);
    T* g_de = g_dl + 3 * N;
    T* g_dv = g_de + 3 * N;
    V2<T>* rhot = (V2<T>*)(sm + lay.rhot);
    double* red = (double*)(sm + lay.red);
    double* stage = (double*)(sm + lay.stage);
    unsigned* cmask = (unsigned*)(sm + lay.cmask);
    unsigned char* uni = sm + lay.uni;

    const int w = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const double L = s.L;
    const T ell = (T)s.ell, bee = (T)s.b_ee, bep = (T)s.b_ep, Zj = (T)s.Zj, kap = (T)s.kappa;
    const double iL = s.iL;
    const T twopiL = T(2.0 * kPi * iL), k2 = twopiL * twopiL;
    const double Zn = 1.0;  // proton charge

    // ---- P0: positions and their (sin, cos)(pi x / L)
    for (int idx = tid; idx < 3 * N; idx += nt) {
        const double x = X[(size_t)w * 3 * N + idx];
        xs[idx] = x;
        xt[idx] = (T)x;
        T sn, cs;
        qsincospi((T)(x * iL), &sn, &cs);
        et[6 * (idx / 3) + idx % 3] = sn;
        et[6 * (idx / 3) + 3 + idx % 3] = cs;
    }
    for (int idx = tid; idx < 9 * N; idx += nt) { f_dl[idx] = 0.0; g_dl[idx] = T(0); }
    for (int idx = tid; idx < N * ((N + 31) / 32); idx += nt) cmask[idx] = 0u;
    __syncthreads();

    // ---- P1: Jastrow gradient / Laplacian per electron, U partial sums.  The
    // partner range is split into nparts slices so that every thread works;
    // the slices are summed in order afterwards.
    const int nparts = nt >= N ? nt / N : 1;
    T* jpart = (T*)uni;
    // Mixed form with N a multiple of 32: each e-e pair is evaluated once, in
    // 32 x 32 tiles of electron blocks (I, J), I <= J, one warp per tile: lane
    // l holds electron 32 I + l and at step k meets electron 32 J + (l + k) mod
    // 32; its row sums stay in the lane and the partner's column sums move one
    // lane per step (shuffle), so that after the tile lane l holds electron
    // 32 J + l's.  A diagonal tile takes steps 1..16 (step 16 on lanes 0-15
    // only).  Each (electron, partner block) has one slot of 5; the slots are
    // summed in block order with the e-n slices below.
    const bool ee_tiles = (N & 31) == 0 && N >= 64;
    T* eepart = jpart + (size_t)5 * 256;   // [N / 32][N][5]
    for (int tt = tid; tt < nparts * N; tt += nt) {
        const int i = tt % N, pi = tt / N;
        const int j0 = (N * pi) / nparts, j1 = (N * (pi + 1)) / nparts;
        T g[3] = {0, 0, 0}, lp = 0, ui = 0;
        const T* ei = et + 6 * i;
        for (int j = ee_tiles ? j1 : j0; j < j1; ++j) {
            if (j == i) continue;
            T sd[3], cd[3], t;
            disp_trig(ei, et + 6 * j, ell, sd, cd, t);
            T u, f1, f2;
            jas_ee_f32(t, bee, u, f1, f2);
            T pp = 0, sq = 0;
#pragma unroll
            for (int mu = 0; mu < 3; ++mu) {
                const T p = ell * sd[mu] * cd[mu];
                g[mu] += T(2) * f1 * p;
                pp += p * p; sq += cd[mu] * cd[mu] - sd[mu] * sd[mu];
            }
            lp += T(4) * f2 * pp + T(2) * f1 * sq;
            if (j > i) ui += u;
        }
        for (int a = j0; a < j1; ++a) {
            T sd[3], cd[3], t;
            disp_trig(ei, s.ptrig + 6 * a, ell, sd, cd, t);
            T u, f1, f2, f3;
            jas_ep_f32(t, bep, Zj, u, f1, f2, f3);
            T pp = 0, sq = 0;
#pragma unroll
            for (int mu = 0; mu < 3; ++mu) {
                const T p = ell * sd[mu] * cd[mu];
                g[mu] += T(2) * f1 * p;
                pp += p * p; sq += cd[mu] * cd[mu] - sd[mu] * sd[mu];
            }
            lp += T(4) * f2 * pp + T(2) * f1 * sq;
            ui += u;
        }
        T* o = jpart + ((size_t)pi * N + i) * 5;
        o[0] = g[0]; o[1] = g[1]; o[2] = g[2]; o[3] = lp; o[4] = ui;
    }
    if (ee_tiles) {
        const int nb = N >> 5, noff = nb * (nb - 1) / 2, ntiles = noff + nb;
        for (int tile = warp; tile < ntiles; tile += nw) {
            int I = 0, J = 0;
            if (tile < noff) {   // off-diagonal tiles, I < J in row-major order
                int r = tile;
                while (r >= nb - 1 - I) { r -= nb - 1 - I; ++I; }
                J = I + 1 + r;
            } else {
                I = J = tile - noff;
            }
            const bool diag = I == J;
            const int i = 32 * I + lane;
            float ei[6];
#pragma unroll
            for (int c = 0; c < 6; ++c) ei[c] = et[6 * i + c];
            float rg[3] = {0.f, 0.f, 0.f}, rl = 0.f, ru = 0.f, cg[3] = {0.f, 0.f, 0.f}, cl = 0.f;
            const int k0 = diag ? 1 : 0, k1 = diag ? 17 : 32;
            for (int k = k0; k < k1; ++k) {
                if (!diag || k < 16 || lane < 16) {
                    const int j = 32 * J + ((lane + k) & 31);
                    float sd[3], cd[3], t;
                    disp_trig(ei, et + 6 * j, ell, sd, cd, t);
                    float u, f1, f2;
                    jas_ee_f32(t, bee, u, f1, f2);
                    float pp = 0.f, sq = 0.f;
#pragma unroll
                    for (int mu = 0; mu < 3; ++mu) {
                        const float pm = ell * sd[mu] * cd[mu], gm = 2.f * f1 * pm;
                        rg[mu] += gm;
                        cg[mu] -= gm;   // p is odd under the exchange of the pair
                        pp += pm * pm;
                        sq += cd[mu] * cd[mu] - sd[mu] * sd[mu];
                    }
                    const float lpv = 4.f * f2 * pp + 2.f * f1 * sq;
                    rl += lpv;
                    cl += lpv;
                    ru += u;
                }
                // the column sums move to the lane that meets their electron next
                const int src = (lane + 1) & 31;
#pragma unroll
                for (int mu = 0; mu < 3; ++mu) cg[mu] = __shfl_sync(0xffffffffu, cg[mu], src);
                cl = __shfl_sync(0xffffffffu, cl, src);
            }
            if (diag) {   // lane l holds column (l + 17) mod 32: column l's come from lane (l + 15) mod 32
                const int src = (lane + 15) & 31;
#pragma unroll
                for (int mu = 0; mu < 3; ++mu) cg[mu] = __shfl_sync(0xffffffffu, cg[mu], src);
                cl = __shfl_sync(0xffffffffu, cl, src);
                T* o = eepart + ((size_t)I * N + i) * 5;
                o[0] = rg[0] + cg[0]; o[1] = rg[1] + cg[1]; o[2] = rg[2] + cg[2]; o[3] = rl + cl; o[4] = ru;
            } else {
                T* o = eepart + ((size_t)J * N + i) * 5;
                o[0] = rg[0]; o[1] = rg[1]; o[2] = rg[2]; o[3] = rl; o[4] = ru;
                T* oc = eepart + ((size_t)I * N + 32 * J + lane) * 5;
                oc[0] = cg[0]; oc[1] = cg[1]; oc[2] = cg[2]; oc[3] = cl; oc[4] = 0.f;
            }
        }
    }
    __syncthreads();
    for (int i = tid; i < N; i += nt) {
        T v[5] = {0, 0, 0, 0, 0};
        for (int pi = 0; pi < nparts; ++pi)
#pragma unroll
            for (int c = 0; c < 5; ++c) v[c] += jpart[((size_t)pi * N + i) * 5 + c];
        if (ee_tiles)
            for (int pb = 0; pb < (N >> 5); ++pb)
#pragma unroll
                for (int c = 0; c < 5; ++c) v[c] += eepart[((size_t)pb * N + i) * 5 + c];
        gU[3 * i] = v[0]; gU[3 * i + 1] = v[1]; gU[3 * i + 2] = v[2];
        lU[i] = v[3]; Ui[i] = v[4];
    }
    __syncthreads();

    // ---- P2b (with the e-e-n-n Jastrow term):
    //   U34 = sum_{i<j} chi_i^T F chi_j = 1/2 sum_i chi_i . w_i,  w_i = F (c - chi_i),  c = sum_j chi_j,
    //   grad_i U34 = sum_a grad chi_a(r_i) w_ia,  lap_i U34 = sum_a lap chi_a(r_i) w_ia,
    // added to grad U, lap U and the per-electron U sums.  c and S_a = sum_j grad chi_a(r_j)
    // stay in the work space for the force terms after P3.  The N^3 sums over b are bound
    // by their loads, so a warp takes several electrons at once: an element of F (global)
    // and one vector of shared memory serve four (here) or two (P3b) of them.
    T* j34c = (T*)uni;               // [N]
    T* j34S = j34c + N;              // [N][3]
    T* j34w = j34S + 3 * N;          // per warp: here c - chi_i of up to four electrons; P3b below
    if (s.fjt) {
        const T zj = (T)s.zeta_j;
        // c and S, the electrons in nparts slices (partials in the warps' work space), summed in order
        for (int tt = tid; tt < nparts * N; tt += nt) {
            const int a = tt % N, pi = tt / N, j0 = (N * pi) / nparts, j1 = (N * (pi + 1)) / nparts;
            T c = 0, g[3] = {0, 0, 0};
            for (int j = j0; j < j1; ++j) {
                RadialDerivs<T> rd;
                c += jas34_orbital(et + 6 * j, s.ptrig + 6 * a, ell, zj, k2, rd);
                for (int mu = 0; mu < 3; ++mu) g[mu] += rd.g[mu];
            }
            T* o = j34w + 4 * (size_t)tt;
            o[0] = c; o[1] = g[0]; o[2] = g[1]; o[3] = g[2];
        }
        __syncthreads();
        for (int idx = tid; idx < 4 * N; idx += nt) {
            T v = 0;
            for (int pi = 0; pi < nparts; ++pi) v += j34w[4 * (size_t)pi * N + idx];
            if (idx & 3) j34S[3 * (idx >> 2) + (idx & 3) - 1] = v;
            else j34c[idx >> 2] = v;
        }
        __syncthreads();
        float4* d4 = (float4*)(j34w + (size_t)warp * 4 * N);     // c_b - chi_b(r_i) of four electrons
        for (int i0 = 4 * warp; i0 < N; i0 += 4 * nw) {
            const int ne = N - i0 < 4 ? N - i0 : 4;
            for (int b = lane; b < N; b += 32) {
                T d[4] = {0, 0, 0, 0};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (e < ne) {
                        T sd[3], cd[3], t;
                        disp_trig(et + 6 * (i0 + e), s.ptrig + 6 * b, ell, sd, cd, t);
                        d[e] = j34c[b] - qexp(-zj * t);
                    }
                d4[b] = make_float4(d[0], d[1], d[2], d[3]);
            }
            __syncwarp();
            T acc[4][5] = {};
            for (int a = lane; a < N; a += 32) {
                const T* fa = s.fjt + a;   // column a = row a (f symmetric): coalesced over lanes
                T wv[4] = {0, 0, 0, 0};
#pragma unroll 4
                for (int b = 0; b < N; ++b) {
                    const T f = fa[(size_t)b * N];
                    const float4 d = d4[b];
                    wv[0] += f * d.x; wv[1] += f * d.y; wv[2] += f * d.z; wv[3] += f * d.w;
                }
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (e < ne) {
                        RadialDerivs<T> rd;
                        const T chi = jas34_orbital(et + 6 * (i0 + e), s.ptrig + 6 * a, ell, zj, k2, rd);
                        for (int mu = 0; mu < 3; ++mu) acc[e][mu] += rd.g[mu] * wv[e];
                        acc[e][3] += rd.lap * wv[e];
                        acc[e][4] += chi * wv[e];
                    }
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (e < ne) {
#pragma unroll
                    for (int c = 0; c < 5; ++c) acc[e][c] = warp_sum(acc[e][c]);
                    if (lane == 0) {
                        const int i = i0 + e;
                        for (int mu = 0; mu < 3; ++mu) gU[3 * i + mu] += acc[e][mu];
                        lU[i] += acc[e][3];
                        Ui[i] += T(0.5) * acc[e][4];
                    }
                }
            __syncwarp();
        }
        __syncthreads();
    }

    // ---- P2: g_i = sum_j D_ij G_ji, l_i = sum_j Lp_ij G_ji (warp per electron,
    // lanes over the orbitals: coalesced rows of D, Lp and G^T)
    // Two electrons at a time: twice the loads in flight, and one packed sum.  The
    // same pass over D and Lp forms Y_ij = -1/2 Lp_ij - grad_i U . D_ij for the
    // orbital force terms, which go into Lp's place (P6 read D and Lp once more
    // before: 4 n values an electron from memory where it now reads n).
    for (int i0 = warp; i0 < N; i0 += 2 * nw) {
        T v[8] = {}, r[2][2][5];                 // [electron][j = lane, lane + 32]: G, D (3), Lp
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int i = i0 + e * nw, sp = i / n, il = i - sp * n;
            const T* grow = Gt + (((size_t)w * 2 + sp) * n + il) * n;
            const T* drow = D + ((size_t)w * N + i) * 3 * n;
            const T* lrow = LpY + ((size_t)w * N + i) * n;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = lane + 32 * h;
                const bool on = i < N && j < n;
                r[e][h][0] = on ? grow[j] : T(0);
                r[e][h][1] = on ? drow[j] : T(0);
                r[e][h][2] = on ? drow[n + j] : T(0);
                r[e][h][3] = on ? drow[2 * n + j] : T(0);
                r[e][h][4] = on ? lrow[j] : T(0);
            }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int i = i0 + e * nw;
            if (i >= N) continue;
            T* lrow = LpY + ((size_t)w * N + i) * n;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = lane + 32 * h;
                const T gj = r[e][h][0], dx = r[e][h][1], dy = r[e][h][2], dz = r[e][h][3], lp = r[e][h][4];
                v[4 * e] += dx * gj; v[4 * e + 1] += dy * gj; v[4 * e + 2] += dz * gj;
                v[4 * e + 3] += lp * gj;
                if (j < n) lrow[j] = T(-0.5) * lp - (gU[3 * i] * dx + gU[3 * i + 1] * dy + gU[3 * i + 2] * dz);
            }
        }
        const T x = warp_sum8(v, lane);
        const int q = lane >> 2, i = i0 + (q >> 2) * nw, c = q & 3;
        if ((lane & 3) == 0 && i < N) {
            if (c < 3) gi[3 * i + c] = x;
            else li[i] = x;
        }
    }
    __syncthreads();

    // ---- P3: kinetic energy and U
    double kin_p = 0.0, u_p = 0.0;
    for (int i = tid; i < N; i += nt) {
        T g2 = 0, t2 = 0;
#pragma unroll
        for (int mu = 0; mu < 3; ++mu) {
            const T g = gi[3 * i + mu], t = g + gU[3 * i + mu];
            g2 += g * g; t2 += t * t;
            vvs[3 * i + mu] = t;     // grad_i ln psi, for the e-n pair terms
        }
        kin_p += (double)(li[i] - g2 + lU[i] + t2);
        u_p += (double)Ui[i];
    }
    const double kin = block_sum(kin_p, red);
    const double Utot = block_sum(u_p, red + 32);

    // ---- P3b (with the e-e-n-n Jastrow term): its terms of d ln psi / dR_a
    // and dE_L / dR_a.  With s_a^(i) = S_a - grad chi_a(r_i), v_ia = sum_b grad chi_b(r_i) f_ba,
    // lam_ia = sum_b lap chi_b(r_i) f_ba and vv_i = g_i + grad_i U:
    //   dlnpsi/dR_a += -sum_i grad chi_a(r_i) w_ia
    //   dE_L/dR_a   += sum_i [ 1/2 (grad lap chi_a(r_i) w_ia + lam_ia s_a^(i))
    //                          + (Hess chi_a(r_i) vv_i) w_ia + (vv_i . v_ia) s_a^(i) ]
    // (the R_a-derivative of -1/2 sum_i [lap_i U34 + 2 vv_i . grad_i U34]).
    if (s.fjt) {
        constexpr int EW = kSplit ? 1 : 2;   // electrons a warp has in hand (shared memory: the split form keeps 3 CTAs)
        const T zj = (T)s.zeta_j;
        // per warp and electron: (grad chi_b, lap chi_b) [N], c_b - chi_b [N]
        float4* gl4 = (float4*)(j34w + (size_t)warp * 5 * EW * N);
        T* df = (T*)(gl4 + EW * N);
        for (int ac = 0; ac < N; ac += 32) {     // a lane's nucleus keeps its sums over the warp's electrons
            const int a = ac + lane < N ? ac + lane : N - 1;
            Sum2 dl[3], de[3];
            for (int i0 = EW * warp; i0 < N; i0 += EW * nw) {
                __syncwarp();
                for (int b = lane; b < N; b += 32)
#pragma unroll
                    for (int e = 0; e < EW; ++e) {
                        const int i = i0 + e < N ? i0 + e : N - 1;
                        RadialDerivs<T> rd;
                        df[e * N + b] = j34c[b] - jas34_orbital(et + 6 * i, s.ptrig + 6 * b, ell, zj, k2, rd);
                        gl4[e * N + b] = make_float4(rd.g[0], rd.g[1], rd.g[2], rd.lap);
                    }
                __syncwarp();
                const T* fa = s.fjt + a;   // column a = row a (f symmetric): coalesced over lanes
                T wv[EW] = {}, v[EW][4] = {};
#pragma unroll 2
                for (int b = 0; b < N; ++b) {
                    const T f = fa[(size_t)b * N];
#pragma unroll
                    for (int e = 0; e < EW; ++e) {
                        const float4 q = gl4[e * N + b];
                        wv[e] += f * df[e * N + b];
                        v[e][0] += q.x * f; v[e][1] += q.y * f; v[e][2] += q.z * f; v[e][3] += q.w * f;
                    }
                }
#pragma unroll
                for (int e = 0; e < EW; ++e) {
                    const int i = i0 + e;
                    if (i >= N) continue;
                    RadialDerivs<T> rd;
                    jas34_orbital(et + 6 * i, s.ptrig + 6 * a, ell, zj, k2, rd);
                    T vv[3], hv[3];
                    for (int mu = 0; mu < 3; ++mu) vv[mu] = vvs[3 * i + mu];
                    hess_mul(rd.h, vv, hv);
                    const T vvv = vv[0] * v[e][0] + vv[1] * v[e][1] + vv[2] * v[e][2];
#pragma unroll
                    for (int mu = 0; mu < 3; ++mu) {
                        const T sa = j34S[3 * a + mu] - rd.g[mu];
                        dl[mu].add(-rd.g[mu] * wv[e]);
                        de[mu].add(T(0.5) * (rd.tl[mu] * wv[e] + v[e][3] * sa) + hv[mu] * wv[e] + vvv * sa);
                    }
                }
            }
            for (int q = 0; q < nw; ++q) {       // the warps' sums in order
                if (q == warp && ac + lane < N)
#pragma unroll
                    for (int mu = 0; mu < 3; ++mu) {
                        f_dl[3 * a + mu] += dl[mu].value();
                        f_de[3 * a + mu] += de[mu].value();
                    }
                __syncthreads();
            }
        }
    }

    // ---- P4a: electron-electron real-space Ewald
    double vee_p = 0.0;
    const T Lt = (T)L;
    const float iLt = 1.f / (float)Lt, rc2 = kRealCut2Mixed * (float)Lt * (float)Lt;
    const bool fast = kap * Lt >= kImageKLMin && kap * Lt <= kImageKLMax;
    // balanced cyclic pairing: electron i with i+d (mod N), d = 1..N/2 (d = N/2 only for i < N/2),
    // the distance range split into nparts slices
    for (int tt = tid; tt < nparts * N; tt += nt) {
        const int i = tt % N, pi = tt / N, half = N / 2;
        const int d0 = 1 + (half * pi) / nparts, d1 = 1 + (half * (pi + 1)) / nparts;
        T v = 0;
        for (int d = d0; d < d1; ++d) {
            const bool skip = 2 * d == N && i >= half;
            const int j = i + d < N ? i + d : i + d - N;      // (i + d) mod N, d < N
            if (skip) continue;
            v += ewald_real_cut<false>(xt[3 * i] - xt[3 * j], xt[3 * i + 1] - xt[3 * j + 1],
                                       xt[3 * i + 2] - xt[3 * j + 2], false, fast, Lt, iLt, rc2, kap, nullptr);
        }
        vee_p += (double)v;
    }
    // ---- P4b: electron-proton pairs (warp per proton, lanes over electrons): the
    // real-space Ewald energy and its R-gradient (Hellmann-Feynman) together with
    // the e-n Jastrow terms of d ln psi/dR and dE_L/dR.  Pairs
    // closer than 0.3 bohr are only flagged here and evaluated afterwards in FP64
    // (one thread per proton, electrons in increasing order): there the 1/r^2
    // Coulomb force and the 1/r^2 part of grad lap u_en cancel (cusp
    // condition), and FP32 rounding of either term would survive the
    // cancellation.  Deferring them keeps FP64 off the common path.
    double vep_p = 0.0;
    T vep_t = 0;
    const int nwords = (N + 31) / 32;
    for (int a = warp; a < N; a += nw) {
        T v = 0, gv[3] = {0, 0, 0}, dl[3] = {0, 0, 0}, de[3] = {0, 0, 0};
        // the nucleus' trig values and position stay in registers over its electrons
        T pa[6], ra[3];
#pragma unroll
        for (int c = 0; c < 6; ++c) pa[c] = s.ptrig[6 * a + c];
#pragma unroll
        for (int c = 0; c < 3; ++c) ra[c] = s.RT[3 * a + c];
        for (int i = lane; i < N; i += 32) {
            T sd[3], cd[3], t;
            disp_trig(et + 6 * i, pa, ell, sd, cd, t);
            const bool close = t < T(0.09);
            if (close) atomicOr(&cmask[a * nwords + (i >> 5)], 1u << (i & 31));
            // Jastrow terms unless close; the Ewald images inside the FP32-level
            // cutoff (a close pair's nearest image is done in FP64)
            if (!close) {
                T vv[3], pl[3], pe[3];
                for (int mu = 0; mu < 3; ++mu) vv[mu] = vvs[3 * i + mu];
                ep_jastrow_f32(sd, cd, ell, k2, bep, Zj, vv, pl, pe);
                for (int mu = 0; mu < 3; ++mu) { dl[mu] += pl[mu]; de[mu] += pe[mu]; }
            }
            v += ewald_real_cut<true>(xt[3 * i] - ra[0], xt[3 * i + 1] - ra[1], xt[3 * i + 2] - ra[2], close, fast, Lt,
                                      iLt, rc2, kap, gv);
        }
        T r[8] = {v, gv[0], gv[1], gv[2], dl[0], dl[1], dl[2], de[0]};
        const T x = warp_sum8(r, lane), d1 = warp_sum(de[1]), d2 = warp_sum(de[2]);
        const int q = lane >> 2;
        if ((lane & 3) == 0) {   // FP32 partials; FP64 only where the sample is accumulated
            if (q == 0) {
                vep_t += -(T)Zn * x;
                g_de[3 * a + 1] = d1;
                g_de[3 * a + 2] = d2;
            } else if (q < 4) {
                g_dv[3 * a + q - 1] = (T)Zn * x;
            } else if (q < 7) {
                g_dl[3 * a + q - 4] = x;
            } else {
                g_de[3 * a] = x;
            }
        }
    }
    {
        // Close pairs in FP64, one thread per pair: the e-n Jastrow terms and
        // the nearest-image real-space Coulomb term (the pair's other images
        // were summed in FP32 above).  Pairs are numbered nucleus by nucleus,
        // electrons in increasing order; each nucleus sums its pairs' results
        // in that order, so the sums do not depend on the thread count.
        int* coff = (int*)uni;                                       // [N + 1] pair offsets
        double* slot = (double*)(uni + (((size_t)(N + 1) * sizeof(int) + 15) & ~size_t(15)));
        const size_t uni_bytes = lay.total - lay.uni;
        const int CH = (int)((uni_bytes - ((size_t)(slot) - (size_t)uni)) / (10 * sizeof(double)));
        __syncthreads();
        if (warp == 0) {   // exclusive scan of the per-nucleus counts
            const int per = (N + 31) / 32, a0 = lane * per;
            int loc = 0;
            for (int a = a0; a < a0 + per && a < N; ++a)
                for (int wd = 0; wd < nwords; ++wd) loc += __popc(cmask[a * nwords + wd]);
            int inc = loc;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            int run = inc - loc;
            for (int a = a0; a < a0 + per && a < N; ++a) {
                coff[a] = run;
                for (int wd = 0; wd < nwords; ++wd) run += __popc(cmask[a * nwords + wd]);
            }
            if (lane == 31) coff[N] = inc;
        }
        __syncthreads();
        const int total = coff[N];
        __syncthreads();   // read by every thread before the phase table below takes coff's place (no pair: no other barrier)
        const double k2d = (2.0 * kPi * iL) * (2.0 * kPi * iL);
        for (int base = 0; base < total; base += CH) {
            const int end = base + CH < total ? base + CH : total;
            for (int t = base + tid; t < end; t += nt) {
                int lo = 0, hi = N;   // nucleus: coff[a] <= t < coff[a + 1]
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (coff[mid] <= t) lo = mid; else hi = mid;
                }
                const int a = lo;
                int k = t - coff[a], i = 0;
                for (int wd = 0; wd < nwords; ++wd) {
                    const unsigned m = cmask[a * nwords + wd];
                    const int c = __popc(m);
                    if (k < c) { i = wd * 32 + nth_set_bit(m, k); break; }
                    k -= c;
                }
                const double dx = xs[3 * i] - s.R[3 * a], dy = xs[3 * i + 1] - s.R[3 * a + 1],
                             dz = xs[3 * i + 2] - s.R[3 * a + 2];
                const double dd[3] = {dx, dy, dz};
                double vv[3], pl[3], pe[3], pv, pg[3];
                for (int mu = 0; mu < 3; ++mu) vv[mu] = (double)gi[3 * i + mu] + (double)gU[3 * i + mu];
                close_pair(dd, L, iL, s.ell, s.kappa, k2d, s.b_ep, s.Zj, vv, pv, pg, pl, pe);
                double* o = slot + (size_t)(t - base) * 10;
                o[0] = pv;
                o[1] = pg[0]; o[2] = pg[1]; o[3] = pg[2];
                for (int mu = 0; mu < 3; ++mu) { o[4 + mu] = pl[mu]; o[7 + mu] = pe[mu]; }
            }
            __syncthreads();
            for (int a = tid; a < N; a += nt) {
                const int lo = coff[a] > base ? coff[a] : base, hi = coff[a + 1] < end ? coff[a + 1] : end;
                if (lo >= hi) continue;
                double vC = 0, gC[3] = {0, 0, 0}, dlC[3] = {0, 0, 0}, deC[3] = {0, 0, 0};
                for (int t = lo; t < hi; ++t) {
                    const double* o = slot + (size_t)(t - base) * 10;
                    vC += o[0];
                    for (int mu = 0; mu < 3; ++mu) { gC[mu] += o[1 + mu]; dlC[mu] += o[4 + mu]; deC[mu] += o[7 + mu]; }
                }
                vep_p += -Zn * vC;
                for (int mu = 0; mu < 3; ++mu) {
                    f_dv[3 * a + mu] += Zn * gC[mu];
                    f_dl[3 * a + mu] += dlC[mu];
                    f_de[3 * a + mu] += deC[mu];
                }
            }
            __syncthreads();
        }
    }
    // ---- P4c: reciprocal space: electron structure factor from per-electron phase tables
    V2<T>* etab = (V2<T>*)uni;
    const int nm = mmax + 1;   // m = 0..mmax; e^{-i m theta} = conj(e^{i m theta})
    for (int idx = tid; idx < 3 * N; idx += nt) {
        T sn, cs;
        qsincospi((T)(2.0 * iL) * xt[idx], &sn, &cs);
        V2<T>* e = etab + (size_t)idx * nm;
        V2<T> cur{T(1), T(0)};
        e[0] = cur;
        for (int m = 1; m <= mmax; ++m) {
            cur = V2<T>{cur.x * cs - cur.y * sn, cur.x * sn + cur.y * cs};
            e[m] = cur;
        }
    }
    __syncthreads();
    double vrec_p = 0.0;
    T vrec_t = 0;
    // A task is two |m_z| of one (m_x, m_y): with ab the x y phase and c the z
    // phase, the four sums of ab.x c.x, ab.y c.y, ab.x c.y, ab.y c.x give rho at
    // both signs of m_z, 12 operations an electron for four vectors (32 one by one).
    for (int tk = tid; tk < ntask; tk += nt) {
        const int4 m = ktask[tk];                 // m_x >= 0, m_y, first |m_z|, index of (m_x, m_y, 0)
        const int my = m.y < 0 ? -m.y : m.y, z1 = m.z + 1 <= mmax ? m.z + 1 : mmax;
        const T sy = m.y < 0 ? T(-1) : T(1);
        T q[2][4] = {};
        for (int i = 0; i < N; ++i) {
            const V2<T>* e = etab + (size_t)3 * i * nm;
            const V2<T> a = e[m.x], b = e[nm + my], c0 = e[2 * nm + m.z], c1 = e[2 * nm + z1];
            const T by = sy * b.y;
            const T x = a.x * b.x - a.y * by, y = a.x * by + a.y * b.x;
            q[0][0] += x * c0.x; q[0][1] += y * c0.y; q[0][2] += x * c0.y; q[0][3] += y * c0.x;
            q[1][0] += x * c1.x; q[1][1] += y * c1.y; q[1][2] += x * c1.y; q[1][3] += y * c1.x;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int mz = m.z + h;
            if (m.x * m.x + m.y * m.y + mz * mz > mmax * mmax) continue;
#pragma unroll
            for (int sg = 0; sg < 2; ++sg) {      // +m_z, -m_z
                if (mz == 0 && (sg || (m.x == 0 && m.y == 0))) continue;
                if (sg && m.x == 0 && m.y == 0) continue;
                const int k = m.w + (sg ? -mz : mz);
                const T re = sg ? q[h][0] + q[h][1] : q[h][0] - q[h][1];
                const T im = sg ? q[h][3] - q[h][2] : q[h][3] + q[h][2];
                const double2 rp = s.rho_p[k];
                const T rr = (T)rp.x - re, ri = (T)rp.y - im;   // electrons carry -1
                const T kw = s.kwt[k];
                if constexpr (!kSplit) {          // proton charge 1
                    const T f = T(2) * kw * twopiL;
                    rhot[k] = V2<T>{f * rr, f * ri};
                } else {
                    rk_out[(size_t)w * 2 * nk + 2 * k] = (float)rr;
                    rk_out[(size_t)w * 2 * nk + 2 * k + 1] = (float)ri;
                }
                vrec_t += kw * (rr * rr + ri * ri);
            }
        }
    }
    vrec_p += (double)vrec_t;
    __syncthreads();
    // ---- P4d: reciprocal-space force on the protons (warp per proton; the
    // split path leaves it to the GEMM)
    if constexpr (!kSplit) {
        // four protons at a time share the loads of rho(k) (scaled by 2 w_k 2 pi / L
        // above) and of the integer vectors
        for (int a0 = 4 * warp; a0 < N; a0 += 4 * nw) {
            T gx[4] = {}, gy[4] = {}, gz[4] = {};
#pragma unroll 2
            for (int k = lane; k < nk; k += 32) {
                const V2<T> rd = rhot[k];
                const T mx = kint[k], my = kint[nk + k], mz = kint[2 * nk + k];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int a = a0 + q < N ? a0 + q : N - 1;
                    const V2<T> e = s.eikRt[(size_t)a * nk + k];
                    const T c = rd.y * e.x - rd.x * e.y;
                    gx[q] += c * mx; gy[q] += c * my; gz[q] += c * mz;
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                gx[q] = warp_sum(gx[q]); gy[q] = warp_sum(gy[q]); gz[q] = warp_sum(gz[q]);
                if (lane == 0 && a0 + q < N) {
                    const int a = a0 + q;
                    g_dv[3 * a] += gx[q]; g_dv[3 * a + 1] += gy[q]; g_dv[3 * a + 2] += gz[q];
                }
            }
        }
    }
    vep_p += (double)vep_t;
    const double vee = block_sum(vee_p, red);
    const double vep = block_sum(vep_p, red + 32);
    const double vrec = block_sum(vrec_p, red);

    __syncthreads();

    // ---- P6: orbital (Pulay) terms, one spin block at a time.  All n x n and
    // B x n products are register-tiled on a zero-padded np x np block (np =
    // padded n, a power of two >= 4):
    //   M1 = Y G,  K = G M1  (= G Y G),  Z = C G,  P = C K  (per tile of C rows)
    // and the basis-derivative contraction is fused onto each Z/P tile.
    const int np = s.np, ldt = np + 4, ng = np / 4;
    const int lnp = __ffs(np) - 1;   // np is a power of two: index arithmetic by shifts (no integer division)
    if constexpr (kSplit) {
        // K = G Y G per spin block for the adjoint kernel, in two buffers: the
        // 4 x 4 register tiles of M1 = Y G overwrite Y^T once every thread has
        // read it, and K^T goes out through the G buffer (coalesced stores).
        T* bufY = (T*)uni;                       // Y^T [j][i], then M1 [i][i']
        T* bufG2 = bufY + (size_t)np * ldt;      // G [j][i], then K^T [i'][j]
        const int r0 = 4 * (tid / ng), c0 = 4 * (tid % ng);
        const bool act = tid < ng * ng;
        for (int sp = 0; sp < 2; ++sp) {
            const T* Gsp = Gt + ((size_t)w * 2 + sp) * n * n;
            for (int idx = tid; idx < np * np; idx += nt) {
                const int il = idx >> lnp, j = idx & (np - 1);
                T g = 0, y = 0;
                if (il < n && j < n) {
                    g = Gsp[il * n + j];
                    y = LpY[((size_t)w * N + sp * n + il) * n + j];
                }
                bufG2[j * ldt + il] = g;
                bufY[j * ldt + il] = y;
            }
            __syncthreads();
            T acc4[4][4] = {};
            if (act) {                           // M1[i][i'] = sum_j Y[i][j] G[j][i']
                for (int j = 0; j < np; ++j) {
                    T y4[4], g4[4];
                    load4(bufY + j * ldt + r0, y4);
                    load4(bufG2 + j * ldt + c0, g4);
#pragma unroll
                    for (int a_ = 0; a_ < 4; ++a_)
#pragma unroll
                        for (int b_ = 0; b_ < 4; ++b_) acc4[a_][b_] += y4[a_] * g4[b_];
                }
            }
            __syncthreads();
            if (act)
#pragma unroll
                for (int a_ = 0; a_ < 4; ++a_)
#pragma unroll
                    for (int b_ = 0; b_ < 4; ++b_) bufY[(r0 + a_) * ldt + c0 + b_] = acc4[a_][b_];
            __syncthreads();
            if (act) {                           // K[j][i'] = sum_i G[j][i] M1[i][i']
#pragma unroll
                for (int a_ = 0; a_ < 4; ++a_)
#pragma unroll
                    for (int b_ = 0; b_ < 4; ++b_) acc4[a_][b_] = 0;
                for (int i = 0; i < np; ++i) {
                    T m4[4];
                    load4(bufY + i * ldt + c0, m4);
#pragma unroll
                    for (int a_ = 0; a_ < 4; ++a_) {
                        const T gji = bufG2[(r0 + a_) * ldt + i];
#pragma unroll
                        for (int b_ = 0; b_ < 4; ++b_) acc4[a_][b_] += gji * m4[b_];
                    }
                }
            }
            __syncthreads();
            if (act)
#pragma unroll
                for (int a_ = 0; a_ < 4; ++a_)
#pragma unroll
                    for (int b_ = 0; b_ < 4; ++b_) bufG2[(c0 + b_) * ldt + r0 + a_] = acc4[a_][b_];
            __syncthreads();
            float* ko = kt_out + ((size_t)w * 2 + sp) * n * n;
            for (int idx = tid; idx < np * np; idx += nt) {
                const int i = idx >> lnp, j = idx & (np - 1);
                if (i < n && j < n) ko[i * n + j] = (float)bufG2[i * ldt + j];
            }
            __syncthreads();
        }
    } else {
    // Rows of C per tile and its stride; the n x n products take 2 x 2 outputs a
    // thread up to n = 32 (256 threads busy; 4 x 4 keeps 64) and 4 x 4 above.  Every
    // sum runs over j in order, whatever the tiling.
    const int RB = np <= 32 ? kPulayRows : 64, ldc = RB + 4;
    T* bufA = (T*)uni;                       // Y^T [j][i], later K [j][i]
    T* bufG = bufA + (size_t)np * ldt;       // G   [j][i] = G_{j,i}
    T* bufM = bufG + (size_t)np * ldt;       // M1  [i][i']
    T* bufS = bufM + (size_t)np * ldt;       // G^T [i][j], later C^T tile [j][b] (stride ldc)
    // out[r][c] = sum_j A[j][r] B[j][c] for TT x TT outputs a thread
    auto square = [&](const T* A, const T* Bm, T* out, auto tile) {
        constexpr int TT = decltype(tile)::value;
        const int ngt = np / TT;
        T acc[TT][TT] = {};
        const int r0 = TT * (tid / ngt), c0 = TT * (tid % ngt);
        const bool on = tid < ngt * ngt;
        if (on)
            for (int j = 0; j < np; ++j) {
                T av[TT], bv[TT];
                if constexpr (TT == 4) {
                    load4(A + j * ldt + r0, av);
                    load4(Bm + j * ldt + c0, bv);
                } else {
                    const float2 a2 = *(const float2*)(A + j * ldt + r0), b2 = *(const float2*)(Bm + j * ldt + c0);
                    av[0] = a2.x; av[1] = a2.y; bv[0] = b2.x; bv[1] = b2.y;
                }
#pragma unroll
                for (int a_ = 0; a_ < TT; ++a_)
#pragma unroll
                    for (int b_ = 0; b_ < TT; ++b_) acc[a_][b_] += av[a_] * bv[b_];
            }
        if (on)
#pragma unroll
            for (int a_ = 0; a_ < TT; ++a_)
#pragma unroll
                for (int b_ = 0; b_ < TT; ++b_) out[(r0 + a_) * ldt + c0 + b_] = acc[a_][b_];
        __syncthreads();
    };
    auto product = [&](const T* A, const T* Bm, T* out) {
        if (np <= 32) square(A, Bm, out, std::integral_constant<int, 2>{});
        else square(A, Bm, out, std::integral_constant<int, 4>{});
    };
    for (int sp = 0; sp < 2; ++sp) {
        const T* Gsp = Gt + ((size_t)w * 2 + sp) * n * n;
        for (int idx = tid; idx < np * np; idx += nt) {
            const int il = idx >> lnp, j = idx & (np - 1);
            T g = 0, y = 0;
            if (il < n && j < n) {
                g = Gsp[il * n + j];
                y = LpY[((size_t)w * N + sp * n + il) * n + j];
            }
            bufS[il * ldt + j] = g;
            bufG[j * ldt + il] = g;
            bufA[j * ldt + il] = y;
        }
        __syncthreads();
        product(bufA, bufG, bufM);               // M1[i][i'] = sum_j Y[i][j] G[j][i']
        product(bufS, bufM, bufA);               // K[j][i'] = sum_i G[j][i] M1[i][i']
        const int B = s.B;
        for (int b0 = 0; b0 < B; b0 += RB) {
            for (int idx = tid; idx < RB * np; idx += nt) {   // C^T tile
                const int bl = idx >> lnp, j = idx & (np - 1);
                bufS[j * ldc + bl] = (b0 + bl < B && j < n) ? s.C[(size_t)(b0 + bl) * n + j] : T(0);
            }
            __syncthreads();
            const int bg = tid / ng, ig = tid % ng;
            const bool act = bg < RB / 4 && b0 + 4 * bg < B;
            T z4[4][4] = {}, p4[4][4] = {};
            if (act) {
                for (int j = 0; j < np; ++j) {
                    T c4[4], g4[4], k4[4];
                    load4(bufS + j * ldc + 4 * bg, c4);
                    load4(bufG + j * ldt + 4 * ig, g4);
                    load4(bufA + j * ldt + 4 * ig, k4);
#pragma unroll
                    for (int a_ = 0; a_ < 4; ++a_)
#pragma unroll
                        for (int b_ = 0; b_ < 4; ++b_) {
                            z4[a_][b_] += c4[a_] * g4[b_];
                            p4[a_][b_] += c4[a_] * k4[b_];
                        }
                }
            }
            // Epilogue.  For chi = exp(-zeta t) with f' = -zeta chi, f'' = zeta^2 chi,
            // f''' = -zeta^3 chi, the radial chain contracts to
            //   grad chi = 2 f' p,  H v = 4 f'' p (p.v) + 2 f' q o v,
            //   grad lap chi = p o (8 f''' |p|^2 + 4 f'' sum q - 2 k^2 f' + 8 f'' q),
            // so the geometry (p, q, p.gU, q o gU) is computed once per
            // (nucleus, electron) and shared by that nucleus' Gaussians.
            T f[24] = {};   // per basis function of the thread: dl (3), de (3)
#pragma unroll
            for (int ii = 0; ii < 4; ++ii) {
                const int il = 4 * ig + ii;
                if (!act || il >= n) continue;
                const int i = sp * n + il;
                const T* gu = gU + 3 * i;
                int a_prev = -1;
                T t = 0, pv[3] = {0, 0, 0}, qv[3] = {0, 0, 0}, pp = 0, sq = 0, pg = 0, qg[3] = {0, 0, 0};
#pragma unroll
                for (int bb = 0; bb < 4; ++bb) {
                    const int b = b0 + 4 * bg + bb;
                    if (b >= B) continue;
                    const int a = b / G, g = b - a * G;
                    if (a != a_prev) {
                        a_prev = a;
                        T sd[3], cd[3];
                        disp_trig(et + 6 * i, s.ptrig + 6 * a, ell, sd, cd, t);
                        pp = 0; sq = 0; pg = 0;
#pragma unroll
                        for (int mu = 0; mu < 3; ++mu) {
                            pv[mu] = ell * sd[mu] * cd[mu];
                            qv[mu] = cd[mu] * cd[mu] - sd[mu] * sd[mu];
                            pp += pv[mu] * pv[mu];
                            sq += qv[mu];
                            pg += pv[mu] * gu[mu];
                            qg[mu] = qv[mu] * gu[mu];
                        }
                    }
                    const T z = s.zetat[g];
                    const T e = qexp(-z * t);
                    const T f1 = -z * e, f2 = z * z * e, f3 = -z * z * z * e;
                    const T A = T(8) * f3 * pp + T(4) * f2 * sq - T(2) * k2 * f1;
                    const T zb = z4[bb][ii], pb = p4[bb][ii];
                    const T g1 = T(2) * f1;
                    const T cp = pb * g1 + zb * T(4) * f2 * pg;   // p terms of pb grad chi + zb H gU
                    const T cq = zb * g1;                          // q o gU term of zb H gU
                    const T hz = T(0.5) * zb;
#pragma unroll
                    for (int mu = 0; mu < 3; ++mu) {
                        // dl -= zb grad chi;  de += pb grad chi + zb (H gU + 1/2 grad lap chi)
                        f[6 * bb + mu] -= zb * g1 * pv[mu];
                        f[6 * bb + 3 + mu] += cp * pv[mu] + cq * qg[mu] + hz * pv[mu] * (A + T(8) * f2 * qv[mu]);
                    }
                }
            }
            // Reduce over the ng threads that share these four basis functions: at each
            // step the pair of threads splits the values between them while they divide
            // (21 exchanges for the 72 of whole values), in the order 1, 2, 4, 8.
            int base = 0;
            auto halve = [&](auto cnt, int o) {
                constexpr int H = decltype(cnt)::value;
                const bool up = ig & o;
#pragma unroll
                for (int k = 0; k < H; ++k) {
                    const T keep = up ? f[k + H] : f[k], give = up ? f[k] : f[k + H];
                    f[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                }
                base += up ? H : 0;
            };
            int left = 24;
            if (ng > 1) { halve(std::integral_constant<int, 12>{}, 1); left = 12; }
            if (ng > 2) { halve(std::integral_constant<int, 6>{}, 2); left = 6; }
            if (ng > 4) { halve(std::integral_constant<int, 3>{}, 4); left = 3; }
            if (ng > 8)
#pragma unroll
                for (int k = 0; k < 3; ++k) f[k] += __shfl_xor_sync(0xffffffffu, f[k], 8);
            if (act && ig < 8)
#pragma unroll
                for (int k = 0; k < 24; ++k)
                    if (k < left) stage[24 * bg + base + k] = (double)f[k];
            __syncthreads();
            {   // one thread per nucleus of this tile sums its basis functions in order
                const int bend = (b0 + RB < B) ? b0 + RB : B;
                const int a_first = b0 / G, a_last = (bend - 1) / G;
                const int a = a_first + tid;
                if (a <= a_last) {
                    const int lo = (a * G > b0) ? a * G : b0, hi = ((a + 1) * G < bend) ? (a + 1) * G : bend;
                    for (int b = lo; b < hi; ++b)
                        for (int mu = 0; mu < 3; ++mu) {
                            f_dl[3 * a + mu] += stage[(b - b0) * 6 + mu];
                            f_de[3 * a + mu] += stage[(b - b0) * 6 + 3 + mu];
                        }
                }
            }
            __syncthreads();
        }
    }

    }

    // ---- P7: accumulate the sample
    const double EL = -0.5 * kin + vee + vep + vrec + s.vconst[0];
    const int N3 = 3 * N;
    const size_t stride = 3 + 9 * (size_t)N;
    double* aw = acc + (size_t)w * stride;
    bool bad = !isfinite(EL);
    for (int c = tid; c < N3; c += nt) {
        const double dl = f_dl[c] + (double)g_dl[c];
        const double de = (f_de[c] + (double)g_de[c]) + (f_dv[c] + (double)g_dv[c]) + s.dvpp[c];
        if (!isfinite(dl) || !isfinite(de)) bad = true;
        aw[3 + c] += dl;
        aw[3 + N3 + c] += EL * dl;
        aw[3 + 2 * N3 + c] += de;
        if (out_dl) { out_dl[(size_t)w * N3 + c] = dl; out_de[(size_t)w * N3 + c] = de; }
    }
    if constexpr (kSplit) {
        for (int idx = tid; idx < 9 * N; idx += nt) {
            const int i = idx / 9, c = idx - 9 * i;
            eg_out[(size_t)w * 9 * N + idx] = (float)(c < 6 ? et[6 * i + c] : gU[3 * i + c - 6]);
        }
        if (tid == 0) elw[w] = EL;
    }
    if (tid == 0) {
        aw[0] += 1.0; aw[1] += EL; aw[2] += EL * EL;
        if (s.vacc) s.vacc[w] += vee + vep + vrec + s.vconst[0];   // V_L, for the virial pressure
        if (out_el) { out_el[w] = EL; out_lnpsi[w] = logdet[2 * w] + logdet[2 * w + 1] + Utot; }
    }
    if (bad) raise_err(s.err, kErrNonfinite);
}

}  // namespace

void launch_measure(const SysView<float>& s, int ntask, const int4* ktask, const float* kint,
                    const double* X, const float* D, float* LpY, const float* Gt,
                    const double* logdet, double* acc, double* out_el, double* out_lnpsi, double* out_dl,
                    double* out_de, float* kt_out, float* eg_out, double* elw, float* rk_out, cudaStream_t st) {
    const bool split = kt_out != nullptr;
    const size_t smem = MLayout(s.N, s.n, s.nk, s.mmax, split).total;
    static bool attr_set[2] = {false, false};
    if (!attr_set[split]) {
        if (split)
            cudaFuncSetAttribute(measure_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        else
            cudaFuncSetAttribute(measure_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        attr_set[split] = true;
    }
    if (split)
        measure_kernel<true><<<s.W, 256, smem, st>>>(s, s.mmax, ntask, ktask, kint, X, D, LpY, Gt, logdet, acc, out_el, out_lnpsi, out_dl,
                                                     out_de, kt_out, eg_out, elw, rk_out);
    else
        measure_kernel<false><<<s.W, 256, smem, st>>>(s, s.mmax, ntask, ktask, kint, X, D, LpY, Gt, logdet, acc, out_el, out_lnpsi, out_dl,
                                                      out_de, nullptr, nullptr, nullptr, nullptr);
}

}  // namespace qmc
