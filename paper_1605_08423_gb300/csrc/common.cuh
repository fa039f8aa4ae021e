// common.cuh -- device helpers shared by the qmcmd kernels (sm_103a).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace qmc {

constexpr double kPi = 3.14159265358979323846;

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11).  Counter words:
// {stream (walker or component), md step, index (move / electron), purpose}.
// ---------------------------------------------------------------------------
enum : uint32_t {
    kPropX = 0, kPropY = 1, kPropZ = 2, kAccept = 3,
    kInitX = 4, kInitY = 5, kInitZ = 6, kLangevin = 7
};

struct Key { uint32_t k0, k1; };

__host__ __device__ inline Key make_key(uint64_t seed) { return Key{(uint32_t)seed, (uint32_t)(seed >> 32)}; }

__device__ __forceinline__ uint4 philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, Key key) {
    uint32_t k0 = key.k0, k1 = key.k1;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
        const uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
        const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
    return make_uint4(c0, c1, c2, c3);
}

// (0,1) uniforms: 53-bit for FP64, 24-bit for FP32.
__device__ __forceinline__ double u53(uint32_t a, uint32_t b) {
    const uint64_t k = ((uint64_t)(a >> 5) << 26) | (uint64_t)(b >> 6);
    return ((double)k + 0.5) * (1.0 / 9007199254740992.0);
}
__device__ __forceinline__ float u24(uint32_t a) { return ((float)(a >> 8) + 0.5f) * (1.0f / 16777216.0f); }

// Standard normal from one Philox block (Box-Muller, cosine branch) and the
// acceptance uniform, in the precision of the form.
template <typename T> struct Draw;
template <> struct Draw<double> {
    __device__ static double normal(uint4 w) {
        const double a = u53(w.x, w.y), b = u53(w.z, w.w);
        return sqrt(-2.0 * log(a)) * cospi(2.0 * b);
    }
    __device__ static double uniform(uint4 w) { return u53(w.x, w.y); }
};
template <> struct Draw<float> {
    __device__ static float normal(uint4 w) {
        const float a = u24(w.x), b = u24(w.z);
        return sqrtf(-2.0f * logf(a)) * cospif(2.0f * b);
    }
    __device__ static float uniform(uint4 w) { return u24(w.x); }
};

// ---------------------------------------------------------------------------
// Math overloads for the two precision forms.
// ---------------------------------------------------------------------------

// exp(x) in FP64 by table and short polynomial (P. T. P. Tang, ACM Trans. Math.
// Softw. 15, 1989): x = (64 m + j) ln2/64 + r, |r| <= a = ln2/128,
//   exp(x) = 2^m (2^(j/64) + 2^(j/64) p(r)),  p(r) = r + r^2/2 + ... + r^5/120,
// the next term r^6/720 (up to 3.5e-17) taken in by economisation (C. Lanczos, Applied
// Analysis, 1956): r^6 = 3/2 a^2 r^4 - 9/16 a^4 r^2 to a^6/32, which leaves 1.1e-18.
// 11 FP64 operations (the library's 18 cost 290 clocks of an SM's FP64 pipe per
// warp); the result is within 1.01 units in the last place (1.28 without that term).
// From |x| = 690 on, where 2^m (..) leaves the normal range, the library's value
// (0 below -746: no call where far images and nuclei are evaluated by the thousand).
static __device__ const double kExp2j64[64] = {
    0x1.0000000000000p+0, 0x1.02c9a3e778061p+0, 0x1.059b0d3158574p+0, 0x1.0874518759bc8p+0,
    0x1.0b5586cf9890fp+0, 0x1.0e3ec32d3d1a2p+0, 0x1.11301d0125b51p+0, 0x1.1429aaea92de0p+0,
    0x1.172b83c7d517bp+0, 0x1.1a35beb6fcb75p+0, 0x1.1d4873168b9aap+0, 0x1.2063b88628cd6p+0,
    0x1.2387a6e756238p+0, 0x1.26b4565e27cddp+0, 0x1.29e9df51fdee1p+0, 0x1.2d285a6e4030bp+0,
    0x1.306fe0a31b715p+0, 0x1.33c08b26416ffp+0, 0x1.371a7373aa9cbp+0, 0x1.3a7db34e59ff7p+0,
    0x1.3dea64c123422p+0, 0x1.4160a21f72e2ap+0, 0x1.44e086061892dp+0, 0x1.486a2b5c13cd0p+0,
    0x1.4bfdad5362a27p+0, 0x1.4f9b2769d2ca7p+0, 0x1.5342b569d4f82p+0, 0x1.56f4736b527dap+0,
    0x1.5ab07dd485429p+0, 0x1.5e76f15ad2148p+0, 0x1.6247eb03a5585p+0, 0x1.6623882552225p+0,
    0x1.6a09e667f3bcdp+0, 0x1.6dfb23c651a2fp+0, 0x1.71f75e8ec5f74p+0, 0x1.75feb564267c9p+0,
    0x1.7a11473eb0187p+0, 0x1.7e2f336cf4e62p+0, 0x1.82589994cce13p+0, 0x1.868d99b4492edp+0,
    0x1.8ace5422aa0dbp+0, 0x1.8f1ae99157736p+0, 0x1.93737b0cdc5e5p+0, 0x1.97d829fde4e50p+0,
    0x1.9c49182a3f090p+0, 0x1.a0c667b5de565p+0, 0x1.a5503b23e255dp+0, 0x1.a9e6b5579fdbfp+0,
    0x1.ae89f995ad3adp+0, 0x1.b33a2b84f15fbp+0, 0x1.b7f76f2fb5e47p+0, 0x1.bcc1e904bc1d2p+0,
    0x1.c199bdd85529cp+0, 0x1.c67f12e57d14bp+0, 0x1.cb720dcef9069p+0, 0x1.d072d4a07897cp+0,
    0x1.d5818dcfba487p+0, 0x1.da9e603db3285p+0, 0x1.dfc97337b9b5fp+0, 0x1.e502ee78b3ff6p+0,
    0x1.ea4afa2a490dap+0, 0x1.efa1bee615a27p+0, 0x1.f50765b6e4540p+0, 0x1.fa7c1819e90d8p+0};
__device__ __forceinline__ double qexp(double x) {
    const double magic = 6755399441055744.0;                     // 1.5 * 2^52
    const int hx = __double2hiint(x);
    if ((hx & 0x7fffffff) >= 0x40859000)                         // |x| >= 690 or NaN; [-inf, -746] on the integer pipe
        return hx >= (int)0xc0875000 && hx < (int)0xfff00001 ? 0.0 : exp(x);
    const double q = fma(x, 0x1.71547652b82fep+6, magic);                          // 64 / ln 2
    const int k = __double2loint(q);
    const double kd = q - magic;
    const double r = fma(-kd, 0x1.473de6af278edp-40, fma(-kd, 0x1.62e42fef00000p-7, x));              // ln 2 / 64 in two parts
    constexpr double a2 = 2.9324524775280846e-5;                  // (ln 2 / 128)^2
    double p = fma(r, 1.0 / 120.0, 1.0 / 24.0 + 1.5 * a2 / 720.0);
    p = fma(p, r, 1.0 / 6.0);
    p = fma(p, r, 0.5 - 0.5625 * a2 * a2 / 720.0);
    p = fma(p * r, r, r);
    const double t = kExp2j64[k & 63], v = fma(t, p, t);
    return __hiloint2double(__double2hiint(v) + ((k >> 6) << 20), __double2loint(v));
}
__device__ __forceinline__ float qexp(float x) { return expf(x); }
__device__ __forceinline__ double qsqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float qsqrt(float x) { return sqrtf(x); }
// Reciprocal and square root of the pair loops.  FP32: the hardware
// approximations (a few ulp), well inside the FP32-level tolerance of the mixed
// form.  FP64: the FP64 pipe issues two multiply-adds a clock and SM, so the
// pair loops are bound by their FP64 operation count; a hardware seed (about
// 20 bits, PTX rcp / rsqrt.approx.ftz.f64) followed by one third-order
// Householder step (Householder 1970; error of the seed cubed, below 2^-57)
// takes 3 and 5 FP64 operations with no slow path:
//   1/x:       e = 1 - x y,    y (1 + e + e^2)
//   1/sqrt x:  e = 1 - x y^2,  y (1 + e/2 + 3 e^2 / 8)
// Within 0.57 and 1.07 units in the last place; x / sqrt x within 2.1.
// Arguments are normal and positive in the pair loops (1 + b r, t > 0).
__device__ __forceinline__ double rcp_seed(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}
__device__ __forceinline__ double rsqrt_seed(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}
__device__ __forceinline__ double qrcp(double x) {
    const double y = rcp_seed(x);
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ float qrcp(float x) { return __fdividef(1.0f, x); }
__device__ __forceinline__ double qrsqrt(double x) {
    const double y = rsqrt_seed(x);
    const double e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(e, 0.375, 0.5), y);
}
__device__ __forceinline__ double qsqrt_pair(double x) {
    // x = 0 (coincident points) gives 0: the sign-and-magnitude word of a
    // non-negative double is zero only there, so no FP64 compare is needed
    return __double_as_longlong(x) > 0 ? x * qrsqrt(x) : 0.0;
}
__device__ __forceinline__ float qsqrt_pair(float x) { return x > 0.f ? x * rsqrtf(x) : 0.f; }
__device__ __forceinline__ double qerfc(double x) { return erfc(x); }
__device__ __forceinline__ float qerfc(float x) { return erfcf(x); }
__device__ __forceinline__ double qrint(double x) { return rint(x); }
__device__ __forceinline__ float qrint(float x) { return rintf(x); }
__device__ __forceinline__ void qsincospi(double x, double* s, double* c) { sincospi(x, s, c); }
__device__ __forceinline__ void qsincospi(float x, float* s, float* c) { sincospif(x, s, c); }

// Four consecutive elements from 16-byte-aligned shared memory.
__device__ __forceinline__ void load4(const float* p, float o[4]) {
    const float4 v = *(const float4*)p;
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}
__device__ __forceinline__ void load4(const double* p, double o[4]) {
    const double2 a = *(const double2*)p, b = *(const double2*)(p + 2);
    o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums of eight values over the warp in nine additions: lane l returns the sum of
// value (l >> 2) (the halves exchange what the
// other keeps).  Each value is added up in the order of warp_sum.
template <typename T>
__device__ __forceinline__ T warp_sum8(T v[8], int lane) {
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const int o = 16 >> s, w = 4 >> s;
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < w; ++k) {
            const T keep = up ? v[k + w] : v[k], give = up ? v[k] : v[k + w];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    T x = v[0];
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    return x;
}
// Deterministic block reduction (fixed tree) of one value per thread; result
// valid in all threads.  `scratch` holds >= 32 elements.
template <typename T>
__device__ T block_sum(T v, T* scratch) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) scratch[wid] = v;
    __syncthreads();
    T t = (lane < nw) ? scratch[lane] : T(0);
    t = warp_sum(t);
    return t;
}

// Device error word bits.
enum : int { kErrNonfinite = 1, kErrSingular = 2, kErrNotPD = 4, kErrTimeout = 8 };

__device__ __forceinline__ void raise_err(int* err, int bit) { atomicOr(err, bit); }

// ---------------------------------------------------------------------------
// Read-only view of one system on the device (passed by value to kernels).
// ---------------------------------------------------------------------------
template <typename T> struct V2 { T x, y; };

template <typename T>
struct SysView {
    int N, n, G, B, W;
    int np;                 // n padded to a power of two >= 4 (tiled products)
    double L, ell;          // box side, L/pi
    double iL;              // 1/L
    double b_ee, b_ep, Zj;  // Jastrow parameters (Zj = e-n cusp amplitude)
    double kappa;           // Ewald splitting
    const double* zeta;     // [G]
    const T* zetat;         // [G] in the working precision
    const T* C;             // [B][n]
    const double* R;        // [N][3]
    const T* RT;            // [N][3] in the working precision
    const T* ptrig;         // [N][6]: sin(pi R/L) xyz, cos(pi R/L) xyz
    int nk;                 // half-space reciprocal vectors
    int mmax;               // reciprocal cutoff |m| <= mmax
    const int4* kvec;       // [nk] (mx, my, mz, 0)
    const double* kw;       // [nk] (4 pi / L^3) exp(-k^2/4 kappa^2) / k^2
    const double2* eikR;    // [N][nk] exp(i k.R_a)
    const V2<T>* eikRt;     // the same in the working precision
    const T* kwt;           // kw in the working precision
    const double2* rho_p;   // [nk] sum_a Z exp(i k.R_a)
    const double* vconst;   // [1] proton-proton real-space + self energy
    const double* dvpp;     // [3N] d(proton-proton real-space energy)/dR
    int* err;
    double* vacc;           // [W] per-walker sums of the sample's potential energy V_L (pressure), or null
    const double* fj;       // [N][N] e-e-n-n Jastrow coefficients (symmetric), or null
    const T* fjt;           // the same in the working precision, or null
    double zeta_j;          // their Gaussians' exponent
    const double* ewt;      // real-space Ewald table (FP64 form, kappa L <= kEwMaxKL), or null: see EwTable
    double ew_h, ew_ih;     // its node spacing in r^2 and the inverse
    bool served;            // the handle's kernels overlap other trajectories' (see launch_sweep)
};

// Twisted boundary conditions: walker w samples twist t = w / Wk (K contiguous
// blocks); the spin-up orbitals carry theta_t, the spin-down ones -theta_t.
struct TwistView {
    int K, Wk;              // twists, walkers per twist
    int M;                  // Bloch-sum images per axis: m = -M..M around the nearest one
    const double* theta;    // [K][3]
    const double2* ph;      // [K][3][2M+1]: exp(i theta_mu m), m = -M..M
};

// Radial-function chain for f(t), t = |d|^2 with d the sin-periodised
// displacement.  Per component: s = sin(pi D/L), c = cos(pi D/L),
//   p = (L/pi) s c  (so dt/dx = 2p),  q = c^2 - s^2  (dp/dx = q),  dq/dx = -(2pi/L)^2 p.
// Given f', f'', f''' (derivatives in t) this returns the gradient, the
// Hessian (symmetric, xx yy zz xy xz yz), the Laplacian and grad(Laplacian).
template <typename T>
struct RadialDerivs {
    T g[3], h[6], lap, tl[3];
};
template <typename T>
__device__ __forceinline__ void radial_chain(const T p[3], const T q[3], T f1, T f2, T f3, T k2,
                                             RadialDerivs<T>& o) {
    const T pp = p[0] * p[0] + p[1] * p[1] + p[2] * p[2];
    const T sq = q[0] + q[1] + q[2];
#pragma unroll
    for (int m = 0; m < 3; ++m) o.g[m] = T(2) * f1 * p[m];
    o.h[0] = T(4) * f2 * p[0] * p[0] + T(2) * f1 * q[0];
    o.h[1] = T(4) * f2 * p[1] * p[1] + T(2) * f1 * q[1];
    o.h[2] = T(4) * f2 * p[2] * p[2] + T(2) * f1 * q[2];
    o.h[3] = T(4) * f2 * p[0] * p[1];
    o.h[4] = T(4) * f2 * p[0] * p[2];
    o.h[5] = T(4) * f2 * p[1] * p[2];
    o.lap = T(4) * f2 * pp + T(2) * f1 * sq;
#pragma unroll
    for (int m = 0; m < 3; ++m)
        o.tl[m] = p[m] * (T(8) * f3 * pp + T(8) * f2 * q[m] + T(4) * f2 * sq - T(2) * k2 * f1);
}

// H v for the packed symmetric Hessian.
template <typename T>
__device__ __forceinline__ void hess_mul(const T h[6], const T v[3], T out[3]) {
    out[0] = h[0] * v[0] + h[3] * v[1] + h[4] * v[2];
    out[1] = h[3] * v[0] + h[1] * v[1] + h[5] * v[2];
    out[2] = h[4] * v[0] + h[5] * v[1] + h[2] * v[2];
}

// Pade pair functions u(rho) and their rho-derivatives:
//   e-e: u = rho / (2 (1 + b rho))      (cusp +1/2)
//   e-n: u = -Zj rho / (1 + b rho)      (cusp -Zj)
template <typename T>
__device__ __forceinline__ void pade_ee(T b, T r, T& u, T& u1, T& u2) {
    const T q = T(1) + b * r, iq = qrcp(q);
    u = T(0.5) * r * iq; u1 = T(0.5) * iq * iq; u2 = -b * iq * iq * iq;
}
template <typename T>
__device__ __forceinline__ void pade_ep(T b, T Zj, T r, T& u, T& u1, T& u2, T& u3) {
    const T q = T(1) + b * r, iq = qrcp(q), iq2 = iq * iq;
    u = -Zj * r * iq; u1 = -Zj * iq2; u2 = T(2) * Zj * b * iq2 * iq; u3 = T(-6) * Zj * b * b * iq2 * iq2;
}

// Radial factors of the Pade terms u = c r / (1 + b r) in t = r^2, from one
// reciprocal square root and one reciprocal: with iq = 1/(1 + b r), ir = 1/r,
//   2 f1 = c iq^2 ir,  4 f2 = -c iq^2 ir^2 (2 b iq + ir),
//   8 f3 = 3 c iq^2 ir^3 (2 b^2 iq^2 + (2 b iq + ir) ir).
__device__ __forceinline__ void pade_factors(double t, double b, double c, double& u, double& c2, double& c4) {
    const double ir = qrsqrt(t), r = t * ir, iq = qrcp(fma(b, r, 1.0));
    const double A = c * iq * iq;
    u = c * r * iq;
    c2 = A * ir;
    c4 = -(c2 * ir) * fma(2.0 * b, iq, ir);
}
__device__ __forceinline__ void pade_factors3(double t, double b, double c, double& c2, double& c4, double& c8) {
    const double ir = qrsqrt(t), r = t * ir, iq = qrcp(fma(b, r, 1.0));
    const double bq = b * iq, h = fma(2.0, bq, ir), C = c * iq * iq * ir * ir;
    c2 = c * iq * iq * ir;
    c4 = -C * h;
    c8 = 3.0 * (C * ir) * fma(h, ir, 2.0 * bq * bq);
}

// Real-space Ewald pair sum over the images r0 + nL with |r0 + nL| < L of the
// minimum-image vector r0, phi(r) = erfc(kappa r)/r; optionally the gradient
// with respect to r0.
template <typename T>
__device__ __forceinline__ T ewald_real(T dx, T dy, T dz, T Lt, T kappa, T* grad, bool skip_min = false) {
    const T iL = T(1) / Lt;
    dx -= Lt * qrint(dx * iL); dy -= Lt * qrint(dy * iL); dz -= Lt * qrint(dz * iL);
    const T r0[3] = {dx, dy, dz};
    T sh[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) sh[m] = r0[m] >= T(0) ? -Lt : Lt;
    T v = 0;
    if (grad) grad[0] = grad[1] = grad[2] = 0;
    const T c2 = T(1.1283791670955126);  // 2 / sqrt(pi)
    // the (at most 8) candidate images inside the cutoff, compacted into a bit
    // mask so that a warp runs the erfc body only max(popcount) times
    unsigned mask = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const T a = r0[0] + ((c & 1) ? sh[0] : T(0));
        const T b = r0[1] + ((c & 2) ? sh[1] : T(0));
        const T e = r0[2] + ((c & 4) ? sh[2] : T(0));
        const T r2 = a * a + b * b + e * e;
        if (r2 < Lt * Lt && r2 > T(0)) mask |= 1u << c;
    }
    if (skip_min) mask &= ~1u;   // the minimum image is evaluated elsewhere
    while (mask) {
        const int c = __ffs(mask) - 1;
        mask &= mask - 1;
        const T a = r0[0] + ((c & 1) ? sh[0] : T(0));
        const T b = r0[1] + ((c & 2) ? sh[1] : T(0));
        const T e = r0[2] + ((c & 4) ? sh[2] : T(0));
        const T r2 = a * a + b * b + e * e;
        const T r = qsqrt(r2), ir = T(1) / r;
        const T ec = qerfc(kappa * r);
        v += ec * ir;
        if (grad) {
            const T dphi = -(ec * ir + c2 * kappa * qexp(-kappa * kappa * r2)) * ir;  // phi'(r)
            const T s = dphi * ir;
            grad[0] += s * a; grad[1] += s * b; grad[2] += s * e;
        }
    }
    return v;
}

// ---------------------------------------------------------------------------
// Real-space Ewald terms from a table (FP64 form).  With x = (kappa r)^2,
//   erf(kappa r)/r  = kappa (2/sqrt pi) F_0(x),   F_n(x) = int_0^1     s^2n exp(-x s^2) ds,
//   erfc(kappa r)/r = kappa (2/sqrt pi) G_0(x),   G_n(x) = int_1^inf  s^2n exp(-x s^2) ds
// (F_n: the Boys functions, S. F. Boys, Proc. R. Soc. A 200, 1950), and
// d/dx F_n = -F_{n+1}, d/dx G_n = -G_{n+1}: the Taylor coefficients about a node
// are (-1)^n F_n / n! times powers of kappa, filled by stable recurrences
// (k_setup.cu).  Both are tabulated in r^2 at nodes i h, h = 0.75 L^2 / 511, to
// degree 7: erf(kappa r)/r for the minimum image (r^2 <= 3/4 L^2, the term
// 1/r - erf(kappa r)/r), erfc(kappa r)/r for the other images (L^2/4 <= r^2 <
// L^2).  |x - x_node| <= 0.0264 for kappa L <= 6, so the remainder is below
// 1e-18 of kappa for the value and 2e-16 kappa^3 for the derivative in r^2,
// under the rounding of the sums they enter.  A value and its derivative cost
// 16 FP64 operations, where erfc, exp, a square root and the divisions took
// about 190; the FP64 pipe is what bounds the pair sums.
constexpr int kEwNodes = 512, kEwTerms = 8;
constexpr int kEwFirstB = 170;            // first node of the erfc table: floor(0.25 L^2 / h)
constexpr double kEwMaxKL = 6.0;

struct EwTable {
    const double* t;    // [2][kEwNodes][kEwTerms]
    double h, ih, L, iL, LL;
};

// Value at r2 (and derivative in r2) of table `which` (0: erf(kappa r)/r, 1: erfc(kappa r)/r).
template <bool kGrad>
__device__ __forceinline__ double ew_eval(const EwTable& T, int which, double r2, double* d) {
    const double magic = 6755399441055744.0;   // 1.5 * 2^52: the sum's low word is the nearest integer
    const double qm = fma(r2, T.ih, magic);
    int i = __double2loint(qm) - (which ? kEwFirstB : 0);
    i = i < 0 ? 0 : (i > kEwNodes - 1 ? kEwNodes - 1 : i);
    const double t = fma(-T.h, qm - magic, r2);
    const double2* c = (const double2*)(T.t + ((size_t)which * kEwNodes + i) * kEwTerms);
    const double2 c67 = c[3], c45 = c[2], c23 = c[1], c01 = c[0];
    double v = fma(c67.y, t, c67.x);
    if (kGrad) {
        double g = fma(c67.y, t, v);
        v = fma(v, t, c45.y); g = fma(g, t, v);
        v = fma(v, t, c45.x); g = fma(g, t, v);
        v = fma(v, t, c23.y); g = fma(g, t, v);
        v = fma(v, t, c23.x); g = fma(g, t, v);
        v = fma(v, t, c01.y); g = fma(g, t, v);
        v = fma(v, t, c01.x);
        *d = g;
    } else {
        v = fma(v, t, c45.y); v = fma(v, t, c45.x); v = fma(v, t, c23.y);
        v = fma(v, t, c23.x); v = fma(v, t, c01.y); v = fma(v, t, c01.x);
    }
    return v;
}

// ewald_real<double> from the table: sum of phi(r) over the images with r < L,
// and when kGrad its gradient in g (overwritten).
template <bool kGrad>
__device__ __forceinline__ double ewald_table(double dx, double dy, double dz, const EwTable& T, double* g) {
    const double magic = 6755399441055744.0, L = T.L;
    dx = fma(-L, fma(dx, T.iL, magic) - magic, dx);
    dy = fma(-L, fma(dy, T.iL, magic) - magic, dy);
    dz = fma(-L, fma(dz, T.iL, magic) - magic, dz);
    const double r0 = dx * dx + dy * dy + dz * dz;
    // moving component m of the minimum image by L away from zero adds L (L - 2 |d_m|) to r^2
    const double e0 = fma(-2.0 * L, fabs(dx), T.LL), e1 = fma(-2.0 * L, fabs(dy), T.LL),
                 e2 = fma(-2.0 * L, fabs(dz), T.LL);
    const double r1 = r0 + e0, r2 = r0 + e1, r3 = r1 + e1, r4 = r0 + e2, r5 = r1 + e2, r6 = r2 + e2, r7 = r3 + e2;
    // positive doubles compare as their bit patterns (integer pipe)
    const long long lim = __double_as_longlong(T.LL);
    auto in = [&](double r) { return __double_as_longlong(r) < lim; };
    unsigned mask = (in(r1) ? 2u : 0u) | (in(r2) ? 4u : 0u) | (in(r3) ? 8u : 0u) | (in(r4) ? 16u : 0u) |
                    (in(r5) ? 32u : 0u) | (in(r6) ? 64u : 0u) | (in(r7) ? 128u : 0u);
    double v = 0, s = 0, s0 = 0, s1 = 0, s2 = 0, d;
    if (__double_as_longlong(r0) > 0) {
        const double ir = qrsqrt(r0);
        v = ir - ew_eval<kGrad>(T, 0, r0, &d);
        if (kGrad) s = fma(-ir * ir, 0.5 * ir, -d);    // d phi / d r^2
    }
    while (mask) {
        const int c = __ffs(mask) - 1;
        mask &= mask - 1;
        // selected, not summed again: selects run on the integer pipe
        const double lo = (c & 2) ? ((c & 1) ? r3 : r2) : r1;                               // c = 1..3
        const double hi = (c & 2) ? ((c & 1) ? r7 : r6) : ((c & 1) ? r5 : r4);               // c = 4..7
        v += ew_eval<kGrad>(T, 1, (c & 4) ? hi : lo, &d);
        if (kGrad) {
            s += d;
            s0 += (c & 1) ? d : 0.0; s1 += (c & 2) ? d : 0.0; s2 += (c & 4) ? d : 0.0;
        }
    }
    if (kGrad) {   // grad = 2 sum d (x + shift): the shifts collected per component
        const double s2x = s + s;
        g[0] = fma(s2x, dx, (dx >= 0.0 ? -2.0 : 2.0) * L * s0);
        g[1] = fma(s2x, dy, (dy >= 0.0 ? -2.0 : 2.0) * L * s1);
        g[2] = fma(s2x, dz, (dz >= 0.0 ? -2.0 : 2.0) * L * s2);
    }
    return v;
}

// Position of the n-th (0-based) set bit of m (n < popc(m)), by halving.
__device__ __forceinline__ int nth_set_bit(unsigned m, int n) {
    int r = 0;
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1) {
        const int cnt = __popc(m & ((1u << w) - 1u));
        if (n >= cnt) { n -= cnt; m >>= w; r += w; }
    }
    return r;
}

// Mixed form: real-space Ewald cutoff radius squared.  erfc(kappa r) at
// r = 0.8 L with kappa = 5 / L is 1.5e-8, below FP32 resolution of the pair
// sums, so images beyond it are dropped (the FP64 form keeps r < L).
constexpr float kRealCut2Mixed = 0.64f;

// erfc(x) for 0 <= x <= 4.1 in FP32 given e = exp(-x^2):
//   erfc(x) = e t P(t),  t = 1 / (1 + x / 2),
// P a degree-8 polynomial fitted (least squares, relative weight) to
// erfc(x) exp(x^2) / t; relative error 3.1e-7 in FP32 arithmetic (the fit and
// its check are in fit_erfc.py beside this package).
__device__ __forceinline__ float erfc_scaled_fit(float x, float e) {
    const float t = __fdividef(1.0f, 1.0f + 0.5f * x);
    float p = -4.711474106e-02f;
    p = p * t + 2.220349312e-01f;
    p = p * t - 3.470333517e-01f;
    p = p * t + 1.025151908e-01f;
    p = p * t + 1.076001227e-01f;
    p = p * t + 1.385983676e-01f;
    p = p * t + 2.617502213e-01f;
    p = p * t + 2.793540657e-01f;
    p = p * t + 2.822951376e-01f;
    return e * t * p;
}

// 2^x by the hardware approximation (PTX ex2.approx.ftz.f32, a few ulp)
__device__ __forceinline__ float ex2_fast(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Nearest integer of x (|x| < 2^22) in FP32 arithmetic: adding and removing
// 1.5 * 2^23 leaves no fraction bits, and round-to-nearest-even does the
// rounding (IEEE rounding of each addition; no reassociation in this build).
// The FMA pipe does it, where rintf's rounding instruction runs on the FP64
// pipe, a fraction of whose rate this part has.
__device__ __forceinline__ float rint_fma(float x) {
    const float m = 12582912.0f;   // 1.5 * 2^23
    return __fsub_rn(__fadd_rn(x, m), m);
}

// exp(y) / t times erfc(sqrt y)/sqrt y and times minus its derivative in y, t = 1/y,
// 4 <= y <= 30: polynomials of degree 5 and 4, relative error 3e-7 and 3.5e-7
// (fitted by fit_erfc.py, fit_image).
__device__ __forceinline__ float erfc_image_p0(float t) {
    float p = -1.099364281e+00f;
    p = p * t + 1.300195098e+00f;
    p = p * t - 7.889494300e-01f;
    p = p * t + 4.046300352e-01f;
    p = p * t - 2.814249396e-01f;
    p = p * t + 5.641801357e-01f;
    return p;
}
__device__ __forceinline__ float erfc_image_p1(float t) {
    float p = -1.091428846e-01f;
    p = p * t + 1.425238252e-01f;
    p = p * t - 1.344549805e-01f;
    p = p * t + 2.817852199e-01f;
    p = p * t + 5.641948581e-01f;
    return p;
}
constexpr float kImageKLMin = 4.0f, kImageKLMax = 6.8f;   // kappa L with every image in the polynomials' range

// Mixed-form real-space Ewald sum of one pair: the images of the minimum-image
// vector inside the FP32-level cutoff (skip_min: leave out the minimum image),
// phi(r) = erfc(kappa r) / r and, when kGrad, its gradient added to grad.
// iL = 1/Lt and rc2 = kRealCut2Mixed Lt^2 come from the caller (loop invariants).
// Nearly every pair has its minimum image inside the cutoff, so that one is
// evaluated outside the lane loop; the other images (r >= L/2, a warp's loop runs
// to its largest lane count) take the short polynomials above where kappa L
// allows it (`fast`), and their gradients are collected as sum of d phi / d r^2
// with the shifted components' parts apart.
template <bool kGrad>
__device__ __forceinline__ float ewald_real_cut(float dx, float dy, float dz, bool skip_min, bool fast, float Lt,
                                                float iL, float rc2, float kappa, float* grad) {
    dx -= Lt * rint_fma(dx * iL); dy -= Lt * rint_fma(dy * iL); dz -= Lt * rint_fma(dz * iL);
    // moving component m of the minimum image by L away from zero adds
    // L (L - 2 |d_m|) > 0 to r^2 (so only the minimum image can sit at r = 0)
    const float r0 = dx * dx + dy * dy + dz * dz;
    const float e0 = Lt * (Lt - 2.f * fabsf(dx)), e1 = Lt * (Lt - 2.f * fabsf(dy)), e2 = Lt * (Lt - 2.f * fabsf(dz));
    const float r1 = r0 + e0, r2_ = r0 + e1, r3 = r1 + e1, r4 = r0 + e2;
    unsigned mask = (r1 < rc2 ? 2u : 0u) | (r2_ < rc2 ? 4u : 0u) | (r3 < rc2 ? 8u : 0u) | (r4 < rc2 ? 16u : 0u) |
                    (r1 + e2 < rc2 ? 32u : 0u) | (r2_ + e2 < rc2 ? 64u : 0u) | (r3 + e2 < rc2 ? 128u : 0u);
    const float c2k = 1.1283791670955126f * kappa;      // 2 kappa / sqrt(pi)
    const float nk2 = -1.4426950408889634f * kappa * kappa;   // -kappa^2 log2(e)
    float v = 0.f, s = 0.f, s0 = 0.f, s1 = 0.f, s2 = 0.f;     // s: phi'(r) / r
    auto direct = [&](float r2, float& sr) {
        const float ir = rsqrtf(r2), r = r2 * ir;
        const float ex = ex2_fast(nk2 * r2);              // exp(-kappa^2 r^2)
        const float ec = erfc_scaled_fit(kappa * r, ex);
        sr = -(ec * ir + c2k * ex) * ir * ir;
        return ec * ir;
    };
    if (r0 < rc2 && r0 > 0.f && !skip_min) v = direct(r0, s);
    const float ik2 = __fdividef(1.f, kappa * kappa), kd = -2.f * kappa * kappa;
    while (mask) {
        const int c = __ffs(mask) - 1;
        mask &= mask - 1;
        float r2 = r0;
        if (c & 1) r2 += e0;
        if (c & 2) r2 += e1;
        if (c & 4) r2 += e2;
        float sr;
        if (fast) {
            const float ir = rsqrtf(r2), t = ir * ir * ik2;
            const float kt = kappa * t * ex2_fast(nk2 * r2);
            v += kt * erfc_image_p0(t);
            sr = kGrad ? kd * kt * erfc_image_p1(t) : 0.f;
        } else {
            v += direct(r2, sr);
        }
        if (kGrad) {
            s += sr;
            if (c & 1) s0 += sr;
            if (c & 2) s1 += sr;
            if (c & 4) s2 += sr;
        }
    }
    if (kGrad) {
        grad[0] += s * dx + s0 * (dx >= 0.f ? -Lt : Lt);
        grad[1] += s * dy + s1 * (dy >= 0.f ? -Lt : Lt);
        grad[2] += s * dz + s2 * (dz >= 0.f ? -Lt : Lt);
    }
    return v;
}

template <typename T>
__device__ __forceinline__ void disp_trig(const T* ei, const T* pj, T ell, T sd[3], T cd[3], T& t) {
    t = 0;
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
        sd[mu] = ei[mu] * pj[3 + mu] - ei[3 + mu] * pj[mu];
        cd[mu] = ei[3 + mu] * pj[3 + mu] + ei[mu] * pj[mu];
        t += sd[mu] * sd[mu];
    }
    t *= ell * ell;
}

}  // namespace qmc
