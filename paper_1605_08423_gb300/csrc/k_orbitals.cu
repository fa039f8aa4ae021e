// k_orbitals.cu -- walker-batched molecular-orbital evaluation, Metropolis
// proposals and walker placement.
//
// Orbitals (SI, determinant basis; Gaussians periodised by the SI's
// r_mu -> (L/pi) sin(pi r_mu / L) substitution):
//   phi_j(r) = sum_b C[b][j] chi_b(r),  chi_b(r) = exp(-zeta_g t),  t = |d(r - R_a)|^2,  b = a*G + g.
// For a batch of rows (one electron position each) this is the dense
// contraction [rows x B] . [B x n]; the basis tile is produced on the fly in
// shared memory and never written to HBM.
#include "common.cuh"
#include "kernels.cuh"

namespace qmc {

// Mixed form.  Q = 1: values (proposal rows / Slater matrix).
// Q = 4: d/dx, d/dy, d/dz, Laplacian (local energy; it needs no values).
template <typename T, int Q, int NP>
__global__ void __launch_bounds__(512) orbitals_simt(SysView<T> s, const double* __restrict__ pos, int nrows,
                                                     T* __restrict__ val, T* __restrict__ grad, T* __restrict__ lap) {
    constexpr int RT = 32, KC = 16, CG = NP / 4;
    __shared__ T rtrig[RT][6];
    __shared__ T chi[Q][KC][RT];
    __shared__ __align__(16) T csm[KC][NP];
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int row0 = blockIdx.x * RT;
    const int n = s.n, B = s.B, G = s.G;
    const T ell = (T)s.ell;

    for (int idx = tid; idx < RT * 3; idx += nthr) {
        const int r = idx / 3, mu = idx % 3, row = row0 + r;
        T sn = 0, cs = 1;
        if (row < nrows) qsincospi((T)(pos[(size_t)row * 3 + mu] / s.L), &sn, &cs);
        rtrig[r][mu] = sn;
        rtrig[r][3 + mu] = cs;
    }
    const int rg = tid / CG, cg = tid % CG;
    const int r0 = 2 * rg, c0 = 4 * cg;
    T acc[Q][2][4];
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int m = 0; m < 4; ++m) acc[q][a][m] = T(0);

    for (int k0 = 0; k0 < B; k0 += KC) {
        __syncthreads();
        for (int idx = tid; idx < KC * NP; idx += nthr) {
            const int kk = idx / NP, j = idx % NP, b = k0 + kk;
            csm[kk][j] = (b < B && j < n) ? s.C[(size_t)b * n + j] : T(0);
        }
        for (int idx = tid; idx < KC * RT; idx += nthr) {
            const int kk = idx / RT, r = idx % RT, b = k0 + kk;
            T v[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) v[q] = T(0);
            if (b < B && row0 + r < nrows) {
                const int a = b / G, g = b - a * G;
                const T* pt = s.ptrig + 6 * a;
                T sd[3], cd[3], t = 0;
#pragma unroll
                for (int mu = 0; mu < 3; ++mu) {
                    const T sx = rtrig[r][mu], cx = rtrig[r][3 + mu], sr = pt[mu], cr = pt[3 + mu];
                    sd[mu] = sx * cr - cx * sr;
                    cd[mu] = cx * cr + sx * sr;
                    t += sd[mu] * sd[mu];
                }
                t *= ell * ell;
                const T z = s.zetat[g];
                const T e = qexp(-z * t);
                if constexpr (Q == 1) {
                    v[0] = e;
                } else {
                    const T f1 = -z * e, f2 = z * z * e;
                    T pp = 0, sq = 0;
#pragma unroll
                    for (int mu = 0; mu < 3; ++mu) {
                        const T p = ell * sd[mu] * cd[mu], qq = cd[mu] * cd[mu] - sd[mu] * sd[mu];
                        v[mu] = T(2) * f1 * p;
                        pp += p * p; sq += qq;
                    }
                    v[Q - 1] = T(4) * f2 * pp + T(2) * f1 * sq;
                }
            }
#pragma unroll
            for (int q = 0; q < Q; ++q) chi[q][kk][r] = v[q];
        }
        __syncthreads();
        if (rg * 2 < RT) {
#pragma unroll 4
            for (int kk = 0; kk < KC; ++kk) {
                T c[4];
#pragma unroll
                for (int m = 0; m < 4; ++m) c[m] = csm[kk][c0 + m];
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const T x0 = chi[q][kk][r0], x1 = chi[q][kk][r0 + 1];
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        acc[q][0][m] += x0 * c[m];
                        acc[q][1][m] += x1 * c[m];
                    }
                }
            }
        }
    }
    if (rg * 2 >= RT) return;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        const int row = row0 + r0 + a;
        if (row >= nrows) continue;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int j = c0 + m;
            if (j >= n) continue;
            if constexpr (Q == 1) {
                val[(size_t)row * n + j] = acc[0][a][m];
            } else {
#pragma unroll
                for (int mu = 0; mu < 3; ++mu) grad[((size_t)row * 3 + mu) * n + j] = acc[mu][a][m];
                lap[(size_t)row * n + j] = acc[Q - 1][a][m];
            }
        }
    }
}

// FP64 form: values of the orbitals (nothing of it needs derivative rows).  The
// FP64 pipe bounds it: per (row, nucleus) the squared distance, per Gaussian one
// exponential, per (row, basis function, orbital) one multiply-add.  256 threads
// take 32 rows and 8 nuclei at a time -- one (row, nucleus) each for the basis,
// TR x TC outputs each for the product -- so that the 128 CTAs of a small call
// (256 walkers of N = 16) keep all four FP64 issue ports of their SMs busy; 64
// threads a CTA took 36.7 us there, and one distance per Gaussian 886 us for
// 65536 rows of N = 64 (now 12.7 and 716 us).  trig: (sin, cos)(pi x / L) of the rows
// where the caller has them (the proposals).
template <int NP, int TR, int TC>
__global__ void __launch_bounds__(256) orbitals64_kernel(SysView<double> s, const double* __restrict__ pos,
                                                         const double* __restrict__ trig, int nrows,
                                                         double* __restrict__ val) {
    constexpr int RT = 32, NA = 8, CG = NP / TC;
    static_assert(RT / TR * CG == 256, "one output tile per thread");
    extern __shared__ __align__(16) double smem[];
    const int n = s.n, G = s.G, N = s.N, KC = NA * G;
    double* rt = smem;                    // [RT][6]
    double* chi = rt + RT * 6;            // [KC][RT]
    double* csm = chi + (size_t)KC * RT;  // [KC][NP]
    const int tid = threadIdx.x, row0 = blockIdx.x * RT;
    if (trig) {
        for (int idx = tid; idx < RT * 6; idx += 256)
            rt[idx] = row0 + idx / 6 < nrows ? trig[(size_t)row0 * 6 + idx] : 0.0;
    } else {
        for (int idx = tid; idx < RT * 3; idx += 256) {
            const int r = idx / 3, mu = idx % 3;
            double sn = 0, cs = 1;
            if (row0 + r < nrows) sincospi(pos[(size_t)(row0 + r) * 3 + mu] / s.L, &sn, &cs);
            rt[r * 6 + mu] = sn;
            rt[r * 6 + 3 + mu] = cs;
        }
    }
    const int r0 = tid / CG * TR, c0 = tid % CG * TC;
    const double ell2 = s.ell * s.ell;
    double acc[TR][TC] = {};
    for (int a0 = 0; a0 < N; a0 += NA) {
        const int na = N - a0 < NA ? N - a0 : NA, rows = na * G;
        __syncthreads();
        for (int idx = tid; idx < rows * NP; idx += 256) {
            const int k = idx / NP, j = idx % NP;
            csm[idx] = j < n ? s.C[(size_t)(a0 * G + k) * n + j] : 0.0;
        }
        {
            const int al = tid >> 5, r = tid & 31;
            if (al < na) {
                const double* pt = s.ptrig + 6 * (a0 + al);
                double t = 0;
#pragma unroll
                for (int mu = 0; mu < 3; ++mu) {
                    const double sd = rt[r * 6 + mu] * pt[3 + mu] - rt[r * 6 + 3 + mu] * pt[mu];
                    t += sd * sd;
                }
                t *= ell2;
                for (int g = 0; g < G; ++g) chi[(al * G + g) * RT + r] = qexp(-s.zeta[g] * t);
            }
        }
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < rows; ++k) {
            double x[TR], c[TC];
#pragma unroll
            for (int a = 0; a < TR; ++a) x[a] = chi[k * RT + r0 + a];
#pragma unroll
            for (int m = 0; m < TC; ++m) c[m] = csm[k * NP + c0 + m];
#pragma unroll
            for (int a = 0; a < TR; ++a)
#pragma unroll
                for (int m = 0; m < TC; ++m) acc[a][m] += x[a] * c[m];
        }
    }
#pragma unroll
    for (int a = 0; a < TR; ++a)
#pragma unroll
        for (int m = 0; m < TC; ++m)
            if (row0 + r0 + a < nrows && c0 + m < n) val[(size_t)(row0 + r0 + a) * n + c0 + m] = acc[a][m];
}

template <int NP, int TR, int TC>
static void launch_orb64(const SysView<double>& s, const double* pos, const double* trig, int nrows, double* val,
                         cudaStream_t st) {
    const size_t smem = (32 * 6 + (size_t)8 * s.G * (32 + NP)) * sizeof(double);
    // allowed once, at n_gauss = 8: the same value from every thread that calls
    static const cudaError_t allowed = cudaFuncSetAttribute(
        orbitals64_kernel<NP, TR, TC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
        (int)((32 * 6 + 8 * 8 * (32 + NP)) * sizeof(double)));
    (void)allowed;
    orbitals64_kernel<NP, TR, TC><<<(nrows + 31) / 32, 256, smem, st>>>(s, pos, trig, nrows, val);
}

void launch_orbitals(const SysView<double>& s, const double* pos, const double* trig, int nrows, double* val,
                     cudaStream_t st) {
    if (s.n <= 8) launch_orb64<8, 1, 1>(s, pos, trig, nrows, val, st);
    else if (s.n <= 16) launch_orb64<16, 1, 2>(s, pos, trig, nrows, val, st);
    else if (s.n <= 32) launch_orb64<32, 1, 4>(s, pos, trig, nrows, val, st);
    else launch_orb64<64, 2, 4>(s, pos, trig, nrows, val, st);
}

template <int Q>
static void launch_orb(const SysView<float>& s, const double* pos, int nrows, float* val, float* grad, float* lap,
                       cudaStream_t st) {
    const int grid = (nrows + 31) / 32;
    if (s.n <= 16)
        orbitals_simt<float, Q, 16><<<grid, 16 * 4, 0, st>>>(s, pos, nrows, val, grad, lap);
    else if (s.n <= 32)
        orbitals_simt<float, Q, 32><<<grid, 16 * 8, 0, st>>>(s, pos, nrows, val, grad, lap);
    else
        orbitals_simt<float, Q, 64><<<grid, 16 * 16, 0, st>>>(s, pos, nrows, val, grad, lap);
}

void launch_orbitals(const SysView<float>& s, const double* pos, int nrows, float* val, float* grad, float* lap,
                     cudaStream_t st) {
    if (grad) launch_orb<4>(s, pos, nrows, nullptr, grad, lap, st);
    else launch_orb<1>(s, pos, nrows, val, nullptr, nullptr, st);
}

// ---------------------------------------------------------------------------
// Proposals of one sweep: Xp = X + sigma xi (Philox normals, purposes 0..2),
// their (sin, cos)(pi x'/L) in the working precision, and the acceptance
// uniforms (purpose 3), index = sweep * N + electron.  A move of electron i
// only ever changes r_i, so every proposal of the sweep is known when the
// sweep starts.  X is wrapped into [0, L) first (the mixed sweep stores
// accepted positions unwrapped).  The Philox stream of walker w is w0 + w
// (w0: the handle's first walker in a walker-sharded run).
// ---------------------------------------------------------------------------
// FP64: one thread per coordinate, then one per uniform (the normal and the trig
// are some 130 FP64 instructions: an electron's three in one thread made a chain
// of 26 us on the 128 warps of a small call, 256 walkers of N = 16; now 9 us).
// FP32: one thread per electron, which writes its trig triple whole (per
// coordinate took 152 us against 108 us for 16384 walkers of N = 128).
template <typename T>
__device__ __forceinline__ void propose_coordinate(int t, int mu, int w, uint32_t idx, double L, double* __restrict__ X,
                                                   double* __restrict__ Xp, T* __restrict__ ptp, Key key, uint32_t md,
                                                   double sigma, uint32_t w0) {
    const double iL = 1.0 / L;
    double x = X[(size_t)t * 3 + mu];
    x -= L * floor(x * iL);
    X[(size_t)t * 3 + mu] = x;
    const T z = Draw<T>::normal(philox(w0 + (uint32_t)w, md, idx, kPropX + mu, key));
    const double xp = x + sigma * (double)z;
    Xp[(size_t)t * 3 + mu] = xp;
    T sn, cs;
    qsincospi((T)(xp * iL), &sn, &cs);
    ptp[(size_t)t * 6 + mu] = sn;
    ptp[(size_t)t * 6 + 3 + mu] = cs;
}

template <typename T>
__global__ void propose_kernel(int W, int N, double L, double* __restrict__ X, double* __restrict__ Xp,
                               T* __restrict__ ptp, T* __restrict__ uacc, Key key, uint32_t md, uint32_t sweep,
                               double sigma, uint32_t w0) {
    const int rows = W * N;
    const ProposeTask task = propose_task((long long)blockIdx.x * blockDim.x + threadIdx.x, rows, sizeof(T) == 8);
    if (task.t < 0) return;
    const int t = task.t, w = t / N, i = t - w * N;
    const uint32_t idx = sweep * (uint32_t)N + (uint32_t)i;
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int mu = 0; mu < 3; ++mu) propose_coordinate<T>(t, mu, w, idx, L, X, Xp, ptp, key, md, sigma, w0);
    } else if (task.mu < 3) {
        propose_coordinate<T>(t, task.mu, w, idx, L, X, Xp, ptp, key, md, sigma, w0);
    }
    if (task.mu == 3) uacc[t] = Draw<T>::uniform(philox(w0 + (uint32_t)w, md, idx, kAccept, key));
}

template <typename T>
void launch_propose(int W, int N, double L, double* X, double* Xp, T* ptp, T* uacc, Key key, uint32_t md,
                    uint32_t sweep, double sigma, uint32_t w0, cudaStream_t st) {
    const int tpb = sizeof(T) == 4 ? 256 : 128;
    propose_kernel<T><<<propose_blocks(W * N, sizeof(T) == 8, tpb), tpb, 0, st>>>(W, N, L, X, Xp, ptp, uacc, key, md, sweep, sigma, w0);
}

// Walker start: electron i next to proton i (up electrons on protons 0..N/2-1,
// down electrons on N/2..N-1) plus 0.5 bohr Gaussian noise, wrapped; the
// Philox stream of walker w is w0 + w.
__global__ void init_walkers_kernel(int W, int N, double L, const double* __restrict__ R, double* __restrict__ X,
                                    Key key, uint32_t w0) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= W * N) return;
    const int w = t / N, i = t - w * N;
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
        const double z = Draw<double>::normal(philox(w0 + (uint32_t)w, 0u, (uint32_t)i, kInitX + mu, key));
        const double x = R[3 * i + mu] + 0.5 * z;
        X[(size_t)t * 3 + mu] = x - L * floor(x / L);
    }
}

void launch_init_walkers(int W, int N, double L, const double* R, double* X, Key key, uint32_t w0, cudaStream_t st) {
    init_walkers_kernel<<<(W * N + 255) / 256, 256, 0, st>>>(W, N, L, R, X, key, w0);
}

template void launch_propose<double>(int, int, double, double*, double*, double*, double*, Key, uint32_t, uint32_t,
                                     double, uint32_t, cudaStream_t);
template void launch_propose<float>(int, int, double, double*, double*, float*, float*, Key, uint32_t, uint32_t,
                                    double, uint32_t, cudaStream_t);

}  // namespace qmc
