// k_twist.cu -- twisted boundary conditions in the FP64 form: Bloch-summed
// Gaussian orbitals, complex Slater inverses, complex Sherman-Morrison sweeps and
// the twist average (the samples are in k_measure64.cu).
//
// SI, basis section: orbitals with phi(r + nL) = exp(i theta.n) phi(r) for
// integer vectors n.  The Gaussians become Bloch functions by the lattice sum
//   chi_{a,g}(r) = sum_n exp(i theta.n) exp(-zeta_g |r - R_a - nL|^2),
// truncated to the images n = k + m, m in [-M, M]^3 around the nearest one k
// (M from the smallest exponent: every omitted image lies more than
// sqrt(40 / zeta_min) away).  The sum factorises over the axes:
//   chi = exp(i theta.k) s_x s_y s_z,
//   s_mu = sum_{m=-M..M} exp(i theta_mu m) exp(-zeta (d_mu - m L)^2),  d = r - R_a - kL,
// and a derivative in r_mu acts on s_mu alone.  The spin-up determinant takes
// the walker's twist theta, the spin-down one -theta (the SI's opposite
// twists); the Jastrow factor is the real one of the Gamma-point form.
// Walkers come in K contiguous blocks of Wk = W / K, block t on twist t.  The
// sampled density is |psi|^2 and the estimators take real parts:
//   E_L = Re(H psi / psi),  d ln|psi| / dR = Re(d ln psi / dR),  dE_L / dR = Re(d (H psi / psi) / dR).
// Complex values are double2 (x = real, y = imaginary part).
#include "bloch.cuh"
#include "common.cuh"
#include "kernels.cuh"

namespace qmc {

// ---------------------------------------------------------------------------
// Orbital rows (walker w = row / N, electron i = row % N): values phi_j(r) [rows][n],
// complex; nothing needs the derivative rows (k_measure64.cu).  The FP64 pipe bounds
// it, mostly by the exponentials: two or three per axis and Gaussian (bloch_near,
// bloch_far), where a sum over all 2M + 1 images and a sincos per pair took 2.29 ms
// for 32768 rows of N = 64 (1.36 ms now).  256 threads take 32 rows and 8 nuclei at a
// time: one (row, nucleus) each for the basis, TR x TC complex outputs for the product
// with the real coefficients.
// ---------------------------------------------------------------------------
template <int NP, int TR, int TC>
__global__ void __launch_bounds__(256) twist_orbitals_kernel(SysView<double> s, TwistView tv,
                                                             const double* __restrict__ pos, int nrows,
                                                             double2* __restrict__ val) {
    constexpr int RT = 32, NA = 8, CG = NP / TC;
    static_assert(RT / TR * CG == 256, "one output tile per thread");
    extern __shared__ __align__(16) double smem[];
    const int n = s.n, Gn = s.G, N = s.N, M = tv.M, KC = NA * Gn;
    double2* chi = (double2*)smem;                   // [KC][RT]
    double* csm = smem + 2 * (size_t)KC * RT;        // [KC][NP]
    const int tid = threadIdx.x, row0 = blockIdx.x * RT;
    const int al = tid >> 5, r = tid & 31, row = row0 + r < nrows ? row0 + r : nrows - 1;
    const int w = row / N, t = w / tv.Wk;
    const double sg = row - w * N < n ? 1.0 : -1.0;
    const double* th = tv.theta + 3 * t;
    const double2* ph = tv.ph + (size_t)t * 3 * (2 * M + 1);
    const double x[3] = {pos[(size_t)row * 3], pos[(size_t)row * 3 + 1], pos[(size_t)row * 3 + 2]};
    __shared__ int images[8][2];                     // per Gaussian: near and far images (n_gauss <= 8)
    if (tid < Gn) {
        images[tid][0] = bloch_near(s.zeta[tid], s.L, M);
        images[tid][1] = bloch_far(s.zeta[tid], s.L, M);
    }
    const int r0 = tid / CG * TR, c0 = tid % CG * TC;
    double2 acc[TR][TC] = {};
    for (int a0 = 0; a0 < N; a0 += NA) {
        const int na = N - a0 < NA ? N - a0 : NA, rows = na * Gn;
        __syncthreads();
        for (int idx = tid; idx < rows * NP; idx += 256) {
            const int k = idx / NP, j = idx % NP;
            csm[idx] = j < n ? s.C[(size_t)(a0 * Gn + k) * n + j] : 0.0;
        }
        if (al < na) {
            double d0[3];
            const double2 P = bloch_min_image(x, s.R + 3 * (a0 + al), s.L, s.iL, M, ph, th, sg, d0);
            for (int g = 0; g < Gn; ++g) {
                const double z = s.zeta[g];
                const int near = images[g][0], far = images[g][1];
                double2 c = P, sa[1];
#pragma unroll
                for (int mu = 0; mu < 3; ++mu) {
                    bloch_axis<0>(d0[mu], z, s.L, near, far, M, ph + mu * (2 * M + 1), sg, sa);
                    c = cmul(c, sa[0]);
                }
                chi[(al * Gn + g) * RT + r] = c;
            }
        }
        __syncthreads();
#pragma unroll 2
        for (int k = 0; k < rows; ++k) {
            double2 xv[TR];
            double c[TC];
#pragma unroll
            for (int a = 0; a < TR; ++a) xv[a] = chi[k * RT + r0 + a];
#pragma unroll
            for (int m = 0; m < TC; ++m) c[m] = csm[k * NP + c0 + m];
#pragma unroll
            for (int a = 0; a < TR; ++a)
#pragma unroll
                for (int m = 0; m < TC; ++m) {
                    acc[a][m].x += xv[a].x * c[m];
                    acc[a][m].y += xv[a].y * c[m];
                }
        }
    }
#pragma unroll
    for (int a = 0; a < TR; ++a)
#pragma unroll
        for (int m = 0; m < TC; ++m)
            if (row0 + r0 + a < nrows && c0 + m < n) val[(size_t)(row0 + r0 + a) * n + c0 + m] = acc[a][m];
}

template <int NP, int TR, int TC>
static void launch_tw_orb(const SysView<double>& s, const TwistView& tv, const double* pos, int nrows, double2* val,
                          cudaStream_t st) {
    const size_t smem = (size_t)8 * s.G * (2 * 32 + NP) * sizeof(double);
    // allowed once, at n_gauss = 8 (with 16 < n <= 32 that is 48 KB, too much beside the static
    // shared memory without asking): the same value from every thread that calls
    static const cudaError_t allowed =
        cudaFuncSetAttribute(twist_orbitals_kernel<NP, TR, TC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(8 * 8 * (2 * 32 + NP) * sizeof(double)));
    (void)allowed;
    twist_orbitals_kernel<NP, TR, TC><<<(nrows + 31) / 32, 256, smem, st>>>(s, tv, pos, nrows, val);
}

void launch_twist_orbitals(const SysView<double>& s, const TwistView& tv, const double* pos, int nrows, double2* val,
                           cudaStream_t st) {
    if (s.n <= 8) launch_tw_orb<8, 1, 1>(s, tv, pos, nrows, val, st);
    else if (s.n <= 16) launch_tw_orb<16, 1, 2>(s, tv, pos, nrows, val, st);
    else if (s.n <= 32) launch_tw_orb<32, 1, 4>(s, tv, pos, nrows, val, st);
    else launch_tw_orb<64, 2, 4>(s, tv, pos, nrows, val, st);
}

// ---------------------------------------------------------------------------
// Complex Gauss-Jordan inverse of walker w's spin block sp (one CTA per block):
// in place with partial pivoting on the largest modulus (Golub & Van Loan
// sec. 3.4), row interchanges undone on the columns at the end.  Output
// Gt[i][j] = (A^-1)_{j,i} and ln|det A| (the sum of ln|pivot|).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) twist_invert_kernel(int N, int n, const double2* __restrict__ Phi,
                                                           double2* __restrict__ Gt, double* __restrict__ logdet,
                                                           int* err) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int w = blockIdx.x >> 1, sp = blockIdx.x & 1;
    const int ld = n + 1;
    double2* Mx = (double2*)smraw;                 // [n][n+1]
    double2* col = Mx + (size_t)n * ld;            // [n]
    int* perm = (int*)(col + n);                   // [n]
    __shared__ int piv_row;
    __shared__ int singular;
    __shared__ double2 ipv_s;
    __shared__ double lsum;
    const int tid = threadIdx.x, nt = blockDim.x;
    const double2* A = Phi + ((size_t)w * N + (size_t)sp * n) * n;
    for (int idx = tid; idx < n * n; idx += nt) Mx[(idx / n) * ld + idx % n] = A[idx];
    if (tid == 0) { singular = 0; lsum = 0.0; }
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        if (tid < 32) {   // argmax |M[i][k]|^2, i >= k (ties -> lowest row)
            double best = -1.0;
            int bi = n;
            for (int i = k + tid; i < n; i += 32) {
                const double2 v = Mx[i * ld + k];
                const double a = v.x * v.x + v.y * v.y;
                if (a > best) { best = a; bi = i; }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const double ob = __shfl_xor_sync(0xffffffffu, best, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
            }
            if (tid == 0) {
                piv_row = bi;
                perm[k] = bi < n ? bi : k;
                if (!(best > 0.0)) singular = 1;
            }
        }
        __syncthreads();
        if (singular) break;
        const int p = piv_row;
        if (p != k) {
            for (int j = tid; j < n; j += nt) {
                const double2 tmp = Mx[k * ld + j];
                Mx[k * ld + j] = Mx[p * ld + j];
                Mx[p * ld + j] = tmp;
            }
            __syncthreads();
        }
        if (tid == 0) {
            const double2 pv = Mx[k * ld + k];
            lsum += 0.5 * log(pv.x * pv.x + pv.y * pv.y);
            ipv_s = cinv(pv);
        }
        for (int i = tid; i < n; i += nt) col[i] = (i == k) ? czero() : Mx[i * ld + k];
        __syncthreads();
        const double2 ipv = ipv_s;
        for (int j = tid; j < n; j += nt) Mx[k * ld + j] = cmul(j == k ? make_double2(1.0, 0.0) : Mx[k * ld + j], ipv);
        __syncthreads();
        for (int idx = tid; idx < n * n; idx += nt) {
            const int i = idx / n, j = idx - i * n;
            if (i == k) continue;
            const double2 base = (j == k) ? czero() : Mx[i * ld + j];
            Mx[i * ld + j] = csub(base, cmul(col[i], Mx[k * ld + j]));
        }
        __syncthreads();
    }
    if (singular) {
        if (tid == 0) {
            raise_err(err, kErrSingular);
            logdet[2 * w + sp] = -INFINITY;
        }
        return;
    }
    for (int k = n - 1; k >= 0; --k) {       // undo the interchanges on the columns
        const int p = perm[k];
        if (p != k)
            for (int i = tid; i < n; i += nt) {
                const double2 tmp = Mx[i * ld + k];
                Mx[i * ld + k] = Mx[i * ld + p];
                Mx[i * ld + p] = tmp;
            }
        __syncthreads();
    }
    double2* out = Gt + ((size_t)w * 2 + sp) * n * n;
    for (int idx = tid; idx < n * n; idx += nt) {
        const int i = idx / n, j = idx - i * n;       // Gt[i][j] = inv[j][i]
        out[idx] = Mx[j * ld + i];
    }
    if (tid == 0) logdet[2 * w + sp] = lsum;
}

void launch_twist_invert(int W, int N, int n, const double2* Phi, double2* Gt, double* logdet, int* err,
                         cudaStream_t st) {
    const size_t smem = (size_t)n * (n + 1) * sizeof(double2) + n * sizeof(double2) + n * sizeof(int);
    static size_t attr = 0;
    if (smem > attr &&
        cudaFuncSetAttribute(twist_invert_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess)
        attr = smem;
    twist_invert_kernel<<<2 * W, n >= 32 ? 256 : 64, smem, st>>>(N, n, Phi, Gt, logdet, err);
}

// ---------------------------------------------------------------------------
// Metropolis sweep with complex Sherman-Morrison updates (one warp per walker;
// the moving spin block's G^T staged in shared memory, row stride n + 1):
//   ratio  R = sum_j phi'_j G^T[i][j],   accept if u < |R|^2 exp(2 dU),
//   G^T[l] <- G^T[l] - (w_l - delta_{l,i}) / R * G^T[i],  w_l = sum_j phi'_j G^T[l][j].
// dU is the real Jastrow difference of the Gamma-point form (with the e-e-n-n
// term when s.fj is set: c_a = sum_j chi_a(r_j) kept per walker, and the pairs
// (i, j != i) change by sum_a (chi_a(r'_i) - chi_a(r_i)) sum_b f_ab (c_b - chi_b(r_i))).  An accepted
// position is wrapped into the box, x = x' - kL; the orbital row of x is
// exp(-i sg theta.k) times that of x', so row i of G^T (column i of the
// inverse) takes the factor exp(i sg theta.k) to stay the inverse of the
// Slater block at the stored positions.
// ---------------------------------------------------------------------------
__host__ __device__ inline size_t twist_sweep_warp_bytes(int N, int n, bool j34) {
    const size_t b = ((size_t)n * (n + 1) + 2 * (size_t)n) * sizeof(double2) +
                     ((size_t)(j34 ? 10 : 7) * N + 6) * sizeof(double);
    return (b + 15) & ~size_t(15);
}

// e-e-n-n Jastrow orbital exp(-zeta |d|^2) between two points given by their
// (sin, cos)(pi x / L) triples (d the sin-periodised displacement)
__device__ __forceinline__ double tw_jas_orbital(const double* a, const double* b, double ell, double zeta) {
    double t = 0;
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
        const double sd = a[mu] * b[3 + mu] - a[3 + mu] * b[mu];
        t += sd * sd;
    }
    return exp(-zeta * ell * ell * t);
}

__device__ __forceinline__ double tw_pair_dist(const double* a, const double* b, double ell) {
    double t = 0;
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
        const double sd = a[mu] * b[3 + mu] - a[3 + mu] * b[mu];
        t += sd * sd;
    }
    return ell * qsqrt_pair(t);
}

// Pade pair term cu r / (1 + cb r) (cu = 1/2: e-e, cu = -Zj: e-n)
__device__ __forceinline__ double tw_pade_u(const double* a, const double* b, double ell, double cb, double cu) {
    const double r = tw_pair_dist(a, b, ell);
    return cu * r * qrcp(fma(cb, r, 1.0));
}

__global__ void __launch_bounds__(256) twist_sweep_kernel(SysView<double> s, TwistView tv, double* __restrict__ X,
                                                          const double* __restrict__ Xp,
                                                          const double* __restrict__ ptp,
                                                          const double* __restrict__ uacc,
                                                          const double2* __restrict__ Phi, double2* __restrict__ Gt,
                                                          unsigned long long* __restrict__ nacc,
                                                          double* __restrict__ Vep, int vep_init) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int N = s.N, n = s.n, ld = n + 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    double* ptr_s = (double*)smraw;                                   // [N][6] proton trig
    const size_t off = ((size_t)6 * N * sizeof(double) + 15) & ~size_t(15);
    const bool j34 = s.fj != nullptr;
    unsigned char* mine = smraw + off + (size_t)warp * twist_sweep_warp_bytes(N, n, j34);
    double2* Gs = (double2*)mine;            // [n][ld]
    double2* rowb = Gs + (size_t)n * ld;     // [n]
    double2* phi = rowb + n;                 // [n]
    double* ptb = (double*)(phi + n);        // [6] the proposal's trig
    double* et = ptb + 6;                    // [N][6] electron trig
    double* vj = et + 6 * N;                 // [N] V_i = sum_a u_en(r_i, R_a), carried as in sweep_kernel
    double* c34 = vj + N;                    // [N] sum over electrons of chi_a (e-e-n-n term)
    double* dif = c34 + N;                   // [N] c_a - chi_a at the moving electron
    double* dch = dif + N;                   // [N] change of chi_a at its proposal
    for (int idx = threadIdx.x; idx < 6 * N; idx += blockDim.x) ptr_s[idx] = s.ptrig[idx];
    __syncthreads();
    const int w = blockIdx.x * wpb + warp;
    if (w >= s.W) return;   // whole warps leave; only warp-level barriers follow

    const double ell = s.ell, bee = s.b_ee, bep = s.b_ep, Zj = s.Zj, L = s.L;
    double* Xw = X + (size_t)w * 3 * N;
    for (int idx = lane; idx < 3 * N; idx += 32) {
        const int i = idx / 3, mu = idx % 3;
        double sn, cs;
        sincospi(Xw[idx] / L, &sn, &cs);
        et[6 * i + mu] = sn;
        et[6 * i + 3 + mu] = cs;
    }
    __syncwarp();
    for (int i = lane; i < N; i += 32) {
        double v = 0;
        if (vep_init)
            for (int a = 0; a < N; ++a) v += tw_pade_u(et + 6 * i, ptr_s + 6 * a, ell, bep, -Zj);
        else
            v = Vep[(size_t)w * N + i];
        vj[i] = v;
    }
    const double zj = s.zeta_j;
    if (j34) {
        for (int a = lane; a < N; a += 32) {
            double c = 0;
            for (int j = 0; j < N; ++j) c += tw_jas_orbital(et + 6 * j, ptr_s + 6 * a, ell, zj);
            c34[a] = c;
        }
    }
    __syncwarp();
    const double* th = tv.theta + 3 * (w / tv.Wk);
    unsigned long long naccept = 0;
    for (int sp = 0; sp < 2; ++sp) {
        double2* G = Gt + ((size_t)w * 2 + sp) * n * n;
        const double sg = sp == 0 ? 1.0 : -1.0;
        for (int idx = lane; idx < n * n; idx += 32) Gs[(idx / n) * ld + idx % n] = G[idx];
        __syncwarp();
        for (int il = 0; il < n; ++il) {
            const int i = sp * n + il;
            const size_t row = (size_t)w * N + i;
            if (lane < 6) ptb[lane] = ptp[row * 6 + lane];
            for (int j = lane; j < n; j += 32) phi[j] = Phi[row * n + j];
            const double u = uacc[row];
            __syncwarp();
            double2 part = czero();
            for (int j = lane; j < n; j += 32) part = cadd(part, cmul(phi[j], Gs[il * ld + j]));
            const double* ei = et + 6 * i;
            // items 0..N-1: u_ee at the proposal, N..2N-1: minus u_ee at the old position
            double du = 0, vnew = 0;
            for (int k = lane; k < 2 * N; k += 32) {
                const bool old = k >= N;
                const int j = old ? k - N : k;
                const double v = tw_pade_u(old ? ei : ptb, et + 6 * j, ell, bee, old ? -0.5 : 0.5);
                du += j != i ? v : 0.0;
            }
            for (int a = lane; a < N; a += 32) vnew += tw_pade_u(ptb, ptr_s + 6 * a, ell, bep, -Zj);
            if (j34) {
                for (int a = lane; a < N; a += 32) {
                    const double old = tw_jas_orbital(ei, ptr_s + 6 * a, ell, zj);
                    dch[a] = tw_jas_orbital(ptb, ptr_s + 6 * a, ell, zj) - old;
                    dif[a] = c34[a] - old;
                }
                __syncwarp();
                for (int a = lane; a < N; a += 32) {
                    const double* fa = s.fj + a;   // f symmetric: column a = row a, consecutive over lanes
                    double wa = 0;
                    for (int b = 0; b < N; ++b) wa += fa[(size_t)b * N] * dif[b];
                    du += dch[a] * wa;
                }
            }
            // the four warp sums in seven additions: each half of the warp keeps two
            // quantities, then each quarter one
            double2 ratio;
            {
                const bool hi = lane & 16, q = lane & 8;
                double a0 = hi ? du : part.x, a1 = hi ? vnew : part.y;
                a0 += __shfl_xor_sync(0xffffffffu, hi ? part.x : du, 16);
                a1 += __shfl_xor_sync(0xffffffffu, hi ? part.y : vnew, 16);
                double x = q ? a1 : a0;
                x += __shfl_xor_sync(0xffffffffu, q ? a0 : a1, 8);
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                ratio = make_double2(__shfl_sync(0xffffffffu, x, 0), __shfl_sync(0xffffffffu, x, 8));
                du = __shfl_sync(0xffffffffu, x, 16);
                vnew = __shfl_sync(0xffffffffu, x, 24);
            }
            du += vnew - vj[i];
            const double prob = (ratio.x * ratio.x + ratio.y * ratio.y) * exp(2.0 * du);
            if (u < prob) {
                for (int j = lane; j < n; j += 32) rowb[j] = Gs[il * ld + j];
                __syncwarp();
                const double2 ir = cinv(ratio);
                for (int l = lane; l < n; l += 32) {
                    double2 wl = czero();
                    for (int j = 0; j < n; ++j) wl = cadd(wl, cmul(phi[j], Gs[l * ld + j]));
                    if (l == il) wl.x -= 1.0;
                    const double2 coef = cmul(wl, ir);
                    for (int j = 0; j < n; ++j) Gs[l * ld + j] = csub(Gs[l * ld + j], cmul(coef, rowb[j]));
                }
                __syncwarp();
                double kth = 0.0;
#pragma unroll
                for (int mu = 0; mu < 3; ++mu) {
                    const double xpl = Xp[row * 3 + mu];
                    kth += th[mu] * floor(xpl / L);
                }
                if (lane < 3) {
                    const double xpl = Xp[row * 3 + lane];
                    Xw[3 * i + lane] = xpl - L * floor(xpl / L);
                }
                // every use of the trig triple is even in its sign, which is all that wrapping changes
                if (lane < 6) et[6 * i + lane] = ptb[lane];
                if (lane == 0) vj[i] = vnew;
                if (kth != 0.0) {
                    double sn, cs;
                    sincos(sg * kth, &sn, &cs);
                    const double2 f = make_double2(cs, sn);
                    for (int j = lane; j < n; j += 32) Gs[il * ld + j] = cmul(Gs[il * ld + j], f);
                }
                if (j34)
                    for (int a = lane; a < N; a += 32) c34[a] += dch[a];
                ++naccept;
            }
            __syncwarp();
        }
        for (int idx = lane; idx < n * n; idx += 32) G[idx] = Gs[(idx / n) * ld + idx % n];
        __syncwarp();
    }
    for (int i = lane; i < N; i += 32) Vep[(size_t)w * N + i] = vj[i];
    if (lane == 0) nacc[w] += naccept;
}

void launch_twist_sweep(const SysView<double>& s, const TwistView& tv, double* X, const double* Xp, const double* ptp,
                        const double* uacc, const double2* Phi, double2* Gt, unsigned long long* nacc, double* vep,
                        bool vep_init, cudaStream_t st) {
    const size_t wb = twist_sweep_warp_bytes(s.N, s.n, s.fj != nullptr);
    const size_t base = ((size_t)6 * s.N * sizeof(double) + 15) & ~size_t(15);
    int wpb = (int)((200u * 1024u - base) / wb);
    // spread over the SMs: 512 walkers of N = 64 at 8 a CTA filled 64 of 152 (2.70 ms a sweep)
    wpb = walkers_per_cta(s.W, wpb < 1 ? 1 : (wpb > 8 ? 8 : wpb));
    const size_t smem = base + (size_t)wpb * wb;
    static size_t attr = 0;
    if (smem > attr &&
        cudaFuncSetAttribute(twist_sweep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess)
        attr = smem;
    twist_sweep_kernel<<<(s.W + wpb - 1) / wpb, 32 * wpb, smem, st>>>(s, tv, X, Xp, ptp, uacc, Phi, Gt, nacc, vep,
                                                                               vep_init ? 1 : 0);
}

// ---------------------------------------------------------------------------
// Twist average of K per-twist results [E, E_err, N_c, accept, f (3N), S (9N^2)]
// (main text: k-point sampling on a Monkhorst-Pack mesh, equal weights; the
// twists are independent estimates):
//   E, accept, f: means;  E_err = sqrt(sum E_err,t^2) / K;  N_c: sum;  S = sum S_t / K^2.
// ---------------------------------------------------------------------------
__global__ void twist_average_kernel(int K, int N3, const double* __restrict__ tout, double* __restrict__ out) {
    const int len = 4 + N3 + N3 * N3;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= len) return;
    double v = 0.0;
    if (c == 1) {
        for (int t = 0; t < K; ++t) {
            const double e = tout[(size_t)t * len + 1];
            v += e * e;
        }
        out[c] = sqrt(v) / K;
        return;
    }
    for (int t = 0; t < K; ++t) v += tout[(size_t)t * len + c];
    if (c == 2) out[c] = v;                                  // N_c
    else if (c < 4 + N3) out[c] = v / K;                     // E, accept, f
    else out[c] = v / ((double)K * K);                       // S
}

void launch_twist_average(int K, int N, const double* tout, double* out, cudaStream_t st) {
    const int len = 4 + 3 * N + 9 * N * N;
    twist_average_kernel<<<(len + 255) / 256, 256, 0, st>>>(K, 3 * N, tout, out);
}

// Twists sharded over processes: a process whose handle averaged K_r of the K
// twists contributes [K_r E, (K_r E_err)^2, N_c, K_r accept, K_r f, K_r^2 S];
// the sum of the contributions over the processes, divided as below, is the
// average over all K twists (the same combination rule, since
// K_r^2 E_err,r^2 = sum_{t in r} E_err,t^2 and K_r^2 S_r = sum_{t in r} S_t).
__global__ void twist_partial_kernel(double Kr, int N3, const double* __restrict__ out, double* __restrict__ part) {
    const int len = 4 + N3 + N3 * N3;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= len) return;
    const double v = out[c];
    if (c == 1) part[c] = (Kr * v) * (Kr * v);
    else if (c == 2) part[c] = v;
    else if (c < 4 + N3) part[c] = Kr * v;
    else part[c] = Kr * Kr * v;
}

__global__ void twist_combine_kernel(double K, int N3, const double* __restrict__ part, double* __restrict__ out) {
    const int len = 4 + N3 + N3 * N3;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= len) return;
    const double v = part[c];
    if (c == 1) out[c] = sqrt(v) / K;
    else if (c == 2) out[c] = v;
    else if (c < 4 + N3) out[c] = v / K;
    else out[c] = v / (K * K);
}

void launch_twist_partial(int Kr, int N, const double* out, double* part, cudaStream_t st) {
    const int len = 4 + 3 * N + 9 * N * N;
    twist_partial_kernel<<<(len + 255) / 256, 256, 0, st>>>((double)Kr, 3 * N, out, part);
}

void launch_twist_combine(int K, int N, const double* part, double* out, cudaStream_t st) {
    const int len = 4 + 3 * N + 9 * N * N;
    twist_combine_kernel<<<(len + 255) / 256, 256, 0, st>>>((double)K, 3 * N, part, out);
}

}  // namespace qmc
